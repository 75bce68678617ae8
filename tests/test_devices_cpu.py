"""The library's host code on two devices of one process, over a runtime without
GPUs (fake_cudart.cpp): every entry point that works on the first works on the
second.

The pointers are the host's, so no call may reach the real runtime, which torch puts
in the process's global symbol scope: the library binds its calls to the runtime it
was linked with (-Bsymbolic) and leaves none open (-z defs), and it runs in a process
of its own, without torch and without a visible device."""
import ctypes as C
import glob
import os
import re
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))


def fake_library(folder):
    import pytest

    from paper_2403_18466_gb300 import build
    cxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    build.build()
    out = os.path.join(folder, "liblbm_fake.so")
    subprocess.run([cxx, "-shared", "-fPIC", "-O1", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-I", inc,
                    "-o", out, os.path.join(HERE, "fake_cudart.cpp"),
                    *sorted(glob.glob(os.path.join(build.BUILD, "*.o")))], check=True)
    return out


def _calls(lib, lbm, mem):
    """(name, status) of a pass over the entry points that launch kernels."""
    ctx, c3 = C.c_void_p(), C.c_void_p()
    prm = lbm.make_params(64, 48, 1, tau=0.6, smag_cs=0.1, force_amp=1e-4, force_mode=1)
    p = [C.addressof(m) for m in mem]
    w = lbm.lbm_weights(*[p[2]] * 6, 0)
    yield "init", lib.lbm_init(C.byref(ctx), C.byref(prm), p[0], p[1], None)
    yield "set_state", lib.lbm_set_state(ctx, p[2])
    for kind in lbm.KINDS.values():
        for n in (1, 4):
            yield f"step {kind} {n}", lib.lbm_step(ctx, n, kind, C.byref(w))
    size = lib.lbm_record_bytes(C.byref(prm), 3, 2)
    for rec, back in (("lbm_forward_record", "lbm_backward"),
                      ("lbm_forward_record_bf16", "lbm_backward_bf16")):
        yield rec, getattr(lib, rec)(ctx, 3, 2, C.byref(w), p[3], size)
        yield back, getattr(lib, back)(ctx, p[2], C.byref(w), p[3], size, p[4], None)
    yield "structure", lib.lbm_structure_functions(ctx, 20, p[4])
    yield "structure", lib.lbm_structure_functions(ctx, 300, p[4])
    yield "spectrum", lib.lbm_energy_spectrum(ctx, 20, p[4])
    yield "box", lib.lbm_box_filter(ctx, 4, p[4])
    large = lbm.make_params(1024, 700, 1, tau=0.6)  # more than four tiles per SM
    big = C.c_void_p()
    yield "init", lib.lbm_init(C.byref(big), C.byref(large), p[0], p[1], None)
    yield "step", lib.lbm_step(big, 4, lbm.LBM_MLP_BF16, C.byref(w))
    prm3 = lbm.lbm3d_params(8, 8, 8, 1, 0.6, 0.1, 1.0, 0.0, 0, 0)
    w3 = lbm.lbm3d_weights(*[p[2]] * 8, 0)
    yield "init 3d", lib.lbm3d_init(C.byref(c3), C.byref(prm3), p[0], p[1], None)
    for kind in lbm.KINDS.values():
        yield f"step 3d {kind}", lib.lbm3d_step(c3, 2, kind, C.byref(w3))
    for c in (ctx, big):
        lib.lbm_destroy(c)
    lib.lbm3d_destroy(c3)


def two_devices(path):
    from paper_2403_18466_gb300 import lbm
    assert "torch" not in sys.modules and os.environ["CUDA_VISIBLE_DEVICES"] == ""
    lib = C.CDLL(path)
    for name, (res, args) in lbm._SIGS.items():
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    mem = [(C.c_char * n)() for n in (1 << 22, 1 << 22, 1 << 22, 1 << 24, 1 << 18)]
    before = lib.fake_launches()
    for device in (0, 1):
        lib.fake_set_device(device)
        bad = [(name, rc) for name, rc in _calls(lib, lbm, mem) if rc != lbm.LBM_OK]
        assert not bad, f"device {device}: {bad}"
    assert lib.fake_launches() - before > 80


def test_second_device_of_a_process(tmp_path):
    import torch  # noqa: F401  (the real runtime in this process must not matter)
    env = {**os.environ, "CUDA_VISIBLE_DEVICES": "", "PYTHONPATH": os.path.dirname(HERE)}
    run = subprocess.run([sys.executable, os.path.abspath(__file__), fake_library(str(tmp_path))],
                         env=env, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr


def test_launchers_hold_no_state_of_the_process():
    """A variable that outlives a launch would be one for all devices and threads
    (noalloc.cu keeps its buffers by device, under a lock)."""
    from paper_2403_18466_gb300 import build
    for src in build._sources() + build._headers():
        if os.path.basename(src) == "noalloc.cu":
            continue
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(src).read(), flags=re.S)
        held = re.findall(r"\bstatic (?!constexpr\b|const\b)[^;({]*[=;]", text)
        assert not held, f"{os.path.basename(src)}: {held}"


if __name__ == "__main__":
    two_devices(sys.argv[1])
