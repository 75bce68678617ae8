"""A CTA of a tensor-core kernel must not leave while something is on its way to
its shared memory: its own bulk copy, or, on the CTA pairs of the D3Q19 step,
an MMA commit of the other CTA.  That is an order of asynchronous events, so the
CPU tests follow the kernels' source."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_18466_gb300", "csrc")


def _block(src, start):
    """Text of the braces that open at or after `start`, and its end."""
    i = src.index("{", start)
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return src[i:j + 1], j + 1
    raise ValueError("unbalanced braces")


def kernel_body(name, kernel):
    """A kernel's body without comments."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return _block(src, src.index(kernel + "(const float"))[0]


def kernel_parts():
    """The D3Q19 step kernel's body as (before the roles, code that only CTA 0
    runs, the rest)."""
    body = kernel_body("d3q19_mlp_tc.cu", "k3_step_mlp_tc")
    roles = body.index("if (warp >= MMA_WARP)")
    issue, end = _block(body, body.index("rank == 0", roles))
    return body[:roles], issue, body[roles:body.index(issue)] + body[end:]


def test_both_ctas_wait_for_every_commit():
    """Every barrier that a commit arrives at in both CTAs is waited for in code
    that both run (CTA 1 issues no MMA, so a wait in the issuers' block is
    CTA 0's alone)."""
    _, issue, both = kernel_parts()
    names = set(re.findall(r"commit_pair\(smem_u32\(&S\.(\w+)", issue))
    assert {"c1a", "c4", "drain"} <= names
    assert "commit_pair" not in both
    for n in sorted(names):
        assert re.search(rf"smem_u32\(&S\.{n}\b", both), n


def test_weight_copy_verdict_is_common_to_the_pair():
    """A CTA whose weights have not landed tells the other one between two
    cluster barriers (the first: the other's error word exists; the second: the
    verdict is read after it), and waits for its copy again before it leaves."""
    before, _, both = kernel_parts()
    order = r"cluster_sync\(\).*wait_done\(smem_u32\(&S\.wload\)\).*record_error\(err\).*" \
            r"cluster_sync\(\).*ok0 = .*err"
    assert re.search(order, before, re.S)
    assert "S.err = 1" not in before
    assert re.search(r"wait_done\(smem_u32\(&S\.wload\)\).*cluster_sync\(\)", both, re.S)


def test_late_weight_copy_of_the_2d_step_is_waited_for_at_the_exit():
    body = kernel_body("mlp_bf16.cu", "k_step_mlp_bf16")
    at = body.index("if (leader && fail)")
    assert "mbar_wait_bounded" in _block(body, at)[0] and "S.wbar" in _block(body, at)[0]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(1024, 64), (1024, 704)])
def test_time_out_in_a_call_of_several_steps(nx, ny):
    """Steps that take their weights with a bulk copy (half-size and full CTAs):
    a wait that runs out gives the status, and the next call is sound again.  (With
    a tile alone on its SM one poll suffices: the thread that committed a GEMM
    stalls at its next memory access until it is done.)"""
    import torch

    from paper_2403_18466_gb300 import inputs, lbm
    dev = "cuda:0"
    w = lbm.weights_struct(torch.tensor(inputs.xavier_mlp(3, out_scale=0.1), dtype=torch.float32,
                                        device=dev))
    g = torch.Generator(device=dev).manual_seed(ny)
    f = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=dev).view(1, 9, 1, 1) * \
        (1 + 0.01 * torch.rand((1, 9, ny, nx), generator=g, device=dev))
    a, b = (lbm.Lattice(nx, ny, 1, tau=0.6, device=dev) for _ in range(2))
    a.set_state(f)
    a.set_wait_limit(1)
    a.step(3, "mlp_bf16", w)
    assert a.status() == lbm.LBM_ERR_TIMEOUT
    a.set_wait_limit(0)
    a.clear_status()
    for lat in (a, b):
        lat.set_state(f)
        lat.step(3, "mlp_bf16", w)
        assert lat.status() == lbm.LBM_OK
    assert torch.equal(a.get_state(), b.get_state())


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,nz", [(5, 3, 2), (16, 8, 2), (64, 32, 20)])
def test_back_to_back_steps_of_a_pair(nx, ny, nz):
    """Steps that follow one another at once, from one pair of CTAs whose second
    tile is empty to pairs on every SM, with a kernel in between that takes over
    the shared memory: the same bits every time, no time-out."""
    import torch

    from paper_2403_18466_gb300 import inputs, lbm
    dev = "cuda:0"
    th = torch.tensor(inputs.xavier_mlp_widths(7, lbm.LBM3D_WIDTHS, bias_scale=0.1,
                                               out_scale=0.001), dtype=torch.float32, device=dev)
    w = lbm.weights3d_struct(th)
    lat = lbm.Lattice3D(nx, ny, nz, 1, tau=0.7, device=dev)
    g = torch.Generator(device=dev).manual_seed(nx)
    rest = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, device=dev) \
        .view(1, 19, 1, 1, 1) * (1 + 0.01 * torch.rand((1, 19, nz, ny, nx), generator=g, device=dev))
    first = None
    for _ in range(4):
        lat.set_state(rest)
        for _ in range(20):
            lat.step(3, "mlp_bf16", w)
            lat.step(1, "mlp_f32", w)
        got = lat.get_state()
        assert lat.status() == lbm.LBM_OK
        first = got if first is None else first
        assert torch.equal(got, first) and torch.isfinite(got).all()
