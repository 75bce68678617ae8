"""Kernels whose tiles run over consecutive nodes of the flattened lattice,
at the sizes where that can go wrong: one node more or less than a tile, tiles
that span rows, planes and lattices of a batch, and narrow lattices.

Tolerances are those of the same kernels' parity tests (one FP32 step: 1e-5 of
each weight).
"""
import numpy as np
import pytest

import oracle.d3q19 as o3
from paper_2403_18466_gb300 import inputs
from test_gpu_d3q19 import _dev, _np, _weights, emulate_tc_step, field3d, lbm, wpe  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


@pytest.mark.parametrize("nx,ny,nz,B", [(31, 1, 1, 1), (11, 3, 1, 1), (8, 4, 2, 1), (5, 3, 3, 3),
                                        (2, 1, 33, 2), (97, 3, 2, 1)])
def test_d3q19_f32_tiles(lbm, nx, ny, nz, B):  # noqa: F811
    """FP32 learned D3Q19 step (tiles of 32 nodes) against the oracle."""
    tau, F = 0.6, 2e-4
    theta = _weights(22)
    lat = lbm.Lattice3D(nx, ny, nz, B, tau=tau, force_amp=F, force_mode=1, device=DEV)
    lat.set_state(_dev(field3d(B, nz, ny, nx, seed=41, neq=0.02)))
    g = o3.stream_push(_np(lat.get_state()))
    th = torch.tensor(theta, dtype=torch.float32, device=DEV)
    lat.step(1, "mlp_f32", lbm.weights3d_struct(th))
    prm = o3.params(tau, force_amp=F, force_mode=1)
    ref = o3.stream_pull(o3.step(o3.MLP, g, prm, np.float32(theta).astype(float)))
    bgk = o3.stream_pull(o3.step(o3.BGK, g, prm))
    got = _np(lat.get_state())
    assert wpe(got, ref) <= 1e-5 and wpe(ref, bgk) > 100 * wpe(got, ref)
    assert lat.status() == lbm.LBM_OK


@pytest.mark.parametrize("nx,ny,nz,B", [(127, 1, 1, 1), (43, 3, 1, 1), (16, 16, 1, 1),
                                        (257, 1, 1, 1), (5, 17, 3, 3), (2, 1, 129, 2)])
def test_d3q19_tc_tile_pairs(lbm, nx, ny, nz, B):  # noqa: F811
    """Tensor-core learned D3Q19 step (pairs of 128-node tiles): within 5e-3 of
    the learned correction of the bf16-rounding restatement, as on whole rows."""
    tau, F, m = 0.6, 2e-4, 1
    theta = _weights(24, out_scale=0.01)
    f = field3d(B, nz, ny, nx, seed=51, neq=0.02)
    lat = lbm.Lattice3D(nx, ny, nz, B, tau=tau, force_amp=F, force_mode=m, device=DEV)
    lat.set_state(_dev(f))
    g = o3.stream_push(_np(lat.get_state()))
    th = torch.tensor(theta, dtype=torch.float32, device=DEV)
    lat.step(1, "mlp_bf16", lbm.weights3d_struct(th))
    got = _np(lat.get_state())
    ref = emulate_tc_step(g, theta, tau, F, m)
    bgk = o3.stream_pull(o3.step(o3.BGK, g, o3.params(tau, force_amp=F, force_mode=m)))
    corr = wpe(ref, bgk)
    assert wpe(got, ref) <= 5e-3 * corr and corr > 1e-3
    assert lat.status() == lbm.LBM_OK


def test_d3q19_tc_many_tiles(lbm):  # noqa: F811
    """Every CTA pair walks several tile pairs that span rows and planes: a
    lattice repeated 5 x 5 along x and y evolves as copies of itself, so each
    copy, whatever tiles it falls into, has the bits of the single lattice."""
    nx, ny, nz, r = 60, 26, 2, 5
    f = _dev(field3d(1, nz, ny, nx, seed=52, neq=0.02))
    w = lbm.weights3d_struct(torch.tensor(_weights(25, out_scale=0.0005), dtype=torch.float32,
                                          device=DEV))
    small = lbm.Lattice3D(nx, ny, nz, 1, tau=0.6, device=DEV)
    large = lbm.Lattice3D(nx * r, ny * r, nz, 1, tau=0.6, device=DEV)
    small.set_state(f)
    large.set_state(f.repeat(1, 1, 1, r, r).contiguous())
    for lat in (small, large):
        lat.step(3, "mlp_bf16", w)
        assert lat.status() == lbm.LBM_OK
    assert torch.equal(large.get_state(), small.get_state().repeat(1, 1, 1, r, r))


@pytest.mark.parametrize("kind", ["bgk", "smag"])
@pytest.mark.parametrize("nx,ny,B", [(1, 1, 1), (3, 5, 2), (9, 8, 1), (64, 64, 1), (128, 128, 1),
                                     (129, 128, 1), (61, 300, 1), (16, 1100, 1), (1100, 15, 2),
                                     (181, 97, 3)])
@pytest.mark.parametrize("n", [2, 3, 4, 7, 16, 17])
def test_several_steps_per_launch(lbm, kind, nx, ny, B, n):  # noqa: F811
    """n steps of one call (several steps per launch, recomputed rings around the
    tiles) have the bits of n calls of one step, end in the same buffer, and
    flag an unstable node alike."""
    g = torch.Generator(device=DEV)
    g.manual_seed(nx + 7 * ny + n)
    rnd = lambda: torch.rand((B, ny, nx), generator=g, device=DEV) - 0.5
    rho, ux, uy = 1 + 0.02 * rnd(), 0.1 * rnd(), 0.1 * rnd()
    args = dict(tau=0.53, smag_cs=0.2, force_amp=1e-4, force_mode=1, device=DEV)
    one, many = lbm.Lattice(nx, ny, B, **args), lbm.Lattice(nx, ny, B, **args)
    for fast in (False, True):
        if fast:  # one node beyond the stability limit
            ux[-1, -1, -1] = 0.45
        for lat in (one, many):
            lat.clear_status()
            lat.init_equilibrium(rho, ux, uy)
        for _ in range(n):
            one.step(1, kind)
        many.step(n, kind)
        assert torch.equal(one.get_state(), many.get_state())
        assert (one.state_buffer() == one.bufs[0].data_ptr()) == \
            (many.state_buffer() == many.bufs[0].data_ptr())
        assert one.status() == many.status() == (lbm.LBM_ERR_UNSTABLE if fast else lbm.LBM_OK)


@pytest.mark.parametrize("nx,ny,B,rmax", [(31, 33, 1, 40), (32, 64, 2, 64), (65, 31, 3, 7),
                                          (300, 260, 1, 256), (1, 9, 1, 3)])
def test_structure_function_strips(lbm, nx, ny, B, rmax):  # noqa: F811
    """Structure functions on strips of 32 lines and several positions per block,
    with ragged ends, more separations than the lattice is wide, and one or more
    slices of threads: against FP64 sums over the same FP32 velocities.  Each
    block's FP32 sums have at most 32 terms, so an entry is within 32 half-ulps
    (2^-24) of its sum of absolute terms plus the three or fewer roundings per
    term of its powers: 40 * 2^-24 of that sum."""
    lat = lbm.Lattice(nx, ny, B, device=DEV)
    g = torch.Generator(device=DEV)
    g.manual_seed(nx)
    lat.set_state(torch.rand((B, 9, ny, nx), generator=g, device=DEV) * 0.01 + 0.1)
    S = lat.structure_functions(rmax).cpu().numpy()
    _, ux, uy = (t.cpu().numpy() for t in lat.moments())
    for r in range(1, rmax + 1):
        dx = (np.roll(ux, -r, axis=2) - ux).astype(float)
        dy = (np.roll(uy, -r, axis=1) - uy).astype(float)
        for p in range(1, 7):
            ref = 0.5 * np.mean(dx ** p + dy ** p)
            tol = 40 * 2.0 ** -24 * 0.5 * np.mean(np.abs(dx) ** p + np.abs(dy) ** p)
            assert abs(S[p - 1, r - 1] - ref) <= tol, (p, r)


def test_structure_functions_of_a_blown_up_field(lbm):  # noqa: F811
    """Velocities so large that FP32 running sums overflow: the sums of the even
    powers stay the finite FP64 ones; with an infinite velocity no sum is finite."""
    nx, ny, rmax = 64, 96, 40
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    ux, uy = ((torch.rand((1, ny, nx), generator=g, device=DEV) - 0.5) * 2e6 for _ in range(2))
    f = torch.zeros((1, 9, ny, nx), device=DEV)
    f[:, 0] = 1.0
    f[:, 1], f[:, 3] = ux / 2, -ux / 2   # rho = 1, j = (ux, uy)
    f[:, 2], f[:, 4] = uy / 2, -uy / 2
    lat = lbm.Lattice(nx, ny, 1, device=DEV)
    lat.set_state(f)
    _, vx, vy = (t.cpu().numpy().astype(float) for t in lat.moments())
    S = lat.structure_functions(rmax).cpu().numpy()
    for r in (1, 7, rmax):
        dx, dy = np.roll(vx, -r, axis=2) - vx, np.roll(vy, -r, axis=1) - vy
        for p in (2, 4, 6):
            ref = 0.5 * np.mean(dx ** p + dy ** p)
            assert abs(S[p - 1, r - 1] / ref - 1) <= 40 * 2.0 ** -24
    f[0, 1, 5, 6] = float("inf")
    lat.set_state(f)
    assert not np.isfinite(lat.structure_functions(rmax).cpu().numpy()).any()


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
@pytest.mark.parametrize("nx,ny,B", [(1, 1, 1), (64, 64, 1), (129, 9, 2), (128, 608, 1),
                                     (128, 609, 1), (250, 700, 1)])
def test_tensor_core_steps_of_one_call(lbm, nx, ny, B, dtype):  # noqa: F811
    """Several tensor-core steps of one call (weights laid out once, half-size
    CTAs up to four tiles per SM) have the bits of calls of one step each."""
    g = torch.Generator(device=DEV)
    g.manual_seed(ny)
    f = torch.rand((B, 9, ny, nx), generator=g, device=DEV) * 0.005 + \
        torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, device=DEV).view(1, 9, 1, 1)
    th = torch.tensor(inputs.xavier_mlp(3, bias_scale=0.2, out_scale=0.1), device=DEV)
    w = lbm.weights_struct(th.to(getattr(torch, dtype)))
    one, many = (lbm.Lattice(nx, ny, B, tau=0.6, force_amp=1e-4, force_mode=1, device=DEV)
                 for _ in range(2))
    for lat in (one, many):
        lat.set_state(f)
    for _ in range(5):
        one.step(1, "mlp_bf16", w)
    many.step(5, "mlp_bf16", w)
    assert torch.equal(one.get_state(), many.get_state())
    assert one.status() == many.status() == lbm.LBM_OK


@pytest.mark.parametrize("nx,ny,B", [(1, 1, 1), (127, 1, 1), (43, 3, 1), (16, 8, 2), (257, 1, 1),
                                     (13, 29, 3), (300, 270, 1)])
def test_f32_adjoint_tiles(lbm, nx, ny, B):  # noqa: F811
    """FP32 learned step and its adjoint (tiles of 128 consecutive nodes, two groups
    per CTA; the last shape gives every group several): one recorded step's
    populations, dL/dtheta and dL/df0 against FP64 torch autograd through a
    restatement of the step, 1e-4 relative as in the adjoint's parity tests."""
    from perf import cases as C
    case = dict(path="train", kind="mlp_f32", tau=0.6, force=1e-3, nx=nx, ny=ny, batch=B)
    f0 = C._populations(C._C2, C._W2, 0.03 * torch.randn(2, B, ny, nx, generator=C._gen(nx),
                                                         device=DEV, dtype=torch.float64),
                        C._gen(ny), 0.05)
    theta = torch.tensor(inputs.xavier_mlp(5, bias_scale=0.3, gain=3.0, out_scale=0.02),
                         dtype=torch.float32, device=DEV)
    g = torch.randn((B, 9, ny, nx), generator=C._gen(3), device=DEV, dtype=torch.float64)
    lat = lbm.Lattice(nx, ny, B, tau=0.6, force_amp=1e-3, force_mode=C.MODE_2D, device=DEV)
    lat.set_state(f0)
    ws = torch.empty(lat.record_bytes(1, 1) // 4, dtype=torch.float32, device=DEV)
    w = lbm.weights_struct(theta)
    lat.forward_record(1, 1, w, ws, "f32")
    dW = torch.empty(lbm.LBM_MLP_NPARAMS, dtype=torch.float32, device=DEV)
    dF = torch.empty((B, 9, ny, nx), dtype=torch.float32, device=DEV)
    lat.backward(g.float(), w, ws, dW, dF, "f32")
    f, th = f0.double().requires_grad_(True), theta.double().requires_grad_(True)
    out = C._stream(C._C2, C._collide(case, C._C2, C._W2, f, "bgk", th))
    (out * g.float().double()).sum().backward()
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())
    assert rel(lat.get_state(), out.detach()) <= 1e-6
    assert rel(dW, th.grad) <= 1e-4 and rel(dF, f.grad) <= 1e-4
    assert lat.status() == lbm.LBM_OK


@pytest.mark.parametrize("kind", ["bgk", "smag"])
@pytest.mark.parametrize("nx,ny,nz,B", [(1, 1, 1, 2), (2, 2, 2, 1), (129, 2, 3, 1), (5, 7, 9, 2)])
def test_d3q19_step_strong_flow(lbm, kind, nx, ny, nz, B):  # noqa: F811
    """D3Q19 steps on even and odd parts of opposite pairs, with every velocity
    and force component large: 1e-5 of each weight against the oracle, as in
    the one-step parity test."""
    lat = lbm.Lattice3D(nx, ny, nz, B, tau=0.52, smag_cs=0.3, force_amp=3e-3, force_mode=1,
                        device=DEV)
    lat.set_state(_dev(field3d(B, nz, ny, nx, seed=61, neq=0.05, mean_u=(0.12, -0.15, 0.09))))
    g = o3.stream_push(_np(lat.get_state()))
    lat.step(1, kind)
    prm = o3.params(0.52, smag_cs=0.3, force_amp=3e-3, force_mode=1)
    ref = o3.stream_pull(o3.step(o3.BGK if kind == "bgk" else o3.SMAG, g, prm))
    assert wpe(_np(lat.get_state()), ref) <= 1e-5
    assert lat.status() == lbm.LBM_OK


@pytest.mark.parametrize("nx,ny,B,cg", [(1, 1, 1, 1), (258, 2, 2, 2), (85 * 3 + 3, 9, 1, 3),
                                        (64, 24, 3, 8), (45, 30, 1, 15), (600, 300, 1, 300),
                                        (514, 257, 1, 257)])
def test_box_filter_widths(lbm, nx, ny, B, cg):  # noqa: F811
    """Box filter against the mean in FP64, rounded and added to w the same way:
    at most the next float (2^-24 below 1) where the sums' last bits move a
    rounding; and a block whose sum overflows FP32 but not its mean."""
    lat = lbm.Lattice(nx, ny, B, tau=0.6, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(nx + cg)
    w = torch.tensor(W2, dtype=torch.float32, device=DEV)[None, :, None, None]
    f = w * (1 + 0.1 * torch.randn(B, 9, ny, nx, generator=g, device=DEV))

    def mean(f):
        d = (f - w).double()
        return d.view(B, 9, ny // cg, cg, nx // cg, cg).mean(dim=(3, 5))

    lat.set_state(f)
    got = lat.box_filter(cg)
    ref = mean(f).float() + w
    assert (got - ref).abs().max().item() <= 2.0 ** -24
    if cg > 2:
        f[0, 5, 0, 0] = f[0, 5, cg - 1, cg - 1] = 3e38
        lat.set_state(f)
        got = lat.box_filter(cg)
        ref = mean(f).float() + w
        assert torch.isfinite(ref).all()
        assert ((got - ref).abs() <= 2.0 ** -23 * ref.abs() + 2.0 ** -24).all()
