"""Several plain steps per launch are taken where they are the faster way: n
steps of one call against n calls of one step, both replayed from a CUDA graph
(no host time in either)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("kind", ["bgk", "smag"])
@pytest.mark.parametrize("nx,ny,B", [(16384, 1, 1), (65536, 2, 1), (61, 1000, 1), (4096, 4, 1),
                                     (2, 2, 4096), (64, 64, 256), (128, 128, 64), (64, 16384, 1),
                                     (500, 4000, 1), (64, 64, 1)])
def test_one_call_is_no_slower_than_single_steps(nx, ny, B, kind):
    """15 % for the noise of a minimum over 20 replays of some 60 us."""
    from paper_2403_18466_gb300 import lbm
    s = torch.cuda.Stream(device=DEV)
    lat = lbm.Lattice(nx, ny, B, tau=0.6, smag_cs=0.1, stream=s, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(nx)
    rnd = lambda: 0.02 * torch.randn(B, ny, nx, generator=g, device=DEV)  # noqa: E731
    ux, uy, rho = rnd(), rnd(), torch.ones(B, ny, nx, device=DEV)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        lat.init_equilibrium(rho, ux, uy)
        lat.step(24, kind)
        lat.step(1, kind)
        lat.step(1, kind)
    torch.cuda.synchronize()
    many, one = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(many, stream=s):
        lat.step(24, kind)
    with torch.cuda.graph(one, stream=s):
        for _ in range(24):
            lat.step(1, kind)
    best = {many: 1e9, one: 1e9}
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    with torch.cuda.stream(s):
        for _ in range(20):
            for graph in (many, one):
                ev[0].record(s)
                graph.replay()
                ev[1].record(s)
                ev[1].synchronize()
                best[graph] = min(best[graph], ev[0].elapsed_time(ev[1]) * 1e3)
    assert lat.status() == lbm.LBM_OK
    print(f"{nx} x {ny} x {B} {kind}: {best[many] / 24:.2f} us per step, single {best[one] / 24:.2f}")
    assert best[many] <= 1.15 * best[one]
