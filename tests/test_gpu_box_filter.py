"""The box filter at a coarse-graining of 1 is a copy of the populations, and costs
no more than one."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("nx,ny,B", [(1, 1, 1), (129, 3, 2), (5, 300, 2), (1024, 1024, 1)])
def test_blocks_of_one_node(nx, ny, B):
    """The populations themselves (get_state), infinite ones too; at 1024^2, where a
    pass takes some 50 us, within 15 % of the subsampling filter's time."""
    from paper_2403_18466_gb300 import lbm
    lat = lbm.Lattice(nx, ny, B, tau=0.6, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(nx)
    f = torch.rand((B, 9, ny, nx), generator=g, device=DEV)
    f[0, 3, 0, 0] = float("inf")
    lat.set_state(f)
    out, ref = lat.box_filter(1), lat.get_state()
    assert torch.equal(out, ref) and torch.isinf(out[0, 3, 0, 0])
    if nx < 1024:
        return
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    best = {}
    for fn in (lat.box_filter, lat.subsample) * 5:
        ev[0].record()
        for _ in range(20):
            fn(1, out)
        ev[1].record()
        ev[1].synchronize()
        best[fn.__name__] = min(best.get(fn.__name__, 1e9), ev[0].elapsed_time(ev[1]) * 50)
    print(best)
    assert best["box_filter"] <= 1.15 * best["subsample"]
