"""Sums and functions that stand in place of wider or slower ones, each against
what it replaces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


@pytest.fixture(scope="module")
def lbm():
    from paper_2403_18466_gb300 import lbm as m
    return m


def test_structure_function_running_sums_hold_a_double(lbm):
    """S^1 of a field whose running sums need 50 bits.  At separation 16 a thread
    meets, in rows 0, 4, 8 and 28 of its strip, the increments A, s1, s2 and -A
    with A about 2^20 and s2 = 3 2^-29 (the -A, -s1, -s2 that complete them lie
    in other blocks, s1 and s2 without A).  Every sum of 32 nodes is exact, and
    so is every FP64 sum of them, so S^1(16) is exactly 0; a running sum that
    drops a bit of s1 + s2 beside A leaves 2^-29 behind."""
    nx, ny, r = 128, 32, 16
    w = np.float32(W)
    f = np.broadcast_to(w[:, None, None], (9, ny, nx)).copy()
    A, e = np.float32(2.0 ** 20), np.float32(3 * 2.0 ** -29)
    for row, sign in ((0, 1), (28, -1)):
        for x in (40, 56, 72):
            f[1, row, x], f[3, row, x] = sign * A / 2, -sign * A / 2
    f[1, 4, 40], f[3, 4, 40] = w[1] + np.float32(0.025), w[3] - np.float32(0.025)
    f[5, 8, 40] = w[5] + e
    lat = lbm.Lattice(nx, ny, 1, device=DEV)
    lat.set_state(torch.tensor(f[None], device=DEV))
    _, ux, uy = (t.cpu().numpy()[0].astype(float) for t in lat.moments())
    s1, s2, big = ux[4, 40], ux[8, 40], ux[0, 40]
    assert s2 == 3 * 2.0 ** -29 and 2.0 ** -5 < s1 < 2.0 ** -4 - s2 and big > 2.0 ** 20
    assert ux[28, 40] == -big and np.float32(s1 + s2) != s1 + s2  # 25 bits
    assert (big + s1 + s2) - big == s1 + s2                       # FP64 holds all of them
    S = lat.structure_functions(256).cpu().numpy()
    assert S[0, r - 1] == 0.0
