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


def test_tanh_of_the_fp32_networks(lbm):
    """tanh of the FP32 learned collision against tanhf, band by band: no larger
    root mean square and maximum error against FP64.  The collision of one step
    is made to show it: with populations d = (0, e, -e, e, -e, 0, ...) about rest
    the input is x = d; the first layer hands on tanh(x_1) = x_1 (|e| < 2^-13),
    the second takes tanh(2^17 x_1), and the last writes that along the same
    pattern, which the conservation layer keeps, so with tau = 1 the second
    population is tanh(2^17 e), rounded nowhere else."""
    n = 1024
    theta = np.zeros(lbm.LBM_MLP_NPARAMS, np.float32)
    w1, w2, w3 = 0, 64 * 9 + 64, 64 * 9 + 64 + 64 * 64 + 64
    theta[w1 + 1] = 1.0
    theta[w2] = 2.0 ** 17
    for i, v in ((1, 1), (2, -1), (3, 1), (4, -1)):
        theta[w3 + 64 * i] = v
    w = lbm.weights_struct(torch.tensor(theta, device=DEV))
    lat = lbm.Lattice(n, n, 1, tau=1.0, device=DEV)
    shift = {1: (1, 0), 2: (0, 1), 3: (-1, 0), 4: (0, -1)}  # c_x, c_y

    def tanh2(a):
        e = a * 2.0 ** -17
        st = lat.state_tensor()
        st.zero_()
        for i, (cx, cy) in shift.items():  # the step pulls d_i(x) = state_i(x - c_i)
            st[0, i] = torch.roll(e if i % 2 else -e, (-cy, -cx), (0, 1))
        lat.step(1, "mlp_f32", w)
        return lat.state_tensor()[0, 1].clone()

    for bands in ([(0, 0.55), (0.55, 0.8), (0.8, 0.9), (0.9, 1), (1, 1.2), (1.2, 1.6), (1.6, 2),
                   (2, 9)], [(0, 0.8), (0.8, 3.8), (3.8, 9), (0, 9)]):
        for lo, hi in bands:
            err = [[], []]
            for k in range(4):
                u = (torch.arange(n * n, device=DEV, dtype=torch.float64) + k / 4 + 0.125) / (n * n)
                a = (lo + (hi - lo) * u).float()
                a[1::2] *= -1
                a = a.view(n, n)
                ref = torch.tanh(a.double())
                for out, f in zip(err, (tanh2(a), torch.tanh(a))):
                    out.append(((f.double() - ref) / ref * 2.0 ** 24).abs().max().item())
                    out.append(((f.double() - ref) / ref * 2.0 ** 24).square().mean().item())
            rms = [np.sqrt(np.mean(e[1::2])) for e in err]
            top = [max(e[::2]) for e in err]
            msg = f"[{lo}, {hi}): rms {rms[0]:.3f} / {rms[1]:.3f}, max {top[0]:.2f} / {top[1]:.2f}"
            print(msg)
            assert rms[0] <= rms[1], msg
            # a maximum over 4 M points is itself a sample: 10 %
            assert top[0] <= 1.1 * top[1], msg
    a = torch.zeros(n, n, device=DEV)
    special = torch.tensor([40.0, -40.0, 0.0, -0.0, 1e30, -1e30], device=DEV)
    a[0, 2:8] = special
    assert torch.equal(tanh2(a)[0, 2:8], torch.tanh(special))
    assert lat.status() == lbm.LBM_OK
    theta[w1 + 1] = 3e38  # an infinite pre-activation in the first layer
    w = lbm.weights_struct(torch.tensor(theta, device=DEV))
    a[0, 2:8] = torch.tensor([1.0, -1.0, float("nan"), 1.0, -1.0, 0.0]) * 2.0 ** 21
    got = tanh2(a)[0, 2:8]
    assert torch.equal(got[[0, 1, 3, 4]], torch.tensor([1.0, -1.0, 1.0, -1.0], device=DEV))
    assert torch.isnan(got[2])
