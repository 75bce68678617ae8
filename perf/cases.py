"""Workloads of the library for performance measurement, through its public entry points.

A case is a dict of plain values: ``path`` names what the program does, the
rest are its sizes and options.  ``listed()`` are the reference cases,
``draw(rng)`` gives another one of the same ranges, ``prepare`` builds what a
program holds before the call (the lattice, its inputs on the GPU, weights),
``run`` is one pass, ``work`` the bytes and operations that pass cannot do
without, and ``exact`` the same results from a plain FP64 restatement in torch
that shares no code with the library.

Paths
  rollout2d   populations in, n fused steps, populations out (lbm_set_state,
              lbm_step, lbm_get_state): BGK DNS, Smagorinsky LES and the
              learned LES (tensor-core and FP32 networks) all run this way
  dns         one training trajectory cut from a DNS: filtered start state,
              one unroll of fine steps, filtered end state, its velocity and
              its anti-streamed populations (what data.generate does per
              trajectory)
  train       one forward + backward of the unrolled loss (autograd.UnrolledLBM)
  diagnostics energy spectrum and structure functions of a state (les.run)
  rollout3d   as rollout2d on D3Q19, learned kinds with the paper's network
"""
import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_2403_18466_gb300 import inputs, lbm
from paper_2403_18466_gb300.autograd import UnrolledLBM

DEV = "cuda"

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # 64^2 periodic grid, FP32 BGK (the Taylor-Green set-up of the parity
        # tests): the smallest lattice in use, where launches are the cost
        dict(name="bgk_64", path="rollout2d", kind="bgk", nx=64, ny=64, batch=1, n=100,
             tau=0.6, force=0.0),
        # 1024^2 Smagorinsky LES under Kolmogorov forcing, run in blocks of 100
        # steps between status checks
        dict(name="smag_1024", path="rollout2d", kind="smag", nx=1024, ny=1024, batch=1, n=100,
             tau=0.51, force=1e-5),
        # one training trajectory of the 2048^2 BGK DNS at coarse-graining 8 and
        # 16 coarse steps (128 fine steps)
        dict(name="dns_2048", path="dns", nx=2048, ny=2048, cg=8, unroll=16, tau=0.503,
             force=1e-5),
        # the trained LES at the size it was trained for: one 256^2 lattice, one
        # unroll of 16 steps
        dict(name="learned_256", path="rollout2d", kind="mlp_bf16", nx=256, ny=256, batch=1, n=16,
             tau=0.500375, force=8e-5, trained=True),
        # the headline lattice: 4096^2, learned collision on the tensor cores
        dict(name="learned_4096", path="rollout2d", kind="mlp_bf16", nx=4096, ny=4096, batch=1,
             n=20, tau=0.6, force=1e-5, trained=False),
        # FP32 learned collision on a batch of lattices of odd width
        dict(name="learned_f32_ragged", path="rollout2d", kind="mlp_f32", nx=333, ny=250, batch=4,
             n=16, tau=0.6, force=1e-5, trained=False),
        # the training configuration: 32 trajectories of 256^2, 16 steps,
        # checkpoint every 4, velocity loss, tensor-core pair
        dict(name="train_bf16", path="train", precision="bf16", nx=256, ny=256, batch=32, n=16,
             ckpt=4, subset=0, tau=0.500375, force=8e-5),
        # the FP32 pair (the one the committed weights were trained with) on
        # eight trajectories, the population loss on |S| = 512 nodes
        dict(name="train_f32", path="train", precision="f32", nx=256, ny=256, batch=8, n=16,
             ckpt=4, subset=512, tau=0.500375, force=8e-5),
        # statistics of one record of the 1024^2 LES: E(k), k <= 512, and
        # S^p(r), r <= 256
        dict(name="diagnostics_1024", path="diagnostics", nx=1024, ny=1024, batch=1, rmax=256,
             kmax=512),
        # D3Q19 Smagorinsky at 128^3
        dict(name="d3q19_smag_128", path="rollout3d", kind="smag", nx=128, ny=128, nz=128, batch=1,
             n=20, tau=0.51, force=1e-6),
        # the paper's network on the tensor cores at its larger LES size, 64^3
        dict(name="d3q19_learned_64", path="rollout3d", kind="mlp_bf16", nx=64, ny=64, nz=64,
             batch=1, n=16, tau=0.6, force=1e-6),
        # the same network in FP32 at the smaller LES size, 32^3
        dict(name="d3q19_learned_f32_32", path="rollout3d", kind="mlp_f32", nx=32, ny=32, nz=32,
             batch=1, n=4, tau=0.6, force=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, v, to):
    """Half of the sizes as drawn, half rounded to a multiple of `to`."""
    return max(to, v // to * to) if rng.random() < 0.5 else v


# (node, step) pairs that keep a drawn case below the largest listed ones
_STEPS_2D = {"bgk": 600_000_000, "smag": 600_000_000, "mlp_bf16": 300_000_000,
             "mlp_f32": 20_000_000}
_STEPS_3D = {"bgk": 200_000_000, "smag": 200_000_000, "mlp_bf16": 8_000_000, "mlp_f32": 100_000}


def draw(rng):
    path = rng.choice(["rollout2d", "rollout2d", "rollout2d", "rollout3d", "rollout3d", "train",
                       "dns", "diagnostics"])
    if path == "rollout2d":
        kind = rng.choice(["bgk", "smag", "mlp_bf16", "mlp_f32"])
        top = 1024 if kind == "mlp_f32" else 4096
        nx, ny = (_odd(rng, _log_int(rng, 48, top), 64) for _ in range(2))
        batch = rng.choice([1, 1, 1, 2, 3, 4]) if nx * ny < 1 << 20 else 1
        n = min(_log_int(rng, 4, 128), max(1, _STEPS_2D[kind] // (nx * ny * batch)))
        case = dict(path=path, kind=kind, nx=nx, ny=ny, batch=batch, n=n,
                    tau=rng.choice([0.51, 0.6]), force=rng.choice([0.0, 1e-5]))
        if kind.startswith("mlp"):
            case.update(tau=0.6, trained=False)
        return case
    if path == "rollout3d":
        kind = rng.choice(["bgk", "smag", "mlp_bf16", "mlp_f32"])
        top = 32 if kind == "mlp_f32" else 64 if kind == "mlp_bf16" else 160
        nx, ny, nz = (_odd(rng, _log_int(rng, 12, 2 * top if d == 0 else top), 8)
                      for d in range(3))
        n = max(1, min(_log_int(rng, 2, 32), _STEPS_3D[kind] // (nx * ny * nz)))
        return dict(path=path, kind=kind, nx=nx, ny=ny, nz=nz, batch=1, n=n,
                    tau=0.6 if kind.startswith("mlp") else 0.51, force=rng.choice([0.0, 1e-6]))
    if path == "train":
        precision = rng.choice(["bf16", "f32"])
        nx, ny = (_odd(rng, _log_int(rng, 64, 512), 32) for _ in range(2))
        n = rng.choice([8, 12, 16])
        nodes = (30_000_000 if precision == "bf16" else 6_000_000) // n
        return dict(path=path, precision=precision, nx=nx, ny=ny,
                    batch=max(1, min(32, nodes // (nx * ny))), n=n, ckpt=rng.choice([1, 4, 5]),
                    subset=512 if precision == "f32" else 0, tau=0.500375, force=8e-5)
    if path == "dns":
        cg, filt = rng.choice([4, 8]), rng.randint(40, 2048 // 8)
        return dict(path=path, nx=cg * filt, ny=cg * rng.randint(40, 2048 // 8), cg=cg,
                    unroll=rng.choice([8, 12, 16]), tau=0.503, force=1e-5)
    nx, ny = (_odd(rng, _log_int(rng, 200, 1024), 8) for _ in range(2))
    return dict(path=path, nx=nx, ny=ny, batch=1, rmax=rng.randint(40, 256),
                kmax=rng.randint(60, 512))


# ---------------------------------------------------------------- inputs
# Stencils in the order of include/lbm.h and include/lbm3d.h.
_C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_C3 = [(0, 0, 0), (-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 1), (0, 1, 0), (1, 0, 0),
       (-1, -1, 0), (-1, 0, -1), (-1, 0, 1), (-1, 1, 0), (0, -1, -1), (0, -1, 1), (0, 1, -1),
       (0, 1, 1), (1, -1, 0), (1, 0, -1), (1, 0, 1), (1, 1, 0)]
_W3 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12

SMAG_CS, MODE_2D = 0.1, 4


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _wave(n, real=False):
    k = torch.fft.rfftfreq(n) if real else torch.fft.fftfreq(n)
    return (2 * math.pi * k).to(device=DEV, dtype=torch.float64)


def _field2d(batch, ny, nx, g, k0=8.0, urms=0.02):
    """Random-phase divergence-free velocity [2][b][y][x] with the spectrum
    E(k) ~ k^4 exp(-2 (k/k0)^2), in FP64."""
    k0 = min(k0, min(nx, ny) / 12)
    psi = torch.fft.rfft2(torch.randn(batch, ny, nx, generator=g, device=DEV, dtype=torch.float64))
    ky, kx = _wave(ny)[:, None], _wave(nx, real=True)[None, :]
    k = torch.sqrt((ky * ny / (2 * math.pi)) ** 2 + (kx * nx / (2 * math.pi)) ** 2)
    amp = k ** 1.5 * torch.exp(-((k / k0) ** 2)) / k.clamp(min=1e-9)
    psi = psi * amp
    ux = torch.fft.irfft2(1j * ky * psi, s=(ny, nx))
    uy = torch.fft.irfft2(-1j * kx * psi, s=(ny, nx))
    s = urms / torch.sqrt(0.5 * (ux ** 2 + uy ** 2).mean())
    return torch.stack([ux * s, uy * s])


def _field3d(batch, nz, ny, nx, g, k0=4.0, urms=0.02):
    """The same in 3D, as the curl of a random vector potential: [3][b][z][y][x]."""
    k0 = min(k0, min(nx, ny, nz) / 5)
    a = torch.fft.rfftn(torch.randn(3, batch, nz, ny, nx, generator=g, device=DEV,
                                    dtype=torch.float64), dim=(2, 3, 4))
    kz, ky, kx = _wave(nz)[:, None, None], _wave(ny)[None, :, None], _wave(nx, real=True)
    k = torch.sqrt((kz * nz) ** 2 + (ky * ny) ** 2 + (kx * nx) ** 2) / (2 * math.pi)
    a = a * (k * torch.exp(-((k / k0) ** 2)) / k.clamp(min=1e-9))
    u = torch.stack([1j * (ky * a[2] - kz * a[1]), 1j * (kz * a[0] - kx * a[2]),
                     1j * (kx * a[1] - ky * a[0])])
    u = torch.fft.irfftn(u, s=(nz, ny, nx), dim=(2, 3, 4))
    return u * (urms / torch.sqrt((u ** 2).mean()))


def _feq(c, w, rho, u):
    """Equilibrium [b][i][...] of rho [b][...] and u [d][b][...]."""
    usq = (u * u).sum(0)
    out = []
    for ci, wi in zip(c, w):
        cu = sum(a * b for a, b in zip(ci, u) if a)
        out.append(wi * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)
                   if any(ci) else wi * rho * (1 - 1.5 * usq))
    return torch.stack(out, 1)


def _populations(c, w, u, g, neq=0.002):
    """Pre-collision populations: the equilibrium of density fluctuations of
    order |u|^2 and velocity u, times 1 + noise of the size of the
    non-equilibrium part; FP32, as a program holds them."""
    rho = 1 + 3 * ((u * u).sum(0) - (u * u).sum(0).mean())
    f = _feq(c, w, rho, u)
    f *= 1 + neq * (2 * torch.rand(f.shape, generator=g, device=DEV, dtype=torch.float64) - 1)
    return f.float()


def _weights(case, seed):
    if case["path"] == "rollout3d":
        a = inputs.xavier_mlp_widths(seed % 1000, lbm.LBM3D_WIDTHS, bias_scale=0.1, out_scale=0.01)
    elif case["path"] == "train":
        # some epochs into the training: near the trained weights
        a = inputs.trained_mlp()
        a = a * (1 + inputs.noise(a.shape, seed, 0.05))
    elif case["trained"]:
        a = inputs.trained_mlp()
    else:
        a = inputs.xavier_mlp(seed % 1000, out_scale=0.3)
    return torch.tensor(a, dtype=torch.float32, device=DEV)


def _inputs(case, seed):
    """The tensors of a case, made from the seed alone."""
    g = _gen(seed)
    if case["path"] == "rollout3d":
        u = _field3d(case["batch"], case["nz"], case["ny"], case["nx"], g)
        t = {"f0": _populations(_C3, _W3, u, g)}
        if case["kind"].startswith("mlp"):
            t["theta"] = _weights(case, seed)
        return t
    B, ny, nx = case.get("batch", 1), case["ny"], case["nx"]
    u = _field2d(B, ny, nx, g)
    t = {"f0": _populations(_C2, _W2, u, g, 0.01 if case["path"] == "train" else 0.002)}
    if case["path"] == "train":
        v = 0.95 * u + _field2d(B, ny, nx, g, urms=0.002)
        t["utx"], t["uty"] = v[0].float(), v[1].float()
        if case["subset"]:
            # targets of the population loss: post-collision populations of the
            # target velocity, near the ones the unroll ends with
            t["idx"] = torch.randperm(B * ny * nx, generator=g, device=DEV)[:case["subset"]].int()
            t["target"] = _populations(_C2, _W2, v, g)
    if case["path"] == "train" or case.get("kind", "").startswith("mlp"):
        t["theta"] = _weights(case, seed)
    return t


def prepare(case, seed):
    s = {"case": case, **_inputs(case, seed)}
    path = case["path"]
    if path == "rollout3d":
        s["lat"] = lbm.Lattice3D(case["nx"], case["ny"], case["nz"], case["batch"],
                                 tau=case["tau"], smag_cs=SMAG_CS, force_amp=case["force"],
                                 device=DEV)
        s["w"] = lbm.weights3d_struct(s["theta"]) if "theta" in s else None
        return s
    if path == "train":
        s["theta"].requires_grad_(True)
        s["unroll"] = UnrolledLBM(case["nx"], case["ny"], case["batch"], case["tau"], case["n"],
                                  case["ckpt"], case["force"], MODE_2D, device=DEV,
                                  precision=case["precision"])
        return s
    s["lat"] = lbm.Lattice(case["nx"], case["ny"], case.get("batch", 1),
                           tau=case.get("tau", 0.51), smag_cs=SMAG_CS,
                           force_amp=case.get("force", 0.0), force_mode=MODE_2D, device=DEV)
    if path == "dns":
        s["coarse"] = lbm.Lattice(case["nx"] // case["cg"], case["ny"] // case["cg"], 1,
                                  tau=(case["tau"] - 0.5) / case["cg"] + 0.5, device=DEV)
    elif path == "diagnostics":
        s["lat"].set_state(s["f0"])
    else:
        s["w"] = lbm.weights_struct(s["theta"]) if "theta" in s else None
    return s


def run(state):
    case, path = state["case"], state["case"]["path"]
    if path in ("rollout2d", "rollout3d"):
        lat = state["lat"]
        lat.set_state(state["f0"])
        lat.step(case["n"], case["kind"], state["w"])
        return {"f": lat.get_state()}
    if path == "dns":
        dns, coarse, cg = state["lat"], state["coarse"], case["cg"]
        dns.set_state(state["f0"])
        start = dns.box_filter(cg)
        dns.step(cg * case["unroll"], "bgk")
        end = dns.box_filter(cg)
        coarse.set_state(end)
        rho, ux, uy = coarse.moments()
        return {"start": start, "rho": rho, "ux": ux, "uy": uy, "post": coarse.stream(end, -1),
                "f": dns.get_state()}
    if path == "train":
        theta = state["theta"]
        theta.grad = None
        if case["subset"]:
            loss = state["unroll"].loss_subset(theta, state["f0"], state["idx"],
                                               target_post=state["target"])
        else:
            loss = state["unroll"].loss(theta, state["f0"], state["utx"], state["uty"])
        loss.backward()
        return {"loss": loss.detach(), "dtheta": theta.grad}
    lat = state["lat"]
    return {"E": lat.energy_spectrum(case["kmax"]), "S": lat.structure_functions(case["rmax"])}


# ---------------------------------------------------------------- work
_FLOPS_BGK_2D, _FLOPS_SMAG_2D = 150, 185
_FLOPS_BGK_3D, _FLOPS_SMAG_3D = 330, 410
_FLOPS_MLP_2D = 2 * (9 * 64 + 64 * 64 + 64 * 9)
_FLOPS_MLP_3D = 2 * (19 * 300 + 300 * 300 + 300 * 100 + 100 * 19)


def _step_flops(path, kind):
    if path == "rollout3d":
        base = _FLOPS_SMAG_3D if kind == "smag" else _FLOPS_BGK_3D
        return base + (_FLOPS_MLP_3D if kind.startswith("mlp") else 0)
    base = _FLOPS_SMAG_2D if kind == "smag" else _FLOPS_BGK_2D
    return base + (_FLOPS_MLP_2D if kind.startswith("mlp") else 0)


def work(case):
    path = case["path"]
    nodes = case["nx"] * case["ny"] * case.get("nz", 1) * case.get("batch", 1)
    if path in ("rollout2d", "rollout3d"):
        q = 19 if path == "rollout3d" else 9
        return {"bytes": 2 * 4 * q * nodes, "flops": nodes * case["n"]
                * _step_flops(path, case["kind"])}
    if path == "dns":
        coarse = nodes // case["cg"] ** 2
        # state in and out; the filtered start, the coarse moments and the
        # anti-streamed target out
        return {"bytes": 4 * (18 * nodes + (9 + 3 + 9) * coarse),
                "flops": nodes * case["cg"] * case["unroll"] * _FLOPS_BGK_2D}
    if path == "train":
        per_step = _FLOPS_BGK_2D + _FLOPS_MLP_2D
        # forward, and the backward's two products per layer
        read = 9 * nodes + (2 * nodes if not case["subset"] else 10 * case["subset"])
        return {"bytes": 4 * (read + 2 * lbm.LBM_MLP_NPARAMS), "flops": 3 * nodes * case["n"]
                * per_step}
    # statistics: the state in, E and S out; 2 velocity components, a 2D FFT
    # and 2 x rmax increments with 6 powers per node
    flops = nodes * (25 + 2 * 2.5 * math.log2(nodes) + 2 * case["rmax"] * 12)
    return {"bytes": 36 * nodes + 8 * (case["kmax"] + 1 + 6 * case["rmax"]), "flops": flops}


# ---------------------------------------------------------------- exact
# A plain FP64 restatement of the method (see include/lbm.h): pull-stream,
# collide, EDM force, one whole-array torch operation after another.


def _stream(c, f, sign=1):
    """f_i(x) <- f_i(x - sign c_i) of [b][i][...] (axes in reverse: x is last)."""
    dims = tuple(range(2, f.dim()))[::-1]
    return torch.stack([torch.roll(f[:, i], tuple(sign * a for a in ci), tuple(d - 1 for d in dims))
                        if any(ci) else f[:, i] for i, ci in enumerate(c)], 1)


def _moments(c, f):
    rho = f.sum(1)
    u = torch.stack([sum(ci[a] * f[:, i] for i, ci in enumerate(c) if ci[a]) / rho
                     for a in range(len(c[0]))])
    return rho, u


def _act(c):
    return torch.tanh if len(c) == 9 else lambda a: torch.nn.functional.leaky_relu(a, 0.01)


def _network(c, theta, x):
    """o [..., Q] of x [..., Q] through the packed MLP."""
    q = len(c)
    dims = [9, 64, 64, 9] if q == 9 else [19, 300, 300, 100, 19]
    at = 0
    for k, (n_in, n_out) in enumerate(zip(dims[:-1], dims[1:])):
        W = theta[at:at + n_in * n_out].view(n_out, n_in)
        b = theta[at + n_in * n_out:at + n_in * n_out + n_out]
        at += n_in * n_out + n_out
        x = x @ W.T + b
        if k + 2 < len(dims):
            x = _act(c)(x)
    return x


def _correction(c, theta, f, feq, rho):
    """rho P o of the learned collision (before its 1/tau), [b][i][...]."""
    x = ((f - feq) / rho[:, None]).movedim(1, -1)
    shape = x.shape
    x = x.reshape(-1, len(c))
    part = 1 << (20 if len(c) == 9 else 17)
    if torch.is_grad_enabled() and theta.requires_grad:
        o = _network(c, theta, x)
    else:
        o = torch.cat([_network(c, theta, p) for p in x.split(part)])
    cc = torch.tensor(c, dtype=torch.float64, device=DEV)
    basis = torch.cat([torch.ones(len(c), 1, dtype=torch.float64, device=DEV), cc], 1)
    o = o - (o @ basis / (basis * basis).sum(0)) @ basis.T
    return rho[:, None] * o.reshape(shape).movedim(-1, 1)


def _force(case, c):
    """Body force per axis, broadcastable against [b][...]."""
    F, d = case.get("force", 0.0), len(c[0])

    def wave(n, mode):
        a = torch.arange(n, device=DEV, dtype=torch.float64)
        # the library holds the force table in FP32
        return (F * torch.sin(2 * math.pi * mode * a / n)).float().double()

    if d == 2:
        return [wave(case["ny"], MODE_2D)[None, :, None], None]
    return [wave(case["ny"], 1)[None, None, :, None], wave(case["nz"], 1)[None, :, None, None],
            wave(case["nx"], 1)[None, None, None, :]]


def _collide(case, c, w, f, kind, theta=None):
    rho, u = _moments(c, f)
    feq = _feq(c, w, rho, u)
    tau = case["tau"]
    if kind == "smag":
        d = len(c[0])
        ne = f - feq
        pp = 0
        for a in range(d):
            for b in range(d):
                p = sum(ci[a] * ci[b] * ne[:, i] for i, ci in enumerate(c) if ci[a] * ci[b])
                pp = pp + p * p
        tau = 0.5 * (tau + torch.sqrt(tau * tau + 18 * SMAG_CS ** 2 * torch.sqrt(2 * pp) / rho))
        tau = tau[:, None]
    out = f + (feq - f) / tau
    if theta is not None:
        out = out + _correction(c, theta, f, feq, rho) / tau
    if case.get("force", 0.0):
        us = torch.stack([u[a] + (Fa / rho if Fa is not None else 0)
                          for a, Fa in enumerate(_force(case, c))])
        out = out + _feq(c, w, rho, us) - feq
    return out


def _rollout(case, c, w, f, n, kind, theta=None):
    for _ in range(n):
        f = _stream(c, _collide(case, c, w, f, kind, theta))
    return f


def _box(f, cg):
    B, q, ny, nx = f.shape
    return f.reshape(B, q, ny // cg, cg, nx // cg, cg).mean((3, 5))


def _exact_train(case, t):
    theta = t["theta"].double().requires_grad_(True)
    f = t["f0"].double()

    def step(a, th):
        return _collide(case, _C2, _W2, a, "bgk", th)

    post = None
    for k in range(case["n"]):
        post = checkpoint(step, f, theta, use_reentrant=False)
        f = _stream(_C2, post)
    if case["subset"]:
        i = t["idx"].long()
        rows = post.movedim(1, -1).reshape(-1, 9)[i]
        want = t["target"].double().movedim(1, -1).reshape(-1, 9)[i]
        loss = ((rows - want) ** 2).sum()
    else:
        _, u = _moments(_C2, f)
        loss = 0.5 * ((u[0] - t["utx"].double()) ** 2 + (u[1] - t["uty"].double()) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "dtheta": theta.grad}


def _exact_diagnostics(case, t):
    _, u = _moments(_C2, t["f0"].double())
    B, ny, nx = u.shape[1:]
    uh = torch.fft.fft2(u)
    ky = torch.fft.fftfreq(ny, 1 / ny, device=DEV, dtype=torch.float64)[:, None]
    kx = torch.fft.fftfreq(nx, 1 / nx, device=DEV, dtype=torch.float64)[None, :]
    shell = torch.round(torch.sqrt(ky ** 2 + kx ** 2)).long().reshape(-1)
    e = 0.5 * (uh.real ** 2 + uh.imag ** 2).sum((0, 1)).reshape(-1) / ((nx * ny) ** 2 * B)
    E = torch.zeros(int(shell.max()) + 1, dtype=torch.float64, device=DEV)
    E.index_add_(0, shell, e)
    if len(E) <= case["kmax"]:
        E = torch.cat([E, E.new_zeros(case["kmax"] + 1 - len(E))])
    S = torch.empty(6, case["rmax"], dtype=torch.float64, device=DEV)
    for r in range(1, case["rmax"] + 1):
        dx = torch.roll(u[0], -r, 2) - u[0]
        dy = torch.roll(u[1], -r, 1) - u[1]
        px, py = dx, dy
        for p in range(6):
            S[p, r - 1] = 0.5 * (px.mean() + py.mean())
            px, py = px * dx, py * dy
    return {"E": E[:case["kmax"] + 1], "S": S}


def exact(case, seed):
    t = _inputs(case, seed)
    path = case["path"]
    if path == "train":
        return _exact_train(case, t)
    if path == "diagnostics":
        return _exact_diagnostics(case, t)
    with torch.no_grad():
        if path == "dns":
            f = t["f0"].double()
            start = _box(f, case["cg"])
            f = _rollout(case, _C2, _W2, f, case["cg"] * case["unroll"], "bgk")
            end = _box(f, case["cg"])
            rho, u = _moments(_C2, end)
            return {"start": start, "rho": rho, "ux": u[0], "uy": u[1],
                    "post": _stream(_C2, end, -1), "f": f}
        c, w = (_C3, _W3) if path == "rollout3d" else (_C2, _W2)
        theta = t["theta"].double() if "theta" in t else None
        return {"f": _rollout(case, c, w, t["f0"].double(), case["n"], case["kind"], theta)}
