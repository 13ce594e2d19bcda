"""Performance cases of the entropic Fourier collision library: what a user's program has it do.

Every case goes through the public Python binding (one call per C entry point) on one GPU.  The
inputs are the repository's synthetic distributions (Maxwellians with bumps, BKW solutions), drawn
on the GPU from the seed.  ``exact`` restates the method in plain torch, FP64, with torch's FFT:

    Q = sum_e a_e S_e - F nu,   a_e = IFFT(M_e Fh),  S_e = IFFT(sum_c w_c M_{e*_c} Fh),  nu = IFFT(L Fh)

with M_u(l) = sigma(l) Phi_u(l . e_u), the modified Jackson filter sigma and the low-rank angular
decomposition of the kernel (arXiv:1704.07369, Secs. 3.2 and 4.1).
"""
import math
import random

import numpy as np
import torch

import paper_1704_07369_gb300 as ef

DEV = "cuda:0"
SIZES = (8, 12, 16, 24, 32, 40, 48, 64)      # grid points per axis the library is built for
RAGGED = (24, 32, 40, 48)                    # sizes of the batched workload
AUDIT = 0.02                                 # share of the cells that the surrogate's audit hands to the plain operator
BAND = 6                                     # |k| <= 6: the surrogate's band
QUAD = {8: (1, 2, 2), 16: (1, 4, 2), 32: (2, 4, 2), 64: (2, 4, 4)}   # 3D rank -> (n_mu, n_phi, n_c)
RES = {"F32": torch.float32, "F64": torch.float64}


def listed():
    return [
        # the 2D model problem: one cell, 100 forward-Euler steps, every step's diagnostics kept
        dict(name="euler_2d_n16_f64_1cell", kind="euler", d=2, N=16, cells=1, kernel="maxwell", R=16, L=8.0, prec="F64", steps=100, dt=0.01, diag=True),
        # the paper's integrator (SSP-RK3) at the finest 2D grid of its convergence tables, a few initial states at once
        dict(name="rk3_2d_n64_f64_4cells", kind="rk3", d=2, N=64, cells=4, kernel="maxwell", R=16, L=8.0, prec="F64", steps=2, dt=0.01),
        # one evaluation of Q for one 3D cell: the smallest 3D call, all latency
        dict(name="collide_n32_f32_1cell", kind="collide", d=3, N=32, cells=1, kernel="maxwell", R=32, L=8.0, prec="F32"),
        # a homogeneous 3D relaxation (BKW) in FP64: one cell, steps with diagnostics
        dict(name="euler_n32_f64_1cell", kind="euler", d=3, N=32, cells=1, kernel="maxwell", R=32, L=8.0, prec="F64", steps=2, dt=0.01, diag=True),
        # a spatially inhomogeneous run: transport between an odd number of cells and collisions, split, then the moments
        dict(name="inhomogeneous_n24_333cells", kind="inhomogeneous", d=3, N=24, cells=333, kernel="hard_sphere", R=16, L=8.0, prec="F32", steps=2, dt=0.005),
        # a small adaptive-grid batch (a rank's share, or one chunk of a streamed batch): uneven N, Euler with diagnostics
        dict(name="ragged_f32_67cells", kind="ragged", d=3, N=0, cells=67, kernel="hard_sphere", R=32, L=8.0, prec="F32", steps=1, dt=0.005, diag=True),
        # the batched workload of the benchmark: 4096 cells of N in {24, 32, 40, 48}, one Euler step with diagnostics
        dict(name="ragged_f32_4096cells", kind="ragged", d=3, N=0, cells=4096, kernel="hard_sphere", R=32, L=8.0, prec="F32", steps=1, dt=0.005, diag=True),
        # training data of the surrogate: Q of a chunk of cells on one grid
        dict(name="collide_n32_f32_2048cells", kind="collide", d=3, N=32, cells=2048, kernel="hard_sphere", R=32, L=8.0, prec="F32"),
        # the precision study's grid in FP32 ...
        dict(name="collide_n64_f32_256cells", kind="collide", d=3, N=64, cells=256, kernel="hard_sphere", R=64, L=10.0, prec="F32"),
        # ... and in FP64 (fewer cells: the same pass is over ten times longer)
        dict(name="collide_n64_f64_24cells", kind="collide", d=3, N=64, cells=24, kernel="hard_sphere", R=64, L=10.0, prec="F64"),
        # the learned surrogate in production: two networks, 2% of the cells audited (the plain operator's Q is delivered for them), Q on the grid
        dict(name="surrogate_n32_16384cells", kind="surrogate", d=3, N=32, cells=16384, kernel="hard_sphere", R=32, L=8.0, prec="F32", hidden=512, layers=4),
        # one training batch of the surrogate's network: loss and gradients
        dict(name="mlp_grad_batch1024", kind="mlp_grad", d=3, N=0, cells=1024, kernel="", R=0, L=8.0, prec="F32", hidden=512, layers=4),
    ]


# ------------------------------------------------------------------ drawn cases ------------

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges; a pass costs no more than the largest listed one."""
    kind = rng.choice(["collide", "collide", "euler", "euler", "ragged", "rk3", "inhomogeneous", "surrogate", "mlp_grad"])
    if kind == "mlp_grad":
        return dict(kind=kind, d=3, N=0, cells=64 * _log_int(rng, 1, 32), kernel="", R=0, L=8.0, prec="F32",
                    hidden=rng.choice([256, 512, 768]), layers=rng.choice([3, 4]))
    if kind == "surrogate":
        return dict(kind=kind, d=3, N=rng.choice([24, 32]), cells=64 * _log_int(rng, 4, 200), kernel="hard_sphere", R=32, L=8.0,
                    prec="F32", hidden=rng.choice([256, 512]), layers=rng.choice([3, 4]))
    if kind == "ragged":
        return dict(kind=kind, d=3, N=0, cells=_log_int(rng, 8, 3500), kernel="hard_sphere", R=rng.choice([16, 32]), L=8.0,
                    prec="F32", steps=1, dt=0.005, diag=rng.random() < 0.7)
    d = 3 if rng.random() < 0.75 else 2
    prec = "F32" if rng.random() < 0.65 else "F64"
    case = dict(kind=kind, d=d, N=rng.choice(SIZES), cells=1, kernel="maxwell", R=rng.choice([8, 16, 32]), L=8.0, prec=prec)
    if d == 3:
        # Maxwell molecules in 3D take 6 times the directions; their tables are for grids up to 32 here
        if case["N"] > 32 or rng.random() < 0.7:
            case["kernel"] = "hard_sphere"
        case["R"] = rng.choice([16, 32, 64])
        if case["R"] == 64:
            case["L"] = 10.0
    if kind == "collide":
        steps = 1
    else:
        steps = rng.choice([1, 2, 4])
        case["steps"], case["dt"] = steps, 0.005
    if kind == "euler":
        case["diag"] = rng.random() < 0.5
    one = _flops_cell(case) * steps * (3 if kind == "rk3" else 1) * (30.0 if prec == "F64" else 1.0)
    top = _flops(listed()[6]) * 0.8
    points = case["N"] ** d * (8 if prec == "F64" else 4)
    case["cells"] = _log_int(rng, 2 if kind == "inhomogeneous" else 1, max(2, min(int(top / one), int(4e9 / points), 40000)))
    return case


# ------------------------------------------------------------------ work -------------------

def _sizes(case):
    """Grid sizes of the cells of a ragged batch (the batch's own, not the seed's)."""
    rng = random.Random(case["cells"])
    return [rng.choice(RAGGED) for _ in range(case["cells"])]


def _first_directions(case):
    if case["d"] == 2:
        return case["R"] // 2
    nmu, nphi, _ = QUAD[case["R"]]
    return nmu * nphi * (6 if case["kernel"] == "maxwell" else 1)


def _flops_cell(case, N=None):
    """One forward real transform, two inverse ones per first direction and one for the loss, and the products."""
    N = N or case["N"]
    pts = N ** case["d"]
    ne = _first_directions(case)
    return (2 * ne + 2) * 2.5 * pts * math.log2(pts) + (2 * ne + 1) * pts + 2 * ne * pts


def _flops(case):
    if case["kind"] == "ragged":
        return sum(_flops_cell(case, N) for N in _sizes(case)) * case["steps"]
    return _flops_cell(case) * case["cells"]


def _widths(case):
    nf = 926
    return [nf + 2] + [case["hidden"]] * (case["layers"] - 1) + [nf]


def work(case):
    el = 8 if case["prec"] == "F64" else 4
    kind, cells = case["kind"], case["cells"]
    if kind == "mlp_grad":
        w = _widths(case)
        par = sum(a * b + b for a, b in zip(w, w[1:]))
        # forward, weight gradient and input gradient (none for the first layer)
        mul = sum(a * b * (3 if i else 2) for i, (a, b) in enumerate(zip(w, w[1:])))
        return {"bytes": 4.0 * (cells * (w[0] + w[-1]) + 2 * par), "flops": 2.0 * mul * cells}
    if kind == "surrogate":
        w = _widths(case)
        pts = case["N"] ** 3
        par = sum(a * b + b for a, b in zip(w, w[1:]))
        net = 2.0 * sum(a * b for a, b in zip(w, w[1:]))
        band = 2 * 2.5 * pts * math.log2(pts)           # the band of F, and the band back to the grid
        plain = 0.02 * _flops_cell(case)
        return {"bytes": float(cells * (8 * pts + 928 * 4 + 8) + 8 * par), "flops": cells * (2 * net + band + plain)}
    if kind == "ragged":
        pts = sum(N ** 3 for N in _sizes(case))
        return {"bytes": float(case["steps"] * (2 * el * pts + (80 * cells if case["diag"] else 0))), "flops": _flops(case)}
    pts = cells * case["N"] ** case["d"]
    if kind == "collide":
        return {"bytes": float(2 * el * pts), "flops": _flops(case)}
    if kind == "euler":
        # several steps of one batch: its state once in and once out, the diagnostics of every step
        return {"bytes": float(2 * el * pts + (80 * cells * case["steps"] if case["diag"] else 0)), "flops": _flops(case) * case["steps"]}
    if kind == "rk3":
        return {"bytes": float(2 * el * pts), "flops": 3 * _flops(case) * case["steps"]}
    # inhomogeneous: each step reads and writes the batch, the moments come from the last one
    return {"bytes": float(2 * el * pts * case["steps"] + 80 * cells), "flops": (_flops(case) + 3 * pts) * case["steps"] + 12 * pts}


# ------------------------------------------------------------------ inputs -----------------

def _axis(N, L):
    return (torch.arange(N, device=DEV, dtype=torch.float64) - N // 2) * (2.0 * L / N)


def _ball(rng, n, d, radius):
    x = rng.normal(size=(n, d))
    return x / np.linalg.norm(x, axis=1, keepdims=True) * radius * rng.uniform(size=(n, 1)) ** (1.0 / d)


def _gauss(v, c, s2, d):
    """exp(-|v - c|^2 / (2 s2)) on the grid for every cell: c [n, d], s2 [n]."""
    out = None
    for a in range(d):
        g = torch.exp(-((v[None, :] - c[:, a:a + 1]) ** 2) / (2 * s2[:, None]))
        g = g.reshape((-1,) + (1,) * a + (v.numel(),) + (1,) * (d - 1 - a))
        out = g if out is None else out * g
    return out


def _mixtures(d, N, L, n, rng):
    """Maxwellians (density and temperature U[0.5, 2], |u| <= 1) times (1 + 0.3 sum of three bumps), renormalised."""
    rho, th, u = rng.uniform(0.5, 2.0, n), rng.uniform(0.5, 2.0, n), _ball(rng, n, d, 1.0)
    ctr = [u + _ball(rng, n, d, 1.0) * (2.0 * np.sqrt(th))[:, None] for _ in range(3)]
    wid = [rng.uniform(0.3, 1.0, n) for _ in range(3)]
    v, h = _axis(N, L), 2.0 * L / N
    out = torch.empty((n,) + (N,) * d, device=DEV, dtype=torch.float64)
    step = max(1, 2 ** 25 // N ** d)
    for a in range(0, n, step):
        s = slice(a, min(n, a + step))
        t = lambda x: torch.as_tensor(x[s], device=DEV)  # noqa: E731
        F = _gauss(v, t(u), t(th), d)
        F = F * (1.0 + 0.3 * sum(_gauss(v, t(c), t(w) ** 2, d) for c, w in zip(ctr, wid)))
        out[s] = F * (t(rho) / (F.flatten(1).sum(1) * h ** d)).reshape((-1,) + (1,) * d)
    return out


def _bkw(d, N, L, n, rng, t_lo, t_hi, spread):
    """BKW solutions at times U[t_lo, t_hi]; with ``spread`` also density, temperature U[0.5, 2] and |u| <= 1."""
    t0 = rng.uniform(t_lo, t_hi, n)
    rho, th = (rng.uniform(0.5, 2.0, n), rng.uniform(0.5, 2.0, n)) if spread else (np.ones(n), np.ones(n))
    u = _ball(rng, n, d, 1.0) if spread else np.zeros((n, d))
    v = _axis(N, L)
    out = torch.empty((n,) + (N,) * d, device=DEV, dtype=torch.float64)
    step = max(1, 2 ** 25 // N ** d)
    for a in range(0, n, step):
        s = slice(a, min(n, a + step))
        col = lambda x: torch.as_tensor(x[s], device=DEV).reshape((-1,) + (1,) * d)  # noqa: E731
        T = col(th)
        S = 1.0 - (torch.exp(-col(t0 * rho) / 8.0) / 2.0 if d == 2 else 0.4 * torch.exp(-col(t0 * rho) / 6.0))
        v2 = sum(((v[None, :] - torch.as_tensor(u[s, a2], device=DEV)[:, None]) ** 2).reshape((-1,) + (1,) * a2 + (N,) + (1,) * (d - 1 - a2))
                 for a2 in range(d)) / T
        if d == 2:
            p = torch.exp(-v2 / (2 * S)) / (2 * math.pi * S) * ((2 * S - 1) / S + (1 - S) / (2 * S * S) * v2)
        else:
            p = torch.exp(-v2 / (2 * S)) / (2 * math.pi * S) ** 1.5 * ((5 * S - 3) / (2 * S) + (1 - S) / (2 * S * S) * v2)
        out[s] = col(rho) * T ** (-d / 2.0) * p
    return out


def _cells(case, seed):
    """The case's cells in FP64 (a list of arrays, one per size, for a ragged batch)."""
    rng = np.random.default_rng(seed)
    d, L, n = case["d"], case["L"], case["cells"]
    if case["kind"] == "ragged":
        Ns = np.array(_sizes(case))
        return {int(N): _mixtures(3, int(N), L, int((Ns == N).sum()), rng) for N in sorted(set(Ns.tolist()))}
    if case["kind"] == "surrogate":
        return _bkw(d, case["N"], L, n, rng, 0.5, 10.0, True)
    if case["kernel"] == "maxwell":
        return _bkw(d, case["N"], L, n, rng, 1.0, 6.0 if n == 1 else 3.0, n > 1)
    return _mixtures(d, case["N"], L, n, rng)


def _packed(case, by_size, dtype):
    """Cells back to back in batch order."""
    Ns = _sizes(case)
    out = torch.empty(sum(N ** 3 for N in Ns), device=DEV, dtype=dtype)
    at, taken = 0, dict.fromkeys(by_size, 0)
    for N in Ns:
        out[at:at + N ** 3] = by_size[N][taken[N]].reshape(-1)
        taken[N] += 1
        at += N ** 3
    return out


def _plan(case, **ex):
    prec = ef.EF_PREC_F64 if case["prec"] == "F64" else ef.EF_PREC_F32
    kernel = ef.EF_KERNEL_MAXWELL if case["kernel"] == "maxwell" else ef.EF_KERNEL_HARD_SPHERE
    return ef.Plan(case["d"], case["N"], case["L"], kernel, case["R"], prec, **ex)


# ------------------------------------------------------------------ the surrogate's network --

def _network(case, seed):
    """He-normal weights and small biases, [out, in] per layer, FP32."""
    rng = np.random.default_rng([seed, 77])
    w = _widths(case)
    out = []
    for i, (a, b) in enumerate(zip(w, w[1:])):
        s = math.sqrt(2.0 / a) * (0.5 if i == len(w) - 2 else 1.0)
        out.append(((rng.standard_normal((b, a)) * s).astype(np.float32), (rng.standard_normal(b) * 0.01).astype(np.float32)))
    return out


def _mlp(case, net, batch):
    w = _widths(case)
    mlp = ef.MLP(w[0], case["hidden"], case["layers"], w[-1], batch, seed=0)
    flat = np.zeros(mlp.nparams, dtype=np.float32)
    for (woff, op, ip, boff), (W, b) in zip(mlp.layout(), net):
        flat[woff:woff + op * ip].reshape(op, ip)[:W.shape[0], :W.shape[1]] = W
        flat[boff:boff + b.size] = b
    mlp.set_params(flat)
    return mlp


def _forward64(net, X):
    """The network in FP64 with its weights as they are stored for the products (bf16)."""
    for i, (W, b) in enumerate(net):
        W = torch.as_tensor(W, device=DEV).bfloat16().double()
        X = X @ W.T + torch.as_tensor(b, device=DEV).double()
        X = torch.relu(X) if i < len(net) - 1 else X
    return X


def _audited(n):
    """Cells that the seeded audit (seed 1) hands to the plain operator."""
    with np.errstate(over="ignore"):
        z = np.uint64(1) + np.uint64(0x9E3779B97F4A7C15) * np.arange(1, n + 1, dtype=np.uint64)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    return np.flatnonzero((z >> np.uint64(40)).astype(np.float64) / 2 ** 24 < np.float64(np.float32(AUDIT)))


def _modes():
    """Band modes |k| <= 6 of the canonical half space, lexicographic; and the slot of k = 0."""
    K = BAND
    ks = [(a, b, c) for a in range(-K, K + 1) for b in range(-K, K + 1) for c in range(K + 1)
          if a * a + b * b + c * c <= K * K and (c > 0 or b > 0 or (b == 0 and a >= 0))]
    return np.array(ks), ks.index((0, 0, 0))


def _band(F):
    """Complex band coefficients [n, modes] of cells [n, N, N, N] (index-origin convention)."""
    ks, _ = _modes()
    N = F.shape[1]
    k = torch.as_tensor(ks, device=DEV) % N
    out = torch.empty(F.shape[0], len(ks), device=DEV, dtype=torch.complex128)
    for a in range(0, F.shape[0], 512):
        h = torch.fft.fftn(F[a:a + 512].double(), dim=(1, 2, 3)) / N ** 3
        out[a:a + 512] = h[:, k[:, 0], k[:, 1], k[:, 2]]
    return out


def _moments64(F, L):
    """mass, momentum, energy and entropy sums of cells [n, N, N, N], FP64."""
    N = F.shape[1]
    v, h3 = _axis(N, L), (2.0 * L / N) ** 3
    rows = []
    for a in range(0, F.shape[0], 512):
        f = F[a:a + 512].double()
        x, y, z = f.sum((2, 3)), f.sum((1, 3)), f.sum((1, 2))
        e = (x @ v ** 2 + y @ v ** 2 + z @ v ** 2) / 2
        eta = torch.where(f > 0, f * torch.log(f.clamp_min(1e-300)), 0.0).sum((1, 2, 3))
        rows.append(torch.stack([x.sum(1), x @ v, y @ v, z @ v, e, eta], 1) * h3)
    return torch.cat(rows)


def _network_inputs(F, L):
    """De-translated, mass-normalised band and the two moment scalars, FP64; and phase, mass mode."""
    ks, zero = _modes()
    fh, mo = _band(F), _moments64(F, L)
    rho, u = mo[:, 0], mo[:, 1:4] / mo[:, :1]
    ph = torch.exp(1j * math.pi / L * (u @ torch.as_tensor(ks.T, device=DEV).double()))
    m = fh[:, zero].real
    x = torch.view_as_real(fh * ph / m[:, None]).flatten(1)
    th = (2 * mo[:, 4] / rho - (u * u).sum(1)) / 3
    kl = mo[:, 5] / rho - torch.log(rho) + 1.5 * (torch.log(2 * math.pi * th) + 1)
    return torch.cat([x, th[:, None], kl[:, None]], 1), ph, m


def _surrogate64(case, seed, F):
    """What the two networks give, FP64: statistics, scores and their mean band."""
    _, zero = _modes()
    x, ph, m = _network_inputs(F, case["L"])
    mu, sd = x.mean(0).float(), x.std(0, unbiased=False).clamp_min(1e-4).float()
    # outputs: unit spread scaled to the size of Q's band relative to m^2
    nu, t = torch.zeros(926, device=DEV), 0.02
    xn = (x - mu.double()) / sd.double()
    bands = []
    for k in (0, 1):
        y = _forward64(_network(case, seed * 2 + k), xn) * float(np.float32(t)) + nu.double()
        bands.append(torch.view_as_complex(y.reshape(-1, 463, 2)) * (m * m)[:, None] / ph)
    q, c = bands
    for b in bands:
        b[:, zero] = 0
    mean = (q + c) / 2
    score = torch.linalg.vector_norm(q - c, dim=1) / torch.linalg.vector_norm(mean, dim=1)
    stats = np.zeros((4, ef.EF_FEATURE_STRIDE), dtype=np.float32)
    stats[1] = 1.0
    stats[0], stats[1], stats[2, :926], stats[3] = mu.cpu().numpy(), sd.cpu().numpy(), nu.cpu().numpy(), t
    return stats, score, mean


# ------------------------------------------------------------------ prepare and run --------

def _units(case):
    """Factors [1, cells, 10] that put the entropy production sum (column 6) per volume, like the entropy."""
    Ns = _sizes(case) if case["kind"] == "ragged" else [case["N"]] * case["cells"]
    out = torch.ones(1, case["cells"], 10, dtype=torch.float64, device=DEV)
    out[0, :, 6] = (2.0 * case["L"] / torch.tensor(Ns, device=DEV, dtype=torch.float64)) ** case["d"]
    return out


def _recorded(case):
    """Step size, count and diagnostics buffers of a recorded Euler run."""
    shape = (case["steps"], case["cells"], 10)
    f32 = case["prec"] == "F32"
    diag = torch.zeros(shape, dtype=torch.float64, device=DEV) if case["diag"] else None
    return dict(dt=case["dt"], steps=case["steps"], f32=f32, diag=diag, units=_units(case) if f32 and case["diag"] else None,
                record=torch.zeros(shape, device=DEV) if f32 and case["diag"] else None)


def prepare(case, seed):
    kind, n = case["kind"], case["cells"]
    dt = RES[case["prec"]]
    if kind == "mlp_grad":
        net = _network(case, seed)
        mlp = _mlp(case, net, n)
        X, T, w, r = _train_batch(case, seed)
        return {"kind": kind, "mlp": mlp, "X": X, "T": T, "w": w, "r": r, "n": n, "loss": torch.zeros(1, device=DEV),
                "grad": torch.zeros(mlp.nparams, device=DEV)}
    cells = _cells(case, seed)
    if kind == "ragged":
        prec = ef.EF_PREC_F32
        kernel = ef.EF_KERNEL_HARD_SPHERE
        plan = ef.Plan(3, None, case["L"], kernel, case["R"], prec, batched_N=_sizes(case))
        plan.set_graph(True)
        return dict(_recorded(case), kind="euler", plan=plan, F=_packed(case, cells, dt), n=n)
    plan = _plan(case)
    F = cells.to(dt)
    state = {"kind": kind, "plan": plan, "F": F, "n": n}
    if kind == "collide":
        state["Q"] = torch.zeros_like(F)
    elif kind == "euler":
        state.update(_recorded(case))
    elif kind == "rk3":
        plan.reserve(n)
        state.update(dt=case["dt"], steps=case["steps"])
    elif kind == "inhomogeneous":
        # Courant number 0.5 at the fastest velocity
        state.update(dt=case["dt"], steps=case["steps"], dx=case["dt"] * case["L"] / 0.5, scratch=torch.zeros_like(F),
                     mom=torch.zeros(n, 10, dtype=torch.float64, device=DEV), f32=case["prec"] == "F32")
    else:
        stats, _, _ = _surrogate64(case, seed, F)
        nets = [_mlp(case, _network(case, seed * 2 + k), n) for k in (0, 1)]
        sur = ef.Surrogate(plan, nets[0], n)
        sur.set_stats(stats.reshape(-1))
        # weights from a seed in place of trained ones: the audit alone decides which cells fall back
        sur.set_policy(1.0, 1e6)
        sur.set_entropy_gate(False)
        sur.set_checker(nets[1], 3e38)
        state.update(sur=sur, q=torch.zeros(n, ef.EF_FEATURE_STRIDE, device=DEV), flags=torch.zeros(n, dtype=torch.int32, device=DEV),
                     score=torch.zeros(n, device=DEV), Q=torch.zeros_like(F))
    return state


def _train_batch(case, seed):
    """Standardised inputs and targets, per-output and per-sample weights, as the trainer makes them."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["cells"]
    X = torch.randn(n, ef.EF_FEATURE_STRIDE, device=DEV, generator=g)
    T = torch.randn(n, ef.EF_FEATURE_STRIDE, device=DEV, generator=g) * 0.5
    w = torch.ones(926, device=DEV)
    _, zero = _modes()
    w[2 * zero:2 * zero + 2] = 0.0
    r = torch.exp(0.5 * torch.randn(n, device=DEV, generator=g))
    return X, T, w, r / r.mean()


def run(s):
    kind = s["kind"]
    if kind == "collide":
        s["plan"].collide(s["F"], s["Q"], ncells=s["n"])
        return s["Q"]
    if kind == "euler":
        s["plan"].euler(s["F"], s["dt"], nsteps=s["steps"], diag=s["diag"], ncells=s["n"])
        if s["diag"] is None:
            return (s["F"],)
        if not s["f32"]:
            return s["F"], s["diag"]
        # an FP32 plan's record: all columns per volume, at the precision they are computed to
        torch.mul(s["diag"], s["units"], out=s["record"])
        return s["F"], s["record"]
    if kind == "rk3":
        s["plan"].rk3(s["F"], s["dt"], nsteps=s["steps"], ncells=s["n"])
        return s["F"]
    if kind == "inhomogeneous":
        s["plan"].inhomogeneous(s["F"], s["scratch"], s["dx"], s["dt"], nsteps=s["steps"])
        s["plan"].moments(s["F"], None, s["mom"])
        return s["F"], s["mom"].float() if s["f32"] else s["mom"]
    if kind == "surrogate":
        s["sur"].infer_ex(s["F"], s["q"], s["flags"], s["n"], score=s["score"], Q=s["Q"], audit_fraction=AUDIT, seed=1, tol=1e-3)
        return {"q": s["q"], "flags": s["flags"], "score": s["score"], "Q": s["Q"]}
    s["mlp"].grad(s["X"], s["T"], s["n"], s["loss"], grad=s["grad"], wmask=s["w"], rowweight=s["r"])
    return s["loss"], s["grad"]


# ------------------------------------------------------------------ exact, in 64 bits ------

def _filter(N):
    """Modified Jackson filter of one axis in FFT order, n = N/2; zero at -N/2."""
    k = np.fft.fftfreq(N, 1.0 / N)
    p = N // 2 + 1
    b, t = np.abs(k), math.pi / p
    s = ((p - b) * np.cos(t * b) + np.sin(t * b) / math.tan(t)) / p
    s[N // 2] = 0.0
    return s


def _radial(x, typ, u, R, T):
    """Radial factor Phi(x): 2D, 3D hard spheres, 3D Maxwell with rate u."""
    a = math.pi * x / T
    if typ == "2d":
        return 2 * R * torch.sinc(R * x / T)
    if typ == "hard_sphere":
        return R * R * (2 * torch.sinc(R * x / T) - torch.sinc(0.5 * R * x / T) ** 2)
    gx, gw = np.polynomial.legendre.leggauss(96)
    out = torch.zeros_like(a)
    for g, w in zip(gx, gw):
        r = 0.5 * R * (g + 1)
        out += (0.5 * R * w) * r * math.exp(-(u * r) ** 2) * torch.cos(a * r)
    return 2 * out


def _multipliers(case, N):
    """[(M_e, Gamma_e)] and the loss table L on the full grid of modes."""
    d, L, R = case["d"], case["L"], 4.0 * case["L"] / (3.0 * math.sqrt(2.0) + 1.0)
    k = torch.fft.fftfreq(N, 1.0 / N, device=DEV, dtype=torch.float64)
    sg1 = torch.as_tensor(_filter(N), device=DEV)
    grids, sg = [], 1.0
    for a in range(d):
        shape = (1,) * a + (N,) + (1,) * (d - 1 - a)
        grids.append(k.reshape(shape))
        sg = sg * sg1.reshape(shape)

    def mult(e, typ, u=0.0):
        return sg * _radial(sum(g * float(x) for g, x in zip(grids, e)), typ, u, R, L)

    out = []
    if d == 2:
        r = case["R"]
        e = [(math.cos(math.pi * t / r), math.sin(math.pi * t / r)) for t in range(r)]
        for t in range(r // 2):
            out.append((mult(e[t], "2d"), 2.0 / r * mult(e[t + r // 2], "2d")))
    else:
        nmu, nphi, nc = QUAD[case["R"]]
        gx, gw = np.polynomial.legendre.leggauss(nmu)
        terms = [(0.0, 1.0)]
        if case["kernel"] == "maxwell":
            ta, tb = math.log(0.4 / R), math.log(35.0 / R)
            tx, tw = np.polynomial.legendre.leggauss(5)
            c = 2 / math.sqrt(math.pi)
            terms = [(0.0, c * math.exp(ta))]
            terms += [(math.exp(ta + 0.5 * (x + 1) * (tb - ta)), c * 0.5 * (tb - ta) * w * math.exp(ta + 0.5 * (x + 1) * (tb - ta))) for x, w in zip(tx, tw)]
        for u, cj in terms:
            for x, w in zip(gx, gw):
                mu = 0.5 * (x + 1)
                st = math.sqrt(1 - mu * mu)
                for b in range(nphi):
                    al = 2 * math.pi * b / nphi
                    ca, sa = math.cos(al), math.sin(al)
                    gam = 0.0
                    for q in range(nc):
                        cp, sp = math.cos(math.pi * q / nc), math.sin(math.pi * q / nc)
                        es = (cp * mu * ca - sp * sa, cp * mu * sa + sp * ca, -cp * st)
                        wt = (1 / math.pi) * (0.5 * w) * (2 * math.pi / nphi) * (math.pi / nc) * cj
                        gam = gam + wt * mult(es, case["kernel"], u)
                    out.append((mult((st * ca, st * sa, mu), case["kernel"], u), gam))
    return out, sum(m * g for m, g in out)


class _Operator:
    def __init__(self, case, N):
        self.pairs, self.loss = _multipliers(case, N)
        self.N, self.dims = N, tuple(range(1, case["d"] + 1))

    def __call__(self, F):
        """(Q, nu) of cells [n, N, ...] in FP64."""
        Q, nu = torch.empty_like(F), torch.empty_like(F)
        step = max(1, 2 ** 25 // self.N ** len(self.dims))
        for a in range(0, F.shape[0], step):
            f = F[a:a + step]
            h = torch.fft.fftn(f, dim=self.dims)
            v = torch.fft.ifftn(h * self.loss, dim=self.dims).real
            g = torch.zeros_like(f)
            for m, s in self.pairs:
                # both tables are even and real: one complex inverse gives the two real factors
                z = torch.fft.ifftn(h * torch.complex(m, s), dim=self.dims)
                g += z.real * z.imag
            Q[a:a + step], nu[a:a + step] = g - f * v, v
        return Q, nu


def _diag64(case, N, F, Q, nu, out):
    d = case["d"]
    v, hd = _axis(N, case["L"]), (2.0 * case["L"] / N) ** d
    f = F.flatten(1)
    ln = torch.where(f > 0, torch.log(f.clamp_min(1e-300)), 0.0)
    res = torch.zeros(F.shape[0], 10, dtype=torch.float64, device=DEV)
    res[:, 0] = f.sum(1) * hd
    for a in range(d):
        marg = F.sum(tuple(x for x in range(1, d + 1) if x != a + 1))
        res[:, 1 + a] = (marg @ v) * hd
        res[:, 4] += 0.5 * hd * (marg @ v ** 2)
    res[:, 5] = (f * ln).sum(1) * hd
    res[:, 7] = f.min(1).values
    if Q is not None:
        res[:, 6] = (Q.flatten(1) * ln).sum(1)
        res[:, 8] = nu.flatten(1).max(1).values
        res[:, 9] = out.flatten(1).min(1).values
    else:
        neg = (-f).clamp_min(0).sum(1)
        res[:, 8] = 2 * neg / (f.sum(1) + 2 * neg)
    return res


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp_grad":
        return _grad64(case, seed)
    if kind == "surrogate":
        F = _cells(case, seed).float()
        _, score, q = _surrogate64(case, seed, F)
        ks, _ = _modes()
        N, n = case["N"], case["cells"]
        rows = torch.as_tensor(_audited(n), device=DEV)
        Qp, _ = _Operator(case, N)(F[rows].double())
        q[rows] = _band(Qp)
        Q = torch.empty(F.shape, dtype=torch.float64, device=DEV)
        k = torch.as_tensor(ks, device=DEV)
        for a in range(0, n, 512):
            h = torch.zeros((min(n, a + 512) - a, N, N, N), dtype=torch.complex128, device=DEV)
            kk, km = k % N, (-k) % N
            h[:, km[:, 0], km[:, 1], km[:, 2]] = q[a:a + 512].conj()
            h[:, kk[:, 0], kk[:, 1], kk[:, 2]] = q[a:a + 512]
            Q[a:a + 512] = torch.fft.ifftn(h, dim=(1, 2, 3)).real * N ** 3
        Q[rows] = Qp
        band = torch.zeros(n, ef.EF_FEATURE_STRIDE, dtype=torch.float64, device=DEV)
        band[:, :926] = torch.view_as_real(q).flatten(1)
        return {"q": band, "flags": None, "score": score, "Q": Q}
    dt = RES[case["prec"]]
    if kind == "ragged":
        Ns = _sizes(case)
        parts, diags = {}, torch.zeros(1, case["cells"], 10, dtype=torch.float64, device=DEV)
        for N, F in _cells(case, seed).items():
            F = F.to(dt).double()
            Q, nu = _Operator(case, N)(F)
            parts[N] = F + case["dt"] * Q
            if case["diag"]:
                rows = torch.as_tensor([i for i, x in enumerate(Ns) if x == N], device=DEV)
                diags[0, rows] = _diag64(case, N, F, Q, nu, parts[N])
            del F, Q, nu
        out = _packed(case, parts, torch.float64)
        return (out, diags * _units(case)) if case["diag"] else (out,)
    F = _cells(case, seed).to(dt).double()
    N = case["N"]
    op = _Operator(case, N)
    if kind == "collide":
        return op(F)[0]
    if kind == "euler":
        rows = []
        for _ in range(case["steps"]):
            Q, nu = op(F)
            new = F + case["dt"] * Q
            if case["diag"]:
                rows.append(_diag64(case, N, F, Q, nu, new))
            F = new
        if not rows:
            return (F,)
        diags = torch.stack(rows)
        return F, diags * _units(case) if case["prec"] == "F32" else diags
    if kind == "rk3":
        h = case["dt"]
        for _ in range(case["steps"]):
            F1 = F + h * op(F)[0]
            F2 = 0.75 * F + 0.25 * (F1 + h * op(F1)[0])
            F = F / 3 + 2.0 / 3.0 * (F2 + h * op(F2)[0])
        return F
    v = _axis(N, case["L"]).reshape((1, N) + (1,) * (case["d"] - 1))
    nu = v * case["dt"] / (case["dt"] * case["L"] / 0.5)
    for _ in range(case["steps"]):
        up = torch.where(nu > 0, torch.roll(F, 1, 0), torch.roll(F, -1, 0))
        F = F - nu.abs() * (F - up)
        F = F + case["dt"] * op(F)[0]
    return F, _diag64(case, N, F, None, None, None)


def _grad64(case, seed):
    X, T, w, r = _train_batch(case, seed)
    widths = _widths(case)
    net = _network(case, seed)
    ps = []
    h = X[:, :widths[0]].double()
    for i, (W, b) in enumerate(net):
        W = torch.as_tensor(W, device=DEV).bfloat16().double().requires_grad_()
        b = torch.as_tensor(b, device=DEV).double().requires_grad_()
        ps.append((W, b))
        h = h @ W.T + b
        h = torch.relu(h) if i < len(net) - 1 else h
    loss = (w.double() * r.double()[:, None] * (h - T[:, :926].double()) ** 2).sum() / (case["cells"] * 926)
    loss.backward()
    pad = lambda x: (x + 63) // 64 * 64  # noqa: E731
    flat = []
    for W, b in ps:
        o, i = W.shape
        G = torch.zeros(pad(o), pad(i), dtype=torch.float64, device=DEV)
        G[:o, :i] = W.grad
        c = torch.zeros(pad(o), dtype=torch.float64, device=DEV)
        c[:o] = b.grad
        flat += [G.flatten(), c]
    return loss.detach().reshape(1), torch.cat(flat)
