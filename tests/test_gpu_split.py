"""Split launches: a batch with fewer cells than the device holds clusters runs the ops of one cell as
several parts, whose gains a finishing launch sums.

Bars: Q against the oracle as in test_gpu_parity.py (FP64 rel-L2 <= 1e-12, FP32 2e-5 of max |Q|).  Against
an unsplit plan (its launch shape pinned): moments and entropy agree to the float-float / FP64 sums
(1e-9 of their scale), values that depend on Q to the parity bar."""
import numpy as np
import pytest
import torch

import oracle
import paper_1704_07369_gb300 as ef
from paper_1704_07369_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [(2, 8, 16, 0, ef.EF_PREC_F64), (2, 16, 16, 0, ef.EF_PREC_F32), (2, 24, 8, 0, ef.EF_PREC_F64),
         (3, 8, 16, 1, ef.EF_PREC_F32), (3, 12, 16, 1, ef.EF_PREC_F64), (3, 12, 8, 0, ef.EF_PREC_F32),
         (3, 16, 16, 1, ef.EF_PREC_F32), (3, 16, 8, 0, ef.EF_PREC_F32), (3, 16, 8, 1, ef.EF_PREC_F64)]


def _cells(d, N, L, n):
    return [inputs.mixture_cell(d, N, L, 900 + i) for i in range(n)]


@pytest.mark.parametrize("d,N,R,kernel,prec", CASES)
@pytest.mark.parametrize("n", [1, 3])
def test_split_against_oracle_and_unsplit(d, N, R, kernel, prec, n, monkeypatch):
    L, dt = 8.0, 0.01
    dtype = torch.float64 if prec == ef.EF_PREC_F64 else torch.float32
    host = _cells(d, N, L, n)
    F = torch.tensor(np.stack(host), dtype=dtype, device="cuda")
    plan = ef.Plan(d, N, L, kernel, R, prec)
    Q = torch.zeros_like(F)
    plan.collide(F, Q, ncells=n)
    F1, F2 = F.clone(), F.clone()
    D1, D2 = (torch.zeros(n, ef.EF_DIAG_STRIDE, dtype=torch.float64, device="cuda") for _ in range(2))
    plan.euler(F1, dt, diag=D1, ncells=n)
    i = plan.info()
    monkeypatch.setenv("EF_SHAPE", "%d:%d:%d:%d:1" % (N, i["cluster"], i["threads"], 3 if (d, N, prec) == (3, 16, 0) else 1))
    one = ef.Plan(d, N, L, kernel, R, prec)
    one.euler(F2, dt, diag=D2, ncells=n)
    torch.cuda.synchronize()
    one.close()
    assert plan.status(sync=1, reset=1) == ef.EF_OK
    p = oracle.Params(d=d, N=N, T=L, kernel=kernel, R=R, J=6)
    scale = 0.0
    for i in range(n):
        ref, q = oracle.collide(p, host[i]), Q[i].double().cpu().numpy()
        scale = max(scale, np.abs(ref).max())
        if prec == ef.EF_PREC_F64:
            assert np.linalg.norm(q - ref) <= 1e-12 * np.linalg.norm(ref)
        else:
            assert np.abs(q - ref).max() <= 2e-5 * np.abs(ref).max()
    tol = 1e-12 if prec == ef.EF_PREC_F64 else 2e-5
    assert (F1 - F2).abs().max().item() <= tol * dt * scale + 1.2e-7 * F.abs().max().item() * (prec == ef.EF_PREC_F32)
    d1, d2 = D1.cpu().numpy(), D2.cpu().numpy()
    for k in (0, 1, 2, 3, 4, 5, 7):
        assert np.abs(d1[:, k] - d2[:, k]).max() <= 1e-9 * max(1.0, np.abs(d2[:, k]).max()), k
    lnf = sum(np.abs(np.log(np.maximum(c, 1e-300))).sum() for c in host)
    assert np.abs(d1[:, 6] - d2[:, 6]).max() <= 2 * tol * scale * lnf
    assert np.abs(d1[:, 8] - d2[:, 8]).max() <= 1e-5 * np.abs(d2[:, 8]).max()
    plan.close()


@pytest.mark.parametrize("prec", [ef.EF_PREC_F32, ef.EF_PREC_F64])
def test_split_calls_of_two_streams(prec):
    """Calls of one plan on two streams share the part workspace: each waits for the other's."""
    N, L = 16, 8.0
    dtype = torch.float64 if prec == ef.EF_PREC_F64 else torch.float32
    F = torch.tensor(np.stack(_cells(3, N, L, 2)), dtype=dtype, device="cuda")
    plan = ef.Plan(3, N, L, ef.EF_KERNEL_HARD_SPHERE, 16, prec)
    ref = [torch.zeros_like(F[:1]) for _ in range(2)]
    for i in range(2):
        plan.collide(F[i:i + 1], ref[i], ncells=1)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [[torch.zeros_like(F[:1]) for _ in range(8)] for _ in range(2)]
    for r in range(8):
        for i in range(2):
            plan.collide(F[i:i + 1], out[i][r], ncells=1, stream=streams[i])
    torch.cuda.synchronize()
    for i in range(2):
        for r in range(8):
            assert torch.equal(out[i][r], ref[i])
    plan.close()


def test_split_calls_under_capture():
    """Captured calls take a workspace of their graph: two graphs replayed side by side, and beside direct
    calls, give the direct calls' results bit for bit; more captures than workspaces stay correct."""
    N, L = 16, 8.0
    F = torch.tensor(np.stack(_cells(3, N, L, 2)), dtype=torch.float32, device="cuda")
    plan = ef.Plan(3, N, L, ef.EF_KERNEL_HARD_SPHERE, 16, ef.EF_PREC_F32)
    ref = [torch.zeros_like(F[:1]) for _ in range(2)]
    for i in range(2):
        plan.collide(F[i:i + 1], ref[i], ncells=1)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [torch.zeros_like(F[:1]) for _ in range(2)]
    graphs = []
    for i in range(2):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[i]):
            for _ in range(3):
                plan.collide(F[i:i + 1], out[i], ncells=1)
        graphs.append(g)
    direct = torch.zeros_like(F[:1])
    for _ in range(6):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                graphs[i].replay()
        plan.collide(F[:1], direct, ncells=1)
    torch.cuda.synchronize()
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1]) and torch.equal(direct, ref[0])
    more = []
    for k in range(8):
        g = torch.cuda.CUDAGraph()
        q = torch.zeros_like(F[:1])
        with torch.cuda.graph(g):
            plan.collide(F[:1], q, ncells=1)
        more.append((g, q))
    for g, q in more:
        g.replay()
    torch.cuda.synchronize()
    for g, q in more:
        assert (q - ref[0]).abs().max().item() <= 2e-5 * ref[0].abs().max().item()
    plan.close()


@pytest.mark.parametrize("N,n", [(16, 1), (24, 2), (40, 3), (48, 1), (48, 5)])
def test_split_step_moments_are_of_the_old_state(N, n):
    """The sums over F of a split FP32 step in place are over the state before the step: against FP64
    sums of that state (a row in FP32, N terms of one sign: N u relative to the sum of magnitudes).
    dt is large, so that a sum over a partly updated state shows."""
    L, dt = 8.0, 0.3
    host = np.stack(_cells(3, N, L, n))
    F = torch.tensor(host, dtype=torch.float32, device="cuda")
    old = F.double().cpu().numpy()
    D = torch.zeros(n, ef.EF_DIAG_STRIDE, dtype=torch.float64, device="cuda")
    plan = ef.Plan(3, N, L, ef.EF_KERNEL_HARD_SPHERE, 32, ef.EF_PREC_F32)
    plan.euler(F, dt, diag=D, ncells=n)
    torch.cuda.synchronize()
    plan.close()
    d, h = D.cpu().numpy(), 2 * L / N
    v = (np.arange(N) - N // 2) * h
    z, y, x = np.meshgrid(v, v, v, indexing="ij")
    with np.errstate(divide="ignore", invalid="ignore"):
        eta = np.where(old > 0, old * np.log(old), 0.0)
    u = N * 2.0 ** -24
    for k, w in ((0, old), (1, old * z), (2, old * y), (3, old * x), (4, 0.5 * old * (x * x + y * y + z * z))):
        assert (np.abs(d[:, k] - h ** 3 * w.sum((1, 2, 3))) <= 2 * u * h ** 3 * np.abs(w).sum((1, 2, 3)) + 1e-12).all(), k
    # the fast logarithm adds 2^-21.4 absolute (CUDA's bound for __logf in [0.5, 2]; relative 2 ulp elsewhere)
    bound = (2 * u * np.abs(eta) + 2.0 ** -20 * np.abs(old)).sum((1, 2, 3))
    assert (np.abs(d[:, 5] - h ** 3 * eta.sum((1, 2, 3))) <= h ** 3 * bound).all()
    assert (d[:, 7] == old.min((1, 2, 3))).all()
