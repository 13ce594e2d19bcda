"""Split launches with their parts pinned: every part count a size's op list allows (two, an uneven share,
the most) against the unsplit launch of the same shape, for uniform and ragged plans, both scatter kinds of
the register kernels and all kernel families.  ef_plan_call_info says in every case that the launch is the
one meant.

Bars, as in test_gpu_split.py: Q and F + dt Q to the parity bars (FP64 rel-L2 1e-12, FP32 2e-5 of max |Q|;
the unsplit kernels' parity with the oracle is tested elsewhere), sums over F to 1e-9 of their scale, the
entropy production to the parity bar times sum |ln F|, max nu to 1e-5."""
import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef
from paper_1704_07369_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DT = 8.0, 0.01
F32, F64, MAXWELL, HARD = ef.EF_PREC_F32, ef.EF_PREC_F64, ef.EF_KERNEL_MAXWELL, ef.EF_KERNEL_HARD_SPHERE
# FP32 3D register kernels (cluster, threads, variant): one and two rows a thread, clusters of one and two
# (scatter behind the barrier) and of three and more (st.async)
REGISTER = [(16, 1, 256, 3), (16, 4, 64, 3), (24, 2, 288, 3), (24, 3, 192, 3), (24, 4, 72, 4), (32, 2, 256, 4), (32, 4, 256, 3),
            (32, 8, 64, 4), (40, 5, 320, 3), (40, 10, 80, 4), (48, 8, 288, 3), (48, 12, 96, 4), (64, 16, 256, 3), (64, 16, 128, 4)]
# the other families in their plan's first shape
OTHERS = [(2, 8, F32), (2, 16, F32), (2, 64, F32), (2, 8, F64), (2, 24, F64), (2, 64, F64), (3, 8, F32), (3, 12, F32),
          (3, 8, F64), (3, 12, F64), (3, 24, F64), (3, 32, F64), (3, 40, F64),
          (3, 48, F64)]
PARTS = (2, 4, 1 << 20)


def _compare(F, out, ref, d, prec, cells):
    """out, ref: (Q, F + dt Q, diagnostics); cells: (offset, size) of each."""
    tol = 1e-12 if prec == F64 else 2e-5
    for c, (off, size) in enumerate(cells):
        f, q, r = F[off:off + size], out[0][off:off + size], ref[0][off:off + size]
        scale = np.abs(r).max()
        if prec == F64:
            assert np.linalg.norm(q - r) <= tol * np.linalg.norm(r), c
        else:
            assert np.abs(q - r).max() <= tol * scale, c
        step = np.abs(out[1][off:off + size] - ref[1][off:off + size]).max()
        assert step <= tol * DT * scale + (1.2e-7 * np.abs(f).max() if prec == F32 else 0.0), c
        a, b = out[2][c], ref[2][c]
        for k in (0, 1, 2, 3, 4, 5, 7):
            assert abs(a[k] - b[k]) <= 1e-9 * max(1.0, abs(b[k])), (c, k)
        assert abs(a[6] - b[6]) <= 2 * tol * scale * np.abs(np.log(np.maximum(f, 1e-300))).sum(), c
        assert abs(a[8] - b[8]) <= 1e-5 * abs(b[8]), c
        assert abs(a[9] - b[9]) <= tol * DT * scale + 1.2e-7 * np.abs(f).max(), c


def _run(plan, F, n, counted):
    Q, G = torch.full_like(F, float("nan")), F.clone()
    D = torch.full((n, ef.EF_DIAG_STRIDE), float("nan"), dtype=torch.float64, device="cuda")
    kw = {"ncells": n} if counted else {}
    plan.collide(F, Q, **kw)
    plan.euler(G, DT, diag=D.view(1, n, -1) if not counted else D, **kw)
    assert plan.status(sync=1, reset=1) == ef.EF_OK
    return [x.double().cpu().numpy().ravel() for x in (Q, G)] + [D.cpu().numpy()]


def _uniform(monkeypatch, d, N, kernel, R, prec, shape, n):
    dtype = torch.float64 if prec == F64 else torch.float32
    host = np.stack([inputs.mixture_cell(d, N, L, 1200 + N + i) for i in range(n)])
    F = torch.tensor(host, dtype=dtype, device="cuda")
    cells = [(i * N ** d, N ** d) for i in range(n)]

    def at(parts):
        monkeypatch.setenv("EF_SHAPE", "%d:%d:%d:%d:%d" % ((N,) + shape + (parts,)))
        plan = ef.Plan(d, N, L, kernel, R, prec)
        call = plan.call_info(n)[0]
        assert (call["cluster"], call["threads"], call["variant"]) == shape
        out = _run(plan, F, n, True)
        plan.close()
        return call["parts"], out

    parts, ref = at(1)
    assert parts == 1
    seen = set()
    for p in PARTS:
        parts, out = at(p)
        assert 2 <= parts <= p
        seen.add(parts)
        _compare(F.double().cpu().numpy().ravel(), out, ref, d, prec, cells)
    assert len(seen) >= 2


@pytest.mark.parametrize("N,cluster,threads,variant", REGISTER)
def test_parts_of_register_kernels(N, cluster, threads, variant, monkeypatch):
    _uniform(monkeypatch, 3, N, HARD, 32, F32, (cluster, threads, variant), 2)


@pytest.mark.parametrize("d,N,prec", OTHERS)
def test_parts_of_other_kernels(d, N, prec, monkeypatch):
    kernel, R = (MAXWELL, 16) if d == 2 else (HARD, 32)
    probe = ef.Plan(d, N, L, kernel, R, prec)
    info, sg = probe.info(), probe.class_info()[0]["sg_global"]
    probe.close()
    assert not sg                     # a shape that can be pinned
    _uniform(monkeypatch, d, N, kernel, R, prec, (info["cluster"], info["threads"], 1), 2)


def test_parts_with_accumulators_in_global_memory():
    """The largest FP64 cells: one cell alone is split, the same cell in a larger batch is not."""
    N, prec, n = 64, F64, 24
    plan = ef.Plan(3, N, L, HARD, 16, prec)
    assert plan.call_info(1)[0]["parts"] > 1
    assert plan.call_info(n)[0]["parts"] == 1
    cell = inputs.mixture_cell(3, N, L, 1300 + N)
    F = torch.tensor(cell, dtype=torch.float64, device="cuda")[None]
    out = _run(plan, F, 1, True)
    many = _run(plan, F.repeat(n, 1, 1, 1), n, True)
    ref = [many[0][-N ** 3:], many[1][-N ** 3:], many[2][-1:]]
    _compare(F.double().cpu().numpy().ravel(), out, ref, 3, prec, [(0, N ** 3)])
    plan.close()


RAGGED = [(3, [24, 32, 24, 48, 16, 32, 64], F32, {16: (4, 64, 3), 24: (3, 192, 3), 32: (2, 256, 4), 48: (8, 288, 3), 64: (16, 256, 3)}),
          (3, [12, 8, 12, 12, 8], F32, None), (3, [16, 24, 12, 16, 8], F64, None), (2, [16, 64, 8, 16, 24], F64, None),
          (2, [16, 48, 8], F32, None)]


@pytest.mark.parametrize("d,sizes,prec,shapes", RAGGED)
def test_parts_of_ragged_plans(d, sizes, prec, shapes, monkeypatch):
    kernel, R = (MAXWELL, 16) if d == 2 else (HARD, 32)
    dtype = torch.float64 if prec == F64 else torch.float32
    if shapes is None:
        monkeypatch.setenv("EF_AUTOTUNE", "0")
        probe = ef.Plan(d, None, L, kernel, R, prec, batched_N=sizes)
        shapes = {c["N"]: (c["cluster"], c["threads"], 1) for c in probe.class_info() if not c["sg_global"]}
        probe.close()
    F = torch.tensor(inputs.pack([inputs.mixture_cell(d, N, L, 1400 + i) for i, N in enumerate(sizes)]), dtype=dtype, device="cuda")
    offs = np.concatenate([[0], np.cumsum([N ** d for N in sizes])])
    cells = [(int(offs[i]), N ** d) for i, N in enumerate(sizes)]

    def at(parts):
        monkeypatch.setenv("EF_SHAPE", ",".join("%d:%d:%d:%d:%d" % ((N,) + s + (parts,)) for N, s in shapes.items()))
        plan = ef.Plan(d, None, L, kernel, R, prec, batched_N=sizes)
        calls = plan.call_info()
        for info, call in zip(plan.class_info(), calls):
            assert (call["cluster"], call["threads"], call["variant"]) == shapes[info["N"]]
        out = _run(plan, F, len(sizes), False)
        plan.close()
        return [c["parts"] for c in calls], out

    parts, ref = at(1)
    assert set(parts) == {1}
    for p in PARTS:
        parts, out = at(p)
        assert all(2 <= x <= p for x in parts)
        _compare(F.double().cpu().numpy().ravel(), out, ref, d, prec, cells)
