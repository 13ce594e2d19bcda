"""Calls of one plan on several streams, and graphs replayed beside each other and beside calls, where the
kernels keep spectra or accumulators in the plan's workspaces: the results of a call alone, bit for bit."""
import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef
from paper_1704_07369_gb300 import inputs

pytestmark = pytest.mark.gpu

F32, F64, MAXWELL, HARD = ef.EF_PREC_F32, ef.EF_PREC_F64, ef.EF_KERNEL_MAXWELL, ef.EF_KERNEL_HARD_SPHERE
# d, N, kernel, R, precision, cell counts: few (split where that pays) and more than a round of clusters
CASES = [(3, 16, HARD, 16, F64, (1, 400)), (2, 24, MAXWELL, 16, F64, (1, 3000)), (2, 16, MAXWELL, 16, F32, (2, 6000)),
         (3, 12, HARD, 16, F32, (3, 2000)), (3, 64, HARD, 8, F64, (1, 12)), (3, 32, HARD, 16, F32, (1, 300))]


def _cells(d, N, n, dtype, seed):
    base = np.stack([inputs.mixture_cell(d, N, 8.0, seed + i) for i in range(4)])
    scale = np.random.default_rng(seed).uniform(0.5, 1.5, size=n)
    F = base[np.arange(n) % 4] * scale.reshape((n,) + (1,) * d)
    return torch.tensor(F, dtype=dtype, device="cuda")


@pytest.mark.parametrize("d,N,kernel,R,prec,counts", CASES)
def test_streams_and_graphs_side_by_side(d, N, kernel, R, prec, counts):
    dtype = torch.float64 if prec == F64 else torch.float32
    plan = ef.Plan(d, N, 8.0, kernel, R, prec)
    F = [_cells(d, N, n, dtype, 600 + 10 * i) for i, n in enumerate(counts)]
    ref = [torch.empty_like(f) for f in F]
    for f, q in zip(F, ref):
        plan.collide(f, q, ncells=f.shape[0])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(4)]
    # calls on two streams, small and large in turn
    out = [[torch.zeros_like(F[(i + r) % 2]) for r in range(4)] for i in range(2)]
    torch.cuda.synchronize()
    for r in range(4):
        for i in range(2):
            k = (i + r) % 2
            plan.collide(F[k], out[i][r], ncells=F[k].shape[0], stream=streams[i])
    torch.cuda.synchronize()
    for r in range(4):
        for i in range(2):
            assert torch.equal(out[i][r], ref[(i + r) % 2]), (r, i)
    graphs, gout = [], []
    for i in range(2):
        g = torch.cuda.CUDAGraph()
        q = torch.zeros_like(F[i])
        with torch.cuda.graph(g, stream=streams[i]):
            for _ in range(2):
                plan.collide(F[i], q, ncells=F[i].shape[0])
        graphs.append(g)
        gout.append(q)
    direct = [torch.zeros_like(f) for f in F]
    torch.cuda.synchronize()
    for r in range(6):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                graphs[i].replay()
            plan.collide(F[i], direct[i], ncells=F[i].shape[0], stream=streams[2 + (r + i) % 2])
    torch.cuda.synchronize()
    for i in range(2):
        assert torch.equal(gout[i], ref[i]), i
        assert torch.equal(direct[i], ref[i]), i
    assert plan.status(sync=1) == ef.EF_OK
    del graphs
    plan.close()
