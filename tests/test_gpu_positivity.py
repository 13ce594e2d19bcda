"""EF_ERR_POSITIVITY of an Euler step is a property of a cell: an updated value below zero and dt nu > 1,
wherever in the cell either is, however many cells the call has and however they are spread over CTAs.

The cell has one negative value in a corner, where nu is smallest (under 6% of its maximum here), and dt is
1.02 / max nu, so that dt nu > 1 only in a few planes around its middle; with 0.98 / max nu nothing is reported."""
import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef
from paper_1704_07369_gb300 import inputs

pytestmark = pytest.mark.gpu

F32, F64, MAXWELL, HARD = ef.EF_PREC_F32, ef.EF_PREC_F64, ef.EF_KERNEL_MAXWELL, ef.EF_KERNEL_HARD_SPHERE
# d, N, R, kernel, precision, cell counts: a few (split over clusters) and more than a round of clusters
CASES = [(2, 16, 16, MAXWELL, F32, (1, 6000)), (2, 24, 8, MAXWELL, F64, (1, 2, 6000)), (3, 8, 16, HARD, F32, (1, 3000)),
         (3, 12, 16, HARD, F32, (2, 1500)), (3, 12, 16, HARD, F64, (1, 1500)), (3, 16, 16, HARD, F32, (1, 3, 700)),
         (3, 24, 16, HARD, F32, (1, 400)), (3, 32, 16, HARD, F64, (1, 4, 100)), (3, 48, 16, HARD, F32, (1, 60)),
         (3, 64, 16, HARD, F64, (1, 20))]
# pinned launch shapes of one N (cluster, threads, variant, parts): register and team kernels
PINNED = [(16, 2, 128, 3, 1), (24, 3, 192, 3, 1), (24, 3, 192, 3, 4), (24, 4, 144, 3, 1), (32, 4, 256, 3, 3), (32, 8, 128, 3, 1),
          (24, 4, 288, 7, 1)]


def _check(plan, d, N, prec, n):
    dtype = torch.float64 if prec == F64 else torch.float32
    cell = inputs.mixture_cell(d, N, 8.0, 5)
    corner = (0,) * d
    cell[corner] = -0.01 * cell.max()
    one = torch.tensor(cell, dtype=dtype, device="cuda")[None]
    diag = torch.zeros(1, ef.EF_DIAG_STRIDE, dtype=torch.float64, device="cuda")
    plan.euler(one.clone(), 0.0, diag=diag, ncells=1)
    numax = diag[0, 8].item()
    assert plan.status(sync=1, reset=1) == ef.EF_OK
    F = 0.5 * one.repeat(n, *([1] * d))                  # half the density, half of nu
    F[n - 1] = one[0]
    for scale, status in ((1.02, ef.EF_ERR_POSITIVITY), (0.98, ef.EF_OK)):
        for with_diag in (False, True):
            G = F.clone()
            D = torch.zeros(n, ef.EF_DIAG_STRIDE, dtype=torch.float64, device="cuda")
            plan.euler(G, scale / numax, diag=D if with_diag else None, ncells=n)
            assert plan.status(sync=1, reset=1) == status, (scale, with_diag)
            assert (G[(n - 1,) + corner] < 0).item()
            if with_diag:
                assert (D[:, 9].cpu().numpy() == G.double().reshape(n, -1).min(1).values.cpu().numpy()).all()
                assert np.allclose(D[n - 1, 8].item(), numax, rtol=1e-5)


@pytest.mark.parametrize("d,N,R,kernel,prec,n", [c[:5] + (n,) for c in CASES for n in c[5]])
def test_positivity_report_does_not_depend_on_the_cell_count(d, N, R, kernel, prec, n):
    plan = ef.Plan(d, N, 8.0, kernel, R, prec)
    _check(plan, d, N, prec, n)
    plan.close()


@pytest.mark.parametrize("N,cluster,threads,variant,parts", PINNED)
def test_positivity_report_of_launch_shapes(N, cluster, threads, variant, parts, monkeypatch):
    monkeypatch.setenv("EF_SHAPE", "%d:%d:%d:%d:%d" % (N, cluster, threads, variant, parts))
    plan = ef.Plan(3, N, 8.0, HARD, 16, F32)
    info = plan.info()
    assert (info["cluster"], info["threads"]) == (cluster, threads)
    _check(plan, 3, N, F32, 2)
    plan.close()
