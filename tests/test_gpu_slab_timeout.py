"""A slab wait of the FP32 register kernels that runs out (EF_SLAB_TIMEOUT_NS makes every slab expect 8 bytes
that nobody sends): EF_ERR_TIMEOUT in the status word, NaN in every output of the launch, one wait in all
and not one for each op and cell, and a device that works afterwards."""
import time

import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef
from paper_1704_07369_gb300 import inputs

pytestmark = pytest.mark.gpu

L, R, HARD = 8.0, 16, ef.EF_KERNEL_HARD_SPHERE


# cluster, threads, variant, parts of N = 24: G in registers (one row, two rows a thread) and in shared
# memory, split and not; clusters of three and more use st.async
@pytest.mark.parametrize("shape,n", [("24:3:192:3:1", 300), ("24:4:72:4:1", 100), ("24:6:96:6:1", 100), ("24:3:192:3:4", 5)])
def test_slab_wait_that_runs_out(shape, n, monkeypatch):
    N = 24
    F = torch.tensor(np.stack([inputs.mixture_cell(3, N, L, 70 + i % 3) for i in range(n)]), dtype=torch.float32, device="cuda")
    monkeypatch.setenv("EF_SHAPE", shape)
    good = ef.Plan(3, N, L, HARD, R, ef.EF_PREC_F32)
    info = good.info()
    assert (info["cluster"], info["threads"]) == tuple(int(x) for x in shape.split(":")[1:3])
    ref = torch.empty_like(F)
    good.collide(F, ref, ncells=n)
    assert good.status(sync=1) == ef.EF_OK
    monkeypatch.setenv("EF_SLAB_TIMEOUT_NS", "1000000")
    bad = ef.Plan(3, N, L, HARD, R, ef.EF_PREC_F32)
    monkeypatch.delenv("EF_SLAB_TIMEOUT_NS")
    Q, G = torch.zeros_like(F), F.clone()
    D = torch.zeros(n, ef.EF_DIAG_STRIDE, dtype=torch.float64, device="cuda")
    t0 = time.monotonic()
    bad.collide(F, Q, ncells=n)
    assert bad.status(sync=1, reset=1) == ef.EF_ERR_TIMEOUT
    bad.euler(G, 0.01, diag=D, ncells=n)
    assert bad.status(sync=1, reset=1) == ef.EF_ERR_TIMEOUT
    assert time.monotonic() - t0 < 2.0
    assert torch.isnan(Q).all() and torch.isnan(G).all()
    assert torch.isnan(D[:, 6]).all()                    # entropy production: from Q
    again = torch.empty_like(F)
    good.collide(F, again, ncells=n)
    assert good.status(sync=1) == ef.EF_OK
    assert torch.equal(again, ref)
    good.close()
    bad.close()
