"""The band of ln max(F, 1e-30) against FP64, with values at the clamp and around 1.

Bars.  PTX documents lg2.approx to 2^-22, absolute for an argument in (0.5, 2) and relative elsewhere; the product
with ln 2 rounds once more (u = 2^-24).  A constant cell's zero mode adds N equal values along each of three
axes: at most 3 (N - 1) roundings.  In a general cell each axis' sum of N products has at most N + 8 roundings
of the sum of magnitudes."""
import math

import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _plan(N, prec):
    return ef.Plan(3, N, 8.0, ef.EF_KERNEL_HARD_SPHERE, 16, prec)


@pytest.mark.parametrize("N", [16, 32])
def test_log_of_constant_cells(N):
    one = np.float32(1.0)
    v = [0.0, -1.0, 1e-45, 1e-38, 9.9e-31, 1e-30, 1.01e-30, 1e-29, 1e-20, 1e-10, 1e-4, 0.1, 0.49, 0.5, 0.51, 0.7, 0.9, 0.999,
         np.nextafter(one, np.float32(0)), one, np.nextafter(one, np.float32(2)), 1.001, 1.1, 1.5, 1.99, 2.0, 2.01, math.e, 10.0, 1e5, 1e20, 3e38]
    c = np.array(v, dtype=np.float32)
    F = torch.tensor(c, device="cuda")[:, None, None, None].repeat(1, N, N, N)
    feat = torch.zeros(len(c), ef.EF_FEATURE_STRIDE, device="cuda")
    plan = _plan(N, ef.EF_PREC_F32)
    ef.ef_features(plan.handle, F, feat, len(c), log_input=1)
    ref = np.log(np.maximum(c, np.float32(1e-30)).astype(np.float64))
    got = feat.double().cpu().numpy()
    zero = int(np.argmax(np.abs(got[0])))                 # the zero mode's real part is the only one not near 0
    near = (c > 0.5) & (c < 2)
    bound = np.where(near, math.log(2) * 2.0 ** -22, 2.0 ** -22 * np.abs(ref)) + (1 + 3 * (N - 1)) * U * np.abs(ref)
    assert (np.abs(got[:, zero] - ref) <= bound).all()
    got[:, zero] = 0
    assert (np.abs(got).max(1) <= 3 * (N + 8) * U * np.abs(ref) + 1e-30).all()
    plan.close()


@pytest.mark.parametrize("N", [16, 24, 32, 48])
def test_log_of_general_cells_against_fp64(N):
    """Values over the whole range of a rarefied cell, a tenth of them at or below the clamp."""
    rng = np.random.default_rng(N)
    F = np.exp(rng.uniform(-75, 2, size=(3, N, N, N)))
    F[rng.uniform(size=F.shape) < 0.05] = 0.0
    F[0] = np.exp(rng.normal(0, 1e-3, size=F[0].shape))   # around 1
    F32 = torch.tensor(F, dtype=torch.float32, device="cuda")
    a = torch.zeros(3, ef.EF_FEATURE_STRIDE, device="cuda")
    b = torch.zeros_like(a)
    p32, p64 = _plan(N, ef.EF_PREC_F32), _plan(N, ef.EF_PREC_F64)
    ef.ef_features(p32.handle, F32, a, 3, log_input=1)
    ef.ef_features(p64.handle, F32.double(), b, 3, log_input=1)
    lnf = np.abs(np.log(np.maximum(F32.double().cpu().numpy(), 1e-30)))
    mean = lnf.mean((1, 2, 3))
    near = math.log(2) * 2.0 ** -22 * (lnf < math.log(2)).mean((1, 2, 3))
    bound = near + (2.0 ** -22 + U + 3 * (N + 8) * U) * mean
    assert (np.abs(a.double().cpu().numpy() - b.double().cpu().numpy()).max(1) <= bound).all()
    p32.close()
    p64.close()
