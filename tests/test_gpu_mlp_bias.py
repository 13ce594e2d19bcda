"""Bias gradients of long training batches: sums of a layer's output gradients over the batch, against
FP64 sums of the same bf16 values.

Bars.  A sum of terms of one sign is added up in a tree of 7 roundings per 64 values, the blocks'
sums as an unevaluated pair, and rounded once: 8 u of it (u = 2^-24).  And no further from the FP64 sum,
rms over the columns, than 256 strided chains and a tree over them, emulated here."""
import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _bf16(x):
    return torch.tensor(x).bfloat16().float().numpy()


def _strided_sum(x):
    """FP32 sums over axis 0: 256 strided chains, a tree over each 32 of them, the 8 results in turn."""
    acc = np.zeros((256, x.shape[1]), np.float32)
    for k in range(0, x.shape[0], 256):
        part = x[k:k + 256]
        acc[:part.shape[0]] += part
    acc = acc.reshape(8, 32, -1)
    while acc.shape[1] > 1:
        h = acc.shape[1] // 2
        acc = acc[:, :h] + acc[:, h:]
    out = np.zeros(x.shape[1], np.float32)
    for w in range(8):
        out += acc[w, 0]
    return out


@pytest.mark.parametrize("B", [64, 4096, 16384])
@pytest.mark.parametrize("nout", [50, 320])
def test_bias_gradient_of_the_last_layer(B, nout):
    rng = np.random.default_rng(B + nout)
    net = ef.MLP(32, 64, 2, nout, B, seed=5)
    X = torch.tensor(rng.normal(size=(B, 32)).astype(np.float32), device="cuda")
    Y = torch.empty(B, net.noutp, device="cuda")
    net.forward(X, Y, B)
    y = Y[:, :nout].cpu().numpy()
    # y - t > 0, spread over eight binary orders, so that a long chain rounds at every step
    t = y - (2.0 ** rng.uniform(-8, 0, size=(B, nout))).astype(np.float32)
    loss = torch.zeros(1, device="cuda")
    grad = torch.zeros(net.nparams, device="cuda")
    net.grad(X, torch.tensor(t, device="cuda"), B, loss, grad)
    torch.cuda.synchronize()
    inv = np.float32(1.0) / (np.float32(B) * np.float32(nout))
    dy = _bf16(np.float32(2.0) * (y - t) * inv)
    assert (dy > 0).all()
    boff = net.layout()[-1][3]
    db = grad.cpu().numpy()[boff:boff + nout].astype(np.float64)
    ref = dy.astype(np.float64).sum(0)
    err = np.abs(db - ref) / ref
    assert err.max() <= 8 * U
    chain = np.abs(_strided_sum(dy).astype(np.float64) - ref) / ref
    assert np.sqrt((err ** 2).mean()) <= max(np.sqrt((chain ** 2).mean()), U / 2)
