"""The persistent tcgen05 product at the edges of its tiling: one and several tiles per CTA, an uneven last
round, each tile width, the shortest K (one block) and outputs wider apart than the network's.

Bar, per 128-row tile: rel-L2 1e-4 against the FP64 oracle with the same bf16 roundings (FP32
accumulation of at most 512 products, and single values on the other side of a rounding)."""
import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nin,nh,nout,B", [
    (32, 64, 64, 152 * 128),            # one tile of 64 columns per SM
    (200, 64, 50, 155 * 128),           # a last round of three tiles
    (64, 128, 192, 80 * 128),           # fewer tiles than SMs
    (60, 192, 320, 153 * 128),
    (100, 256, 256, 311 * 128),         # three rounds of 256 columns, the last uneven
])
@pytest.mark.parametrize("wide", [0, 4])
def test_forward_tiles(nin, nh, nout, B, wide):
    rng = np.random.default_rng(B + nh)
    net = ef.MLP(nin, nh, 2, nout, B, seed=3)
    X = rng.normal(size=(B, nin)).astype(np.float32)
    Y = torch.full((B, net.noutp + wide), 7.0, device="cuda")
    net.forward(torch.tensor(X, device="cuda"), Y, B)
    torch.cuda.synchronize()
    assert net.status() == ef.EF_OK
    y = Y.cpu().numpy()
    assert (y[:, net.noutp:] == 7.0).all()
    Xp = np.zeros((B, net.ninp))
    Xp[:, :nin] = X
    ref, _ = omlp.forward(omlp.unpack(net.params(), net.layout()), Xp, bf=True)
    d = ((y[:, :net.noutp] - ref) ** 2).reshape(B // 128, -1).sum(1)
    assert (np.sqrt(d) <= 1e-4 * np.sqrt((ref ** 2).reshape(B // 128, -1).sum(1))).all()
