"""Where ef_mlp_forward may write: pairs of values, so rows of an even stride from an 8-byte boundary; anything
else is refused before a launch.  Outputs off the 16-byte boundaries that the tcgen05 product stores to go
through the mma.sync product.

Bar: rel-L2 1e-4 per 128 rows between the two products (FP32 accumulation in another order), the same bits
where both calls take one product."""
import numpy as np
import pytest
import torch

import paper_1704_07369_gb300 as ef

pytestmark = pytest.mark.gpu


def _net(B):
    return ef.MLP(100, 128, 2, 128, B, seed=4)


@pytest.mark.parametrize("B", [64, 20480])
@pytest.mark.parametrize("offset", [2, 4, 6])
def test_outputs_off_the_16_byte_boundary(B, offset):
    net = _net(B)
    X = torch.tensor(np.random.default_rng(B).normal(size=(B, 100)).astype(np.float32), device="cuda")
    ref = torch.empty(B, net.noutp, device="cuda")
    net.forward(X, ref, B)
    buf = torch.full((B * net.noutp + 16,), 7.0, device="cuda")
    Y = buf[offset:offset + B * net.noutp].view(B, net.noutp)
    net.forward(X, Y, B)
    torch.cuda.synchronize()
    assert net.status() == ef.EF_OK
    assert (buf[:offset] == 7.0).all() and (buf[offset + B * net.noutp:] == 7.0).all()
    if B == 64 or offset % 4 == 0:
        assert torch.equal(Y, ref)
    else:
        d = (Y.double() - ref.double()).view(-1, 128 * net.noutp).pow(2).sum(1)
        assert (d.sqrt() <= 1e-4 * ref.double().view(-1, 128 * net.noutp).pow(2).sum(1).sqrt()).all()


@pytest.mark.parametrize("offset", [1, 3])
def test_outputs_off_the_8_byte_boundary_are_refused(offset):
    B = 64
    net = _net(B)
    X = torch.zeros(B, 100, device="cuda")
    buf = torch.full((B * net.noutp + 16,), 7.0, device="cuda")
    with pytest.raises(ef.EfError) as e:
        net.forward(X, buf[offset:offset + B * net.noutp].view(B, net.noutp), B)
    assert e.value.status == "EF_ERR_INVALID_ARG"
    torch.cuda.synchronize()
    assert (buf == 7.0).all()
