"""Gradients of the learned network at the edges of its training kernels:
one hit, a full eight-hit tile and one more, around the 128-hit slices of the
fully connected layer's gradient, and one hit past one tile for each of the
persistent blocks.  Reference: the float64 oracle with bfloat16 operands."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import net as onet
from paper_1903_06838_gb300 import pd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(n, seed):
    rng = np.random.default_rng(seed)
    flat = onet.flatten(onet.init_params(seed)).astype(np.float32)
    x = rng.normal(0.0, 0.3, (n, 25))
    x[:, 12] += rng.uniform(0.3, 3.0, n)
    counts = rng.integers(0, 5, n).astype(np.uint8)
    tgt = rng.uniform(-0.5, 0.5, (n, 2)).astype(np.float32)
    mask = (rng.random(n) < 0.7).astype(np.uint8)
    mask[0] = 1
    net = pd.pd_net_create(4096, seed=0)
    pd.pd_net_set_params(net, flat)
    return net, onet.unflatten(flat.astype(np.float64)), (x.astype(np.float32), counts, tgt, mask)


@pytest.mark.parametrize("n", [1, 8, 9, 127, 129, 2433])
def test_gradients_at_tile_edges(n):
    net, P, host = _case(n, 10 + n)
    dev = [torch.from_numpy(a).cuda() for a in host]
    grads = torch.full((pd.pd_net_num_params() + 1,), 7.0, device="cuda")
    loss = torch.ones(1, device="cuda")  # the call adds to it
    # past the first float: four-byte alignment only
    pd.pd_net_gradients(net, *(d.data_ptr() for d in dev), n, float(host[3].sum()), 10.0,
                        grads.data_ptr() + 4, loss.data_ptr())
    again = torch.empty(pd.pd_net_num_params(), device="cuda")
    pd.pd_net_gradients(net, *(d.data_ptr() for d in dev), n, float(host[3].sum()), 10.0,
                        again.data_ptr(), 0)
    torch.cuda.synchronize()
    ref_loss, ref, _ = onet.loss_and_grad(P, host[0].astype(np.float64), *host[1:], 10.0,
                                          operand=onet.bf16)
    # float32 sums against float64 ones: a value next to a rounding boundary
    # may take the other bfloat16 (2^-8 of that value), so a whole gradient
    # differs by less than 2^-8 of its norm; the loss, computed from float32
    # outputs, by the same bound
    assert abs(loss.item() - 1.0 - ref_loss) < 2.0 ** -8 * abs(ref_loss)
    assert grads[0].item() == 7.0
    for g in (grads[1:], again):
        got = onet.unflatten(g.cpu().numpy().astype(np.float64))
        for k in onet.ORDER:
            a, c = got[k].ravel(), ref[k].ravel()
            assert np.linalg.norm(a - c) <= 2.0 ** -8 * np.linalg.norm(c), k
