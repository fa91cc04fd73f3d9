"""One hit that outweighs its batch, at the places where the training kernels
could lose it: alone in the second tile of a persistent block, in the last
and ragged tile of a block's third, and first and last of the batch.  The bound
is that of the other gradient tests, and the reference without the hit is far
past it.  Reference: the float64 oracle with bfloat16 operands."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import net as onet
from paper_1903_06838_gb300 import pd

torch = pytest.importorskip("torch")

TILE, BLOCKS_PER_SM = 8, 2
BOUND = 2.0 ** -8  # of a tensor's norm (tests/test_gpu_net_train.py)

#        hits of the batch from the hits of one round of all blocks, place of the hit
PLACES = {
    "alone_in_second_tile": (lambda r: r + 1, lambda n, r: n - 1),
    "last_of_ragged_third": (lambda r: 2 * r + 13, lambda n, r: n - 1),
    "first_of_second_round": (lambda r: 2 * r, lambda n, r: r),
    "last_of_first_round": (lambda r: r + 3, lambda n, r: r - 1),
    "first": (lambda r: r + 1, lambda n, r: 0),
}


def _case(place, sms):
    per_round = TILE * BLOCKS_PER_SM * sms
    n = PLACES[place][0](per_round)
    at = PLACES[place][1](n, per_round)
    rng = np.random.default_rng(n + at)
    flat = onet.flatten(onet.init_params(n)).astype(np.float32)
    x = rng.normal(0.0, 0.3, (n, 25)).astype(np.float32)
    x[:, 12] += rng.uniform(0.3, 3.0, n).astype(np.float32)
    counts = rng.integers(0, 5, n).astype(np.uint8)
    tgt = rng.uniform(-0.5, 0.5, (n, 2)).astype(np.float32)
    mask = np.zeros(n, np.uint8)
    # the only hit with an offset, and far from it
    x[at] = np.linspace(1.0, 3.0, 25)
    tgt[at] = (40.0, -40.0)
    mask[at] = 1
    return flat, (x, counts, tgt, mask), at


def _reference(flat, host):
    P = onet.unflatten(flat.astype(np.float64))
    loss, grads, _ = onet.loss_and_grad(P, host[0].astype(np.float64), *host[1:], 10.0,
                                        operand=onet.bf16)
    return loss, grads


@pytest.mark.parametrize("place", ["alone_in_second_tile", "first"])
def test_reference_without_the_hit_is_past_the_bound(place):
    flat, host, at = _case(place, 152)
    loss, ref = _reference(flat, host)
    less, without = _reference(flat, [np.delete(a, at, 0) for a in host])
    assert abs(loss - less) > 0.5 * abs(loss)
    for k in onet.ORDER:
        assert np.linalg.norm(ref[k] - without[k]) > 0.5 * np.linalg.norm(ref[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("place", list(PLACES))
def test_gradients_hold_the_hit(place):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    flat, host, _ = _case(place, sms)
    n = len(host[0])
    net = pd.pd_net_create(n, seed=0)
    pd.pd_net_set_params(net, flat)
    dev = [torch.from_numpy(a).cuda() for a in host]
    grads = torch.empty(pd.pd_net_num_params(), device="cuda")
    loss = torch.zeros(1, device="cuda")
    pd.pd_net_gradients(net, *(d.data_ptr() for d in dev), n, 1.0, 10.0, grads.data_ptr(),
                        loss.data_ptr())
    torch.cuda.synchronize()
    ref_loss, ref = _reference(flat, host)
    assert abs(loss.item() - ref_loss) < BOUND * abs(ref_loss)
    got = onet.unflatten(grads.cpu().numpy().astype(np.float64))
    for k in onet.ORDER:
        assert np.linalg.norm(got[k] - ref[k]) <= BOUND * np.linalg.norm(ref[k]), k
