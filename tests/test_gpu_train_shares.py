"""The batched training step's shares: a CTA works for one material where the
materials' CTAs fit the grid, and takes an even share that crosses from one
material into the next where they do not (one large material beside many small
ones, more materials than SMs).  Every material's loss and gradient equal its
single-material step's: the same products, sums in another order (1e-5
relative, as for the other batches).
"""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import rel_err, to_np

pytestmark = pytest.mark.gpu

SHAPES = [dict(width=64, height=64, channels=6, c0=8, c1=8, k_in=32),
          dict(width=128, height=64, channels=12, c0=16, c1=12, k_in=48),
          dict(width=32, height=32, channels=3, c0=3, c1=5, k_in=32)]
BATCHES = {
    "one_tile_each": [100, 128, 1],
    "partly_filled": [385, 1300, 129, 0, 900],
    "a_round": [8000, 8000, 0, 8000, 8000, 8000],
    "rounds": [30_000, 77_001, 12_000],
    "one_large": [200_001] + [37, 128, 0, 129] * 15,
    "more_than_sms": [64 + 3 * (i % 40) for i in range(170)],
}


@pytest.mark.parametrize("name", list(BATCHES))
def test_equals_single_steps(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cases = [make_case(seed=180 + k, **s) for k, s in enumerate(SHAPES)]
    targets = [ntc.Target(gen.box_mip_chain_u8(gen.synthetic_texture(c.width, c.height, c.channels,
                                                                     seed=1180))) for c in cases]
    batches = BATCHES[name]
    trainers = []
    for i in range(len(batches)):
        c = cases[i % 3]
        w = c.weights
        tr = ntc.Trainer(c.width, c.height, c.channels, c.c0, c.c1, c.bits0, c.bits1, c.q0, c.q1, c.val0,
                         c.val1, w[0::2], w[1::2], c.k_in, ntc.PREC_F16, total_steps=50)
        tr.step_t.fill_(i % 7)
        trainers.append(tr)
    tb = ntc.TrainBatch(trainers, [targets[i % 3] for i in range(len(batches))], batches, 77,
                        flags=ntc.FLAG_GRAD_ONLY)
    loss = ntc.ntc_train_step_batched(tb).cpu().numpy()
    assert ntc.ntc_device_status() == ntc.OK
    for i, (tr, n) in enumerate(zip(trainers, batches)):
        got = to_np(tr.grad)
        if n == 0:
            assert loss[i] == 0 and not np.any(got)
            continue
        tr.grad.zero_()
        one = ntc.ntc_train_step(tr, targets[i % 3], n, 77 + i, flags=ntc.FLAG_GRAD_ONLY).item()
        assert abs(one - loss[i]) <= 1e-5 * one, i
        assert rel_err(got, to_np(tr.grad)) <= 1e-5, i
