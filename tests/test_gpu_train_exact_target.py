"""The training loss against a target that the decoder meets exactly: 255 is
1.0 (the product of 255 and the rounded 1/255 rounds to one), so an identity
output of one has no error, and the loss and every gradient are zero."""
import numpy as np
import pytest
import torch

import paper_2305_17105_gb300 as ntc
from _cases import make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, ntc.FLAG_CROPS])
@pytest.mark.parametrize("shape", [dict(c0=8, c1=8), dict(c0=16, c1=12, interp0=1, act=1),
                                   dict(c0=12, c1=12, hidden_layers=3)])
def test_no_error_no_gradient(shape, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = make_case(seed=0, width=64, height=64, channels=5, out_act=1, **shape)
    for a in case.weights:
        a[...] = 0
    case.weights[-1][...] = 1
    tr = ntc.Trainer(64, 64, 5, case.c0, case.c1, 4, 4, case.q0, case.q1, case.val0, case.val1,
                     case.weights[0::2], case.weights[1::2], case.k_in, ntc.PREC_F16, case.act, 1,
                     total_steps=10, interp0=case.interp0)
    target = ntc.Target([np.full((64 >> m, 64 >> m, 5), 255, np.uint8) for m in range(7)])
    loss = ntc.ntc_train_step(tr, target, 700, 3, flags=flags | ntc.FLAG_GRAD_ONLY).item()
    assert ntc.ntc_device_status() == ntc.OK
    assert loss == 0.0
    assert not torch.any(tr.grad)
