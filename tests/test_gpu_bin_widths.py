"""Decode at the ends of the bin widths that the half-precision dequantisation
takes (powers of two in [2^-6, 2^6]), and one past: bilinear and learned G0,
4-bit (the fast layout) and 2-bit grids (the lattice form).  The first layer's
grid columns are scaled down by the same power of two, so the decoder sees
inputs of the usual size; FP16 decode's bar against the oracle, 2e-3."""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [2.0 ** -7, 2.0 ** -6, 32.0, 64.0, 128.0])
@pytest.mark.parametrize("shape", [
    dict(c0=12, c1=16), dict(c0=8, c1=12, bits0=2),
    dict(c0=12, c1=16, interp0=1), dict(c0=16, c1=12, interp0=1, hidden_layers=3),
    dict(c0=8, c1=12, bits0=2, interp0=1), dict(c0=12, c1=20, interp0=1, hidden_layers=3),
])
def test_bin_width(q, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = make_case(seed=172, width=128, height=64, channels=8, q0=q, q1=q, act=1, out_act=1, **shape)
    slots = (4 if case.interp0 else 1) * case.c0 + case.c1
    case.weights[0][:, :slots] *= np.float32(2.0 ** -4 / q)
    mat, md = device_material(case, precision=ntc.PREC_F16)
    uvl = gen.random_queries(3 * 128 + 17, md.mips, seed=4172)
    got = to_np(ntc.ntc_decode(mat, torch.from_numpy(uvl).to(DEV)))
    assert ntc.ntc_device_status() == ntc.OK
    assert np.abs(got - md.decode(uvl)).max() <= 2e-3
