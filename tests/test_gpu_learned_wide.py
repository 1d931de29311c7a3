"""Learned interpolation with more than 16 channels in both grids (K = 144
inside the tensor-core decode): packed 2- and 4-bit grids with two hidden
layers take the lattice form, with three the float form, whose pipelines
still fit in shared memory.  Against the oracle at the FP16 decode's bar,
2e-3.
"""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c0,b0,c1,b1", [(17, 4, 17, 4), (20, 4, 20, 4), (20, 2, 17, 4), (18, 4, 20, 2)])
@pytest.mark.parametrize("hidden_layers", [2, 3])
@pytest.mark.parametrize("channels", [8, 9, 15])
def test_both_grids_above_16_channels(c0, b0, c1, b1, hidden_layers, channels):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = make_case(seed=171, width=128, height=64, channels=channels, c0=c0, c1=c1, bits0=b0,
                     bits1=b1, act=1, out_act=1, interp0=1, hidden_layers=hidden_layers)
    mat, md = device_material(case, precision=ntc.PREC_F16)
    q = gen.random_queries(5 * 128 + 77, md.mips, seed=4171)
    q[:, 2] += np.float32(0.3)
    uvl = torch.from_numpy(q).to(DEV)
    for filt, want in ((ntc.FILTER_NEAREST, md.decode(q)),
                       (ntc.FILTER_TRILINEAR, md.decode_trilinear(q)),
                       (ntc.FILTER_STOCHASTIC, md.decode_stochastic(q, 5, 6))):
        got = to_np(ntc.ntc_decode(mat, uvl, filter=filt, noise_seed=5, noise_step=6))
        assert ntc.ntc_device_status() == ntc.OK
        assert np.abs(got - want).max() <= 2e-3, filt
