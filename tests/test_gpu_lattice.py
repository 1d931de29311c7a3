"""The lattice form of the generic layout (packed grids of 2 and 4 bits off the
fast layout) against the float form, reached through the warpgroup-pipeline
kernel (K <= 48), and against the oracle.

Both forms build the same FP16 rows (every blended value is exact), so their
outputs differ at most by the order in which the tensor core adds a row's
products: 1e-6 for outputs in [0, 1].  Against the oracle: the FP16 decode's
bar, 2e-3.
"""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ntc.lib()
    yield
    ntc.ntc_set_decode_warpgroups(0)


def _uvl(q):
    return torch.from_numpy(np.ascontiguousarray(q, np.float32)).to(DEV)


def _queries(md, n=128 * 3 + 17):
    q = gen.random_queries(n, md.mips, seed=4160)
    q[:4] = [[0.0, 0.0, 0.0], [0.999999, 0.999999, 0.0], [np.nan, 2.0, 99.0], [0.5, -1.0, -3.0]]
    return q


# every cell size (1 to 16 bytes) and every group remainder of both widths
@pytest.mark.parametrize("c0,b0,c1,b1", [
    (1, 2, 2, 4), (3, 2, 4, 4), (5, 2, 3, 2), (8, 2, 12, 4), (9, 2, 7, 2), (12, 2, 10, 4),
    (16, 2, 1, 4), (17, 2, 4, 4), (20, 2, 12, 2), (4, 4, 20, 4), (17, 4, 9, 2), (12, 4, 18, 4),
    (2, 4, 1, 2),
])
@pytest.mark.parametrize("filt", [ntc.FILTER_NEAREST, ntc.FILTER_TRILINEAR, ntc.FILTER_STOCHASTIC])
def test_equals_the_float_form(c0, b0, c1, b1, filt):
    case = make_case(seed=160, width=128, height=64, channels=5, c0=c0, c1=c1, bits0=b0, bits1=b1,
                     k_in=48)
    mat, md = device_material(case, precision=ntc.PREC_F16)
    q = _queries(md)
    q[4:, 2] += np.float32(0.3)
    got = ntc.ntc_decode(mat, _uvl(q), filter=filt, noise_seed=3)
    ntc.ntc_set_decode_warpgroups(4)
    ref = ntc.ntc_decode(mat, _uvl(q), filter=filt, noise_seed=3)
    assert ntc.ntc_device_status() == ntc.OK
    # (a NaN coordinate has NaN trilinear weights in both)
    assert torch.allclose(got, ref, rtol=0, atol=1e-6, equal_nan=True)
    if filt == ntc.FILTER_NEAREST:
        assert np.abs(to_np(got) - md.decode(q)).max() <= 2e-3


@pytest.mark.parametrize("c0,b0,c1,b1", [(8, 2, 12, 4), (12, 4, 20, 4), (12, 2, 10, 4), (3, 2, 5, 2),
                                         (18, 4, 3, 4)])
@pytest.mark.parametrize("hidden_layers", [2, 3])
@pytest.mark.parametrize("channels", [9, 11, 16])
def test_learned_matches_oracle(c0, b0, c1, b1, hidden_layers, channels):
    """Learned interpolation (K up to 112), with the outputs stored by the row's
    thread (9 channels, 16) and through shared memory (11)."""
    case = make_case(seed=161, width=64, height=128, channels=channels, c0=c0, c1=c1, bits0=b0,
                     bits1=b1, act=1, out_act=1, interp0=1, hidden_layers=hidden_layers)
    mat, md = device_material(case, precision=ntc.PREC_F16)
    q = _queries(md)
    got = to_np(ntc.ntc_decode(mat, _uvl(q)))
    assert ntc.ntc_device_status() == ntc.OK
    assert np.abs(got - md.decode(q)).max() <= 2e-3
