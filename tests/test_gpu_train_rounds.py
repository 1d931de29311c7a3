"""The fused step at the sizes where its pipelines per CTA change (one, two,
three and two again, by the tiles of the call and the SMs), on the decoder of
unit contributions: every sum is a multiple of 1/16 below 2^20 and exact in
FP32 in any order, so the grids' gradients equal the oracle's."""
import numpy as np
import pytest
import torch

from _gpu import DEV, to_np
from test_gpu_runs import _backward, _unit_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [dict(c0=8, c1=12), dict(c0=7, c1=5), dict(c0=8, c1=8, interp0=1)])
@pytest.mark.parametrize("tiles", ["n", "n+1", "2n", "2n+1", "3n", "3n+1"])
def test_every_tile_counts_once(tiles, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rounds, _, more = tiles.partition("+")
    n = (int(rounds[:-1] or 1) * sms + int(more or 0)) * 128 - 5
    case = _unit_case(shape)
    xym = np.array([[0, 0, 6], [0, 0, 5], [1, 0, 5], [0, 1, 5], [1, 1, 5]], np.int32)[np.arange(n) * 7 % 5]
    g0 = [torch.zeros(v.shape, device=DEV) for v in case.val0]
    g1 = [torch.zeros(v.shape, device=DEV) for v in case.val1]
    md, dout = _backward(case, xym, g0, g1)
    ref = md.backward_xym(xym, dout.astype(np.float64))
    for got, want in zip(g0 + g1, ref["grid0"] + ref["grid1"]):
        np.testing.assert_array_equal(to_np(got), want)
