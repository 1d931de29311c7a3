"""The grid scatter of coherent texels (given queries, crops): a warp's 32
texels are merged into one reduction per run of equal cells.

The decoder is built so that every contribution to a cell is one power of two
(one live unit per layer, weights of one, upstream gradient 1/4), so every sum
below is exact in FP32 and the comparisons are equalities.
"""
import numpy as np
import pytest
import torch

import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, to_np

pytestmark = pytest.mark.gpu

SIDE, DOUT = 64, 0.25
SHAPES = [
    dict(c0=8, c1=8),
    dict(c0=16, c1=12),
    dict(c0=12, c1=16, act=1, hidden_layers=3),
    dict(c0=8, c1=8, interp0=1),            # the staged form: learned G0
    dict(c0=16, c1=12, interp0=1, act=1),
    dict(c0=12, c1=16, interp0=1, act=1, hidden_layers=3),
]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ntc.lib()


def _unit_case(shape):
    """One live unit per layer: Z = 8 + sum of the (zero) features, every
    derivative 1, so dX = dout at every grid slot."""
    case = make_case(seed=0, width=SIDE, height=SIDE, channels=1, out_act=1, **shape)
    slots = (4 if case.interp0 else 1) * case.c0 + case.c1
    for a in case.weights + case.val0 + case.val1:
        a[...] = 0
    case.weights[0][0, :slots] = 1
    for w in case.weights[2::2]:
        w[0, 0] = 1
    case.weights[1][0] = 8
    return case


def _texels(xym):
    side = np.maximum(1, SIDE >> xym[:, 2])
    return np.stack([(xym[:, 0] + 0.5) / side, (xym[:, 1] + 0.5) / side, xym[:, 2]],
                    1).astype(np.float32)


def _backward(case, xym, g0, g1):
    mat, md = device_material(case, precision=ntc.PREC_F16, packed=False)
    dout = np.full((len(xym), 1), DOUT, np.float32)
    ntc.ntc_backward(mat, torch.from_numpy(_texels(xym)).to(DEV), torch.from_numpy(dout).to(DEV),
                     ntc.grads_struct(mat, g0, g1,
                                      [torch.zeros(a.shape, device=DEV) for a in case.weights[0::2]],
                                      [torch.zeros(a.shape, device=DEV) for a in case.weights[1::2]]))
    assert ntc.ntc_device_status() == ntc.OK
    return md, dout


@pytest.mark.parametrize("shape", SHAPES)
def test_one_reduction_per_warp_of_equal_texels(shape):
    """Every texel is the one-texel mip's, and the gradients start at 32 x 2^23
    contributions: the sum of 32 is one unit in their last place, half of it
    would round away."""
    case = _unit_case(shape)
    n, last = 5 * 128 + 3 * 32, SIDE.bit_length() - 1
    xym = np.tile(np.array([[0, 0, last]], np.int32), (n, 1))
    # on the one-texel mip each of the four cells takes a quarter (learned G0: all)
    each = (DOUT if case.interp0 else DOUT / 4, DOUT / 4)
    g = [[torch.full(v.shape, e * 2.0 ** 28, device=DEV) for v in vals]
         for vals, e in zip((case.val0, case.val1), each)]
    md, dout = _backward(case, xym, *g)
    ref = md.backward_xym(xym, dout.astype(np.float64))
    for got, want, e in zip(g, (ref["grid0"], ref["grid1"]), each):
        assert np.count_nonzero(want[-1]) == 4 * want[-1].shape[-1]
        for a, b in zip(got, want):
            np.testing.assert_array_equal(to_np(a) - e * 2.0 ** 28, b)


@pytest.mark.parametrize("shape", SHAPES)
def test_runs_of_every_length(shape):
    """Runs of 1 to 40 texels over five texels of the two smallest mips, across
    the middle and the end of a warp's 32, and a ragged last tile."""
    case = _unit_case(shape)
    rng = np.random.default_rng(7)
    five = np.array([[0, 0, 6], [0, 0, 5], [1, 0, 5], [0, 1, 5], [1, 1, 5]], np.int32)
    pick = np.repeat(rng.integers(0, 5, 200), rng.integers(1, 41, 200))[:9 * 128 + 77]
    xym = five[pick]
    g0 = [torch.zeros(v.shape, device=DEV) for v in case.val0]
    g1 = [torch.zeros(v.shape, device=DEV) for v in case.val1]
    md, dout = _backward(case, xym, g0, g1)
    ref = md.backward_xym(xym, dout.astype(np.float64))
    for got, want in zip(g0 + g1, ref["grid0"] + ref["grid1"]):
        np.testing.assert_array_equal(to_np(got), want)
