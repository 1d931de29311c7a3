"""Edges of the tiled FP32 kernels: 32-query warp tiles and 32-texel training
tiles, their remainders, every number of tiles in flight (K decides it) and
channel counts that are not multiples of four.

Tolerances: decoded values 1e-5 absolute (an FP32 sum of at most 128 products
of magnitude <= 1, outputs in [0, 1] or of order 1).  Gradients 1e-4 relative
per tensor: FP32 sums of at most ~10^4 terms, each within 2^-24 of its value
and partly cancelling.
"""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import oracle
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, rel_err, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ntc.lib()


def _uvl(q):
    return torch.from_numpy(np.ascontiguousarray(q, np.float32)).to(DEV)


# K = 32..64: 16 warps; 96 with two hidden layers: 12, with three: 8; 128: 8
@pytest.mark.parametrize("shape", [
    dict(channels=16, c0=8, c1=8, k_in=32),
    dict(channels=1, c0=5, c1=3, bits0=1, bits1=8, k_in=64, act=1),
    dict(channels=9, c0=16, c1=12, k_in=96, act=1, out_act=1, interp0=1),
    dict(channels=8, c0=12, c1=20, k_in=96, act=1, out_act=1, interp0=1, hidden_layers=3),
    dict(channels=7, c0=20, c1=12, k_in=128, act=1, out_act=1, interp0=1, hidden_layers=3),
])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 16 * 32 + 1])
def test_decode_tile_edges(shape, n):
    case = make_case(seed=31, width=128, height=64, **shape)
    mat, md = device_material(case)
    q = gen.random_queries(n, md.mips, seed=4031)
    got = to_np(ntc.ntc_decode(mat, _uvl(q)))
    assert np.abs(got - md.decode(q)).max() < 1e-5
    q[:, 2] += np.float32(0.41)
    got = to_np(ntc.ntc_decode(mat, _uvl(q), filter=ntc.FILTER_TRILINEAR))
    assert np.abs(got - md.decode_trilinear(q)).max() < 1e-5


def test_decode_several_tiles_per_warp():
    """More tiles than the chip holds warps, and a ragged last one; the FP16
    weights of an FP16 material widened on load."""
    case = make_case(seed=32, width=256, height=256, channels=5, c0=8, c1=12, k_in=48)
    mat, md = device_material(case, precision=ntc.PREC_F16)
    n = 152 * 16 * 32 + 32 * 9 + 7
    q = gen.random_queries(n, md.mips, seed=4032)
    got = to_np(ntc.ntc_decode(mat, _uvl(q), flags=ntc.FLAG_SIMT))
    at = np.r_[0:200, n // 2:n // 2 + 200, n - 200:n]
    assert np.abs(got[at] - md.decode(q[at])).max() < 1e-5


@pytest.mark.parametrize("shape", [
    dict(channels=8, c0=8, c1=8, k_in=32),
    dict(channels=16, c0=16, c1=20, k_in=64, act=1),
    dict(channels=3, c0=7, c1=6, k_in=48, out_act=1),
    dict(channels=5, c0=8, c1=12, k_in=64, act=1, interp0=1),
])
@pytest.mark.parametrize("n", [1, 31, 33, 2 * 152 * 32 + 32 * 5 + 9])
def test_backward_tile_edges(shape, n):
    """1 and 31: one ragged tile; 33: two; the last: more tiles than CTAs."""
    case = make_case(seed=34, width=64, height=64, **shape)
    mat, md = device_material(case, packed=False)
    q = gen.random_texel_queries(64, 64, md.mips, n, seed=4034)
    dout = np.random.default_rng(34).standard_normal((n, case.channels)).astype(np.float32)
    zeros = lambda arrays: [torch.zeros(a.shape, device=DEV) for a in arrays]
    g0, g1 = zeros(case.val0), zeros(case.val1)
    w, b = zeros(case.weights[0::2]), zeros(case.weights[1::2])
    ntc.ntc_backward(mat, _uvl(q), _uvl(dout), ntc.grads_struct(mat, g0, g1, w, b))
    m = np.floor(q[:, 2]).astype(np.int64)
    side = np.maximum(1, 64 >> m)
    xym = np.stack([np.floor(q[:, 0] * side), np.floor(q[:, 1] * side), m], 1).astype(np.int32)
    ref = md.backward_xym(xym, dout.astype(np.float64))
    wb = [t for pair in zip(w, b) for t in pair]
    for got, want in zip(g0 + g1 + wb, ref["grid0"] + ref["grid1"] + ref["w"]):
        assert rel_err(to_np(got), want) <= 1e-4
