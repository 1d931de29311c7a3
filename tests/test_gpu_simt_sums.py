"""How the FP32 adjoint sums weight gradients: a tile of 32 texels by itself,
then the tiles of a CTA, then the CTAs of a cluster, then in memory.

The decoder is built so that every texel adds its upstream gradient to each
element compared.  The first tile adds 2^24 in all and every other texel 1, so
each of the sums above is a multiple of 32 below 2^25 and exact in FP32, in any
order; a running total that took the texels one by one would drop the ones of
the first tile's CTA.
"""
import numpy as np
import pytest
import torch

import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 32 * 7, 32 * 152 * 2 + 64, 1 << 18])
def test_weight_gradients_are_summed_tile_by_tile(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = make_case(seed=0, width=64, height=64, channels=1, c0=8, c1=8, k_in=32, out_act=1)
    for a in case.weights + case.val0 + case.val1:
        a[...] = 0
    w1, b1, w2, b2, w3, b3 = case.weights
    b1[...], w2[...], w3[...] = 1, np.eye(64), 1
    mat, _ = device_material(case, packed=False)
    uvl = torch.tensor([[0.5, 0.5, 6.0]], device=DEV).repeat(n, 1)  # the one-texel mip: LOD input 1
    dout = torch.ones(n, 1, device=DEV)
    dout[:32] = 2.0 ** 19
    total = 2.0 ** 24 + n - 32
    w = [torch.zeros(a.shape, device=DEV) for a in (w1, w2, w3)]
    b = [torch.zeros(a.shape, device=DEV) for a in (b1, b2, b3)]
    zeros = lambda vals: [torch.zeros(v.shape, device=DEV) for v in vals]
    ntc.ntc_backward(mat, uvl, dout, ntc.grads_struct(mat, zeros(case.val0), zeros(case.val1), w, b))
    lod = case.c0 + case.c1 + 12
    for got in (w[0][:, lod], w[1], w[2], *b):
        assert (to_np(got) == total).all()
