"""The FP32 adjoint's grid is a whole number of clusters: CTAs without a tile
add nothing to the weight gradients.

Few tiles, so that one to three CTAs of the last cluster get none, and large
first-layer weights, which would show in a bias gradient.  1e-4 relative per
tensor, as for every gradient of this kernel (FP32 sums of at most 10^3 terms).
"""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, rel_err, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_in,n", [(32, 1), (64, 32 * 5), (32, 32 * 6 - 3), (64, 32 * 9 + 1)])
def test_ctas_without_a_tile_add_nothing(k_in, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = make_case(seed=35, width=64, height=64, channels=3, c0=8, c1=8, k_in=k_in, out_act=1)
    case.weights[0] *= 64
    mat, md = device_material(case, packed=False)
    q = gen.random_texel_queries(64, 64, md.mips, n, seed=4035)
    dout = np.random.default_rng(35).standard_normal((n, 3)).astype(np.float32)
    m = np.floor(q[:, 2]).astype(np.int64)
    side = np.maximum(1, 64 >> m)
    xym = np.stack([np.floor(q[:, 0] * side), np.floor(q[:, 1] * side), m], 1).astype(np.int32)
    ref = md.backward_xym(xym, dout.astype(np.float64))["w"]
    qd, dd = torch.from_numpy(q).to(DEV), torch.from_numpy(dout).to(DEV)
    zeros = lambda arrays: [torch.zeros(a.shape, device=DEV) for a in arrays]
    for _ in range(20):
        w, b = zeros(case.weights[0::2]), zeros(case.weights[1::2])
        ntc.ntc_backward(mat, qd, dd, ntc.grads_struct(mat, zeros(case.val0), zeros(case.val1), w, b))
        for got, want in zip([t for pair in zip(w, b) for t in pair], ref):
            assert rel_err(to_np(got), want) <= 1e-4
