"""Tensor-core decode, several tiles per pipeline: consecutive tiles share the
columns of the accumulators and of the hidden rows, and a row's value depends
on its own query alone.  So a call whose pipelines take several tiles equals,
bit for bit, calls in which each takes one and no next tile follows.
"""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material

pytestmark = pytest.mark.gpu

FORMS = {
    "fast": dict(channels=16, c0=12, c1=12),
    "rows": dict(channels=9, c0=12, c1=12),
    "lattice": dict(channels=8, c0=12, c1=20),
    "third": dict(channels=12, c0=16, c1=12, act=1, out_act=1, interp0=1, hidden_layers=3),
    "float": dict(channels=8, c0=12, c1=12, bits0=8),
}


@pytest.mark.parametrize("form,precision", [(f, ntc.PREC_F16) for f in FORMS] + [("fast", ntc.PREC_F8)])
@pytest.mark.parametrize("filt", [ntc.FILTER_NEAREST, ntc.FILTER_STOCHASTIC, ntc.FILTER_TRILINEAR])
def test_equals_calls_of_one_tile_per_pipeline(form, precision, filt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = make_case(seed=170, width=256, height=128, **FORMS[form])
    if precision == ntc.PREC_F8:
        mat, md = device_material(case)
        q8 = [ntc.ntc_f8_quantize_weights(w, 64) for w in mat.weights]
        scale = torch.cat([s.reshape(1) for _, s in q8] + [torch.full((3,), 0.25, device=DEV)])
        mat = mat.with_(weights=[w for w, _ in q8], precision=ntc.PREC_F8, scale=scale, k_in=64)
    else:
        mat, md = device_material(case, precision=precision)
    rows = 128 // (8 if filt == ntc.FILTER_TRILINEAR else 1)
    one = torch.cuda.get_device_properties(0).multi_processor_count * 4 * rows  # <= a tile per pipeline
    n = 6 * one + 37
    q = gen.random_queries(n, md.mips, seed=4170)
    q[:, 2] += np.float32(0.3)
    q = torch.from_numpy(q).to(DEV)
    decode = lambda x: ntc.ntc_decode(mat, x, filter=filt, noise_seed=5)
    for _ in range(3):
        got = decode(q)
        assert ntc.ntc_device_status() == ntc.OK
        if filt == ntc.FILTER_STOCHASTIC:  # the jitter goes by the query's number
            assert torch.equal(got[:one], decode(q[:one]))
        else:
            for i in range(0, n, one):
                assert torch.equal(got[i:i + one], decode(q[i:i + one].clone()))
