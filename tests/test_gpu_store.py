"""Output stores of the tensor-core decode: rows of every width and type, and
a batch's output blocks at every alignment, against the single-material
decode of the same queries (same arithmetic: equal values)."""
import numpy as np
import pytest
import torch

import ntc_inputs as gen
import oracle
import paper_2305_17105_gb300 as ntc
from _cases import make_case
from _gpu import DEV, device_material, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ntc.lib()


def _uvl(q):
    return torch.from_numpy(np.ascontiguousarray(q, np.float32)).to(DEV)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.uint8])
@pytest.mark.parametrize("filt", [ntc.FILTER_NEAREST, ntc.FILTER_TRILINEAR])
@pytest.mark.parametrize("channels", [(4, 8, 12, 16), (3, 16, 5, 9), (2, 12, 6, 16)])
def test_batched_blocks_at_every_alignment(dtype, filt, channels):
    nq = [129, 131, 7, 1]   # blocks start at odd multiples of the channel counts
    mats = [device_material(make_case(seed=140 + i, width=64, height=64, channels=c, c0=12, c1=12,
                                      k_in=48), precision=ntc.PREC_F16)[0]
            for i, c in enumerate(channels)]
    qs = [gen.random_queries(n, 7, seed=4140 + i) for i, n in enumerate(nq)]
    for q in qs:
        q[:, 2] += np.float32(0.3)
    batch = ntc.Batch(mats, nq, filter=filt)
    guard = torch.full((int(batch.desc.total_outputs) + 64,), 7, dtype=dtype, device=DEV)
    out = ntc.ntc_decode_batched(batch, _uvl(np.concatenate(qs)), out=guard)
    assert ntc.ntc_device_status() == ntc.OK
    assert bool((out[-64:] == 7).all())
    for i, (m, q) in enumerate(zip(mats, qs)):
        got = out[batch.o_offsets[i]:batch.o_offsets[i + 1]].view(len(q), m.channels)
        assert torch.equal(got, ntc.ntc_decode(m, _uvl(q), out_dtype=dtype, filter=filt)), i


@pytest.mark.parametrize("precision", [ntc.PREC_F32, ntc.PREC_F16])
@pytest.mark.parametrize("channels", [1, 2, 7, 12, 16])
def test_trilinear_rows(precision, channels):
    """The exchange that leaves two channels of a query on each of its lanes:
    every channel count, a ragged last tile, wrapped and out-of-range texels."""
    case = make_case(seed=150, width=64, height=32, channels=channels, c0=8, c1=12, k_in=48)
    mat, md = device_material(case, precision=precision)
    rng = np.random.default_rng(150)
    q = np.empty((16 * 9 + 5, 3), np.float32)
    q[:, :2] = rng.uniform(-1.5, 2.5, (len(q), 2))
    q[:, 2] = rng.uniform(-0.5, md.mips + 0.5, len(q))
    tol = 2e-3 if precision == ntc.PREC_F16 else 1e-5   # the forms' decode bars
    for dtype in (torch.float32, torch.float16):
        got = to_np(ntc.ntc_decode(mat, _uvl(q), out_dtype=dtype, filter=ntc.FILTER_TRILINEAR))
        half = 5e-4 if dtype == torch.float16 else 0.0
        assert np.abs(got - md.decode_trilinear(q)).max() <= tol + half


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.uint8])
@pytest.mark.parametrize("channels", [8, 9, 13, 15])
@pytest.mark.parametrize("precision", ["f16", "f8"])
def test_rows_through_shared_memory(dtype, channels, precision):
    """A call whose rows pass through shared memory against one of 16 channels
    with the same first weights, stored row by row: the same values, nothing
    written past the last row (a tile boundary, a warp's and a ragged end)."""
    case = make_case(seed=151, width=64, height=64, channels=channels, c0=12, c1=12, k_in=64)
    mat, md = device_material(case, precision=ntc.PREC_F16)
    pad = lambda t: torch.cat([t, torch.zeros(16 - channels, *t.shape[1:], dtype=t.dtype, device=DEV)])
    full = mat.with_(channels=16, weights=mat.weights[:2] + [pad(mat.weights[2])],
                     biases=mat.biases[:2] + [pad(mat.biases[2])])
    if precision == "f8":
        scale = torch.tensor([2.0 ** -9, 2.0 ** -9, 2.0 ** -9, 2.0 ** -8, 2.0 ** -7, 2.0 ** -6],
                             device=DEV)
        e4 = lambda t: (t.float() * 512).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
        mat = mat.with_(weights=[e4(w) for w in mat.weights], precision=ntc.PREC_F8, scale=scale)
        full = full.with_(weights=[e4(w) for w in full.weights], precision=ntc.PREC_F8, scale=scale)
    for n in (1, 31, 33, 128, 161, 5 * 128 * 2 + 77):
        q = _uvl(gen.random_queries(n, md.mips, seed=4151))
        out = torch.full((n * channels + 64,), 7, dtype=dtype, device=DEV)
        got = ntc.ntc_decode(mat, q, out=out)[:n * channels].view(n, channels)
        assert torch.equal(got, ntc.ntc_decode(full, q, out_dtype=dtype)[:, :channels]), n
        assert bool((out[n * channels:] == 7).all())
    assert ntc.ntc_device_status() == ntc.OK
