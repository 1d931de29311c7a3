"""Material.struct, packed in one call, against the fields of the ABI struct
set one by one (host tensors: only their addresses are looked at)."""
import pytest
import torch

import paper_2305_17105_gb300 as ntc


def _material(hidden_layers=2, **kw):
    grids = lambda sides, c: [torch.zeros(s, 2 * s, c) for s in sides]
    shapes = [(64, 32)] + [(64, 64)] * (hidden_layers - 1) + [(5, 64)]
    return ntc.Material(128, 64, 5, 8, 4, 4, 2, 0.125, 0.5, grids((16, 4, 1), 8), grids((8, 2, 1), 4),
                        [torch.zeros(s) for s in shapes], [torch.zeros(s[0]) for s in shapes], 32, **kw)


def _by_field(m):
    s = ntc.ntc_material()
    for f in ("width", "height", "channels", "mips", "levels", "c0", "c1", "bits0", "bits1", "q0", "q1",
              "encoding", "k_in", "act", "out_act", "precision", "interp0"):
        setattr(s, f, getattr(m, f))
    s.hidden, s.hidden_layers = 64, len(m.weights) - 1
    for j in range(m.levels):
        g0, g1 = m.grids0[j], m.grids1[j]
        s.lv[j].g0_h, s.lv[j].g0_w, s.lv[j].g1_h, s.lv[j].g1_w = *g0.shape[:2], *g1.shape[:2]
        s.lv[j].grid0, s.lv[j].grid1 = g0.data_ptr(), g1.data_ptr()
    at = [0, 1, len(m.weights) - 1]
    for l in range(3):
        s.w[l], s.b[l] = m.weights[at[l]].data_ptr(), m.biases[at[l]].data_ptr()
    if len(m.weights) == 4:
        s.w_h3, s.b_h3 = m.weights[2].data_ptr(), m.biases[2].data_ptr()
    if m.scale is not None:
        s.scale = m.scale.data_ptr()
    if m.codebook0 is not None:
        s.vq_books, s.codebook0 = m.codebook0.shape[0], m.codebook0.data_ptr()
    return s


@pytest.mark.parametrize("kw", [
    {}, dict(hidden_layers=3), dict(scale=torch.ones(6), act=1, out_act=1),
    dict(interp0=1, precision=ntc.PREC_F16, codebook0=torch.zeros(2, 256, 8)),
])
@pytest.mark.parametrize("levels", [3, 2, 1])
def test_equals_field_by_field(kw, levels):
    """Also with fewer levels than the material holds grids for."""
    m = _material(**kw).with_(levels=levels)
    assert bytes(m.struct) == bytes(_by_field(m))


def test_more_levels_than_grids_is_refused():
    with pytest.raises(IndexError):
        _material().with_(levels=4).struct
