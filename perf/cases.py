"""What this framework's performance is measured on.

A user of the library compresses materials (training steps, one material or
many side by side, FP16 or plain FP32, independent texels or crops), decodes
them (a streamed tile, a whole mip, a frame, random access at scale, many
materials at once; FP16, FP8-E4M3 or FP32) and differentiates through the
decode inside a larger program.  The listed cases are those calls at the
sizes of the repository's own workloads; ``draw`` gives others of the same
ranges.  ``exact`` restates the method in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_2305_17105_gb300 as ntc

DEV = "cuda"
HIDDEN = 64
START_STEP, TOTAL_STEPS = 1000, 100_000  # a training run resumed from a checkpoint
PRECISIONS = {"f32": ntc.PREC_F32, "f16": ntc.PREC_F16, "f8": ntc.PREC_F8}
FILTERS = {"nearest": ntc.FILTER_NEAREST, "trilinear": ntc.FILTER_TRILINEAR,
           "stochastic": ntc.FILTER_STOCHASTIC}
OUT = {"f32": torch.float32, "f16": torch.float16, "u8": torch.uint8}

# Grids of a plain material (channels x bits of G0 and of G1): the repository's
# workloads at 4 bits, and the four storage profiles of the paper's table.
PLAIN_GRIDS = [(8, 4, 8, 4), (12, 4, 12, 4), (16, 4, 16, 4), (16, 4, 12, 4)]
PROFILES = [(8, 2, 12, 4), (12, 4, 20, 4), (12, 2, 10, 4), (16, 4, 12, 4)]


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _decode(side, channels, grids, n, *, precision="f16", form="plain", hidden_layers=2,
            queries="random", filter="nearest", out="f16"):
    c0, b0, c1, b1 = grids
    return {"kind": "decode", "side": side, "channels": channels, "c0": c0, "bits0": b0, "c1": c1,
            "bits1": b1, "precision": precision, "form": form, "hidden_layers": hidden_layers,
            "n": n, "queries": queries, "filter": filter, "out": out}


def _train(side, channels, grids, batch, *, precision="f16", form="plain", hidden_layers=2,
           crops=False):
    c0, b0, c1, b1 = grids
    return {"kind": "train", "side": side, "channels": channels, "c0": c0, "bits0": b0, "c1": c1,
            "bits1": b1, "precision": precision, "form": form, "hidden_layers": hidden_layers,
            "batch": batch, "crops": crops}


def listed():
    return [
        # one page of a streamed virtual texture, filled when it is first seen:
        # the smallest call, where latency and launches count
        {"name": "tile_f16", **_decode(1024, 12, (12, 4, 12, 4), 1000, out="f16")},
        # the plain method, FP32 everywhere: every texel of mip 0 of a 256^2 x 8
        # material (the reference form a user checks the others against)
        {"name": "plain_f32", **_decode(256, 8, (8, 4, 8, 4), 65536, precision="f32",
                                        queries="raster", out="f32")},
        # random access at scale (rays that hit one material): 2^24 queries of a
        # 4096^2 x 16 material over its whole mip chain
        {"name": "random_f16", **_decode(4096, 16, (12, 4, 12, 4), 1 << 24)},
        # a rendered 4K frame with trilinear filtering, 8 decodes per pixel
        {"name": "frame_trilinear_f16", **_decode(4096, 16, (12, 4, 12, 4), 3840 * 2160,
                                                  queries="camera", filter="trilinear")},
        # the same view at 1080p in FP8-E4M3, written as 8-bit texels
        {"name": "frame_trilinear_f8", **_decode(4096, 16, (12, 4, 12, 4), 1920 * 1080,
                                                 precision="f8", queries="camera",
                                                 filter="trilinear", out="u8")},
        # the paper's decoder (learned interpolation, hardGELU, three hidden
        # layers) on its 0.5 profile: 20-channel G1, a ragged number of queries
        {"name": "paper_form_f16", **_decode(2048, 9, (12, 4, 20, 4), 1_000_003, form="paper",
                                             hidden_layers=3)},
        # a scene's materials decoded in one launch, uneven sizes, channel
        # counts and numbers of hits
        {"name": "batched_decode", "kind": "decode_batched", "materials": 24, "n": 1 << 20,
         "log2_lo": 8, "log2_hi": 12, "shapes": 7, "out": "f16"},
        # compression, plain method in FP32: one step of 4,096 texels
        {"name": "train_plain_f32", **_train(256, 8, (8, 4, 8, 4), 4096, precision="f32")},
        # compression of a 2048^2 x 12 material: one step of 2^18 texels
        {"name": "train_f16", **_train(2048, 12, (16, 4, 16, 4), 1 << 18)},
        # compression as the paper does it: its decoder, eight 256^2 crops
        {"name": "train_paper_crops", **_train(2048, 9, (16, 4, 12, 4), 8 * 65536, form="paper",
                                               crops=True)},
        # the materials of a scene compressed side by side, one step of each
        {"name": "train_batched", "kind": "train_batched", "materials": 10, "batch": 1 << 16,
         "log2_lo": 8, "log2_hi": 11, "shapes": 11},
        # the decode inside a larger differentiable program: forward, and the
        # adjoint into grids and weights, with quantisation noise
        {"name": "autograd_f16", "kind": "autograd", "side": 1024, "channels": 12, "c0": 12,
         "bits0": 4, "c1": 12, "bits1": 4, "precision": "f16", "form": "plain",
         "hidden_layers": 2, "n": 100_003, "noise": True},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["decode"] * 5 + ["decode_batched"] + ["train"] * 3 + ["train_batched"] +
                      ["autograd"])
    channels = rng.randint(3, 16)
    if kind == "decode":
        precision = rng.choice(["f16", "f16", "f8", "f32"])
        form = "plain" if precision == "f8" else rng.choice(["plain", "plain", "paper"])
        filt = rng.choice(["nearest", "nearest", "trilinear", "stochastic"])
        most = (1 << 18 if precision == "f32" else 1 << 23) // (8 if filt == "trilinear" else 1)
        return _decode(1 << rng.randint(8, 12), channels,
                       rng.choice(PROFILES if form == "paper" else PLAIN_GRIDS + PROFILES),
                       log(500, most), precision=precision, form=form,
                       hidden_layers=rng.choice([2, 3]) if precision != "f8" and form == "paper" else 2,
                       queries=rng.choice(["random", "camera", "raster"]), filter=filt,
                       out=rng.choice(["f16", "f16", "f32", "u8"]))
    if kind == "decode_batched":
        return {"kind": kind, "materials": rng.randint(4, 24), "n": log(4000, 1 << 20),
                "log2_lo": 8, "log2_hi": rng.randint(9, 12), "shapes": rng.randint(100, 10**6),
                "out": rng.choice(["f16", "f32", "u8"])}
    if kind == "train":
        precision = rng.choice(["f16", "f16", "f32"])
        form = "plain" if precision == "f32" else rng.choice(["plain", "paper"])
        return _train(1 << rng.randint(8, 11), channels,
                      rng.choice(PROFILES if form == "paper" else PLAIN_GRIDS),
                      log(1000, 1 << (15 if precision == "f32" else 18)), precision=precision,
                      form=form, hidden_layers=rng.choice([2, 3]) if form == "paper" else 2,
                      crops=rng.random() < 0.4)
    if kind == "train_batched":
        return {"kind": kind, "materials": rng.randint(3, 10), "batch": log(2000, 1 << 16),
                "log2_lo": 8, "log2_hi": rng.randint(9, 11), "shapes": rng.randint(100, 10**6)}
    c0, b0, c1, b1 = rng.choice(PLAIN_GRIDS)
    return {"kind": kind, "side": 1 << rng.randint(8, 11), "channels": channels, "c0": c0,
            "bits0": b0, "c1": c1, "bits1": b1, "precision": rng.choice(["f16", "f16", "f32"]),
            "form": "plain", "hidden_layers": 2, "n": log(1000, 1 << 17),
            "noise": rng.random() < 0.5}


def _parts(case):
    """The materials of a many-material case, each as a case of its own, with
    its queries ("n") or texels per step ("batch")."""
    r = torch.Generator().manual_seed(case["shapes"])
    pick = lambda lo, hi: int(torch.randint(lo, hi + 1, (1,), generator=r))
    out = []
    for _ in range(case["materials"]):
        side, channels = 1 << pick(case["log2_lo"], case["log2_hi"]), (8, 12, 16)[pick(0, 2)]
        c = (8, 12, 16)[pick(0, 2)] if case["kind"] == "train_batched" else 12
        one = {"side": side, "channels": channels, "c0": c, "bits0": 4, "c1": c, "bits1": 4,
               "precision": "f16", "form": "plain", "hidden_layers": 2, "crops": False}
        if case["kind"] == "decode_batched":
            one["n"] = case["n"] * pick(20, 100) // 100 + pick(0, 127)
        else:
            one["batch"] = case["batch"]
        out.append(one)
    return out


# ---------------------------------------------------------------------------
# sizes
# ---------------------------------------------------------------------------
def _used(c):
    return (4 if c["form"] == "paper" else 1) * c["c0"] + c["c1"] + 13


def _k_in(c):
    step = 32 if c["precision"] == "f8" else 16
    return -(-_used(c) // step) * step


def _pyramid(side):
    """[(G0 side, G1 side)] per feature level, largest first."""
    out = []
    while True:
        g0 = max(1, side >> (2 * len(out) + 2))
        if out and g0 < 4:
            return out
        out.append((g0, max(1, g0 >> 1)))


def _cell_bytes(c, bits):
    b = 1
    while 8 * b < c * bits:
        b *= 2
    return b


def _bin(bits):
    return 2.0 / (1 << bits)  # features in [-1, 1]


def _mlp_flops(c):
    return 2 * (_used(c) * HIDDEN + HIDDEN * HIDDEN * (c["hidden_layers"] - 1) +
                HIDDEN * c["channels"])


def _values(c):
    """Grid values and MLP weights and biases: what a training step updates."""
    grids = sum(a * a * c["c0"] + b * b * c["c1"] for a, b in _pyramid(c["side"]))
    return grids + HIDDEN * (_k_in(c) + 1) + (c["hidden_layers"] - 1) * HIDDEN * (HIDDEN + 1) + \
        c["channels"] * (HIDDEN + 1)


def work(case):
    kind = case["kind"]
    if kind in ("decode_batched", "train_batched"):
        one = {"kind": "decode", "filter": "nearest", "out": case["out"]} \
            if kind == "decode_batched" else {"kind": "train"}
        every = [work({**p, **one}) for p in _parts(case)]
        return {m: sum(w[m] for w in every) for m in ("bytes", "flops")}
    if kind == "decode":
        n, texels = case["n"], case["n"] * (8 if case["filter"] == "trilinear" else 1)
        cells = [_cell_bytes(case["c0"], case["bits0"]), _cell_bytes(case["c1"], case["bits1"])]
        grids = sum(a * a * cells[0] + b * b * cells[1] for a, b in _pyramid(case["side"]))
        touched = min(grids, 4 * texels * sum(cells))
        element = {"f32": 4, "f16": 2, "u8": 1}[case["out"]]
        return {"bytes": n * (12 + case["channels"] * element) + touched,
                "flops": texels * _mlp_flops(case)}
    if kind == "train":  # parameters and both moments read and written, the batch's target texels read
        return {"bytes": 24 * _values(case) + case["batch"] * case["channels"],
                "flops": 3 * case["batch"] * _mlp_flops(case)}
    # autograd: the queries and upstream gradient in, the values read, their gradient and the output written
    n = case["n"]
    return {"bytes": n * (12 + 8 * case["channels"]) + 8 * _values(case),
            "flops": 3 * n * _mlp_flops(case)}


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _model(case, g, packed):
    """Grid indices (as an exported material has them: bell-shaped over the
    levels) or float values uniform over the clamp range, and MLP weights
    U(+-1/sqrt(fan in)), layer order."""
    grids0, grids1 = [], []
    for a, b in _pyramid(case["side"]):
        for side, c, bits, out in ((a, case["c0"], case["bits0"], grids0),
                                   (b, case["c1"], case["bits1"], grids1)):
            n = 1 << bits
            if packed:
                v = torch.randn(side, side, c, generator=g, device=DEV) * (n / 5) + n / 2
                out.append(v.round().clamp(0, n - 1).to(torch.int32))
            else:
                out.append((_rand(g, side, side, c) * (n - 0.5) - (n - 1) / 2) * _bin(bits))
    w, b = [], []
    k = _k_in(case)
    shapes = [(k, HIDDEN)] + [(HIDDEN, HIDDEN)] * (case["hidden_layers"] - 1) + \
        [(HIDDEN, case["channels"])]
    for i, (fi, fo) in enumerate(shapes):
        bound = 1.0 / math.sqrt(_used(case) if i == 0 else fi)
        w.append((_rand(g, fo, fi) * 2 - 1) * bound)
        b.append((_rand(g, fo) * 2 - 1) * bound)
    w[0][:, _used(case):] = 0
    return grids0, grids1, w, b


def _mips(case):
    return case["side"].bit_length()


def _queries(case, g):
    """[n, 3] rows (u, v, lod)."""
    n, mips, side = case["n"], _mips(case), case["side"]
    if case.get("queries", "random") == "random":
        q = _rand(g, n, 3)
        q[:, 2] = torch.floor(q[:, 2] * mips)
    elif case["queries"] == "raster":  # texel centres of mip 0, row by row, from a random row on
        i = torch.arange(n, device=DEV) + side * int(torch.randint(0, side, (1,), generator=g, device=DEV))
        q = torch.stack([(i % side + 0.5) / side, (i // side % side + 0.5) / side,
                         torch.zeros(n, device=DEV)], dim=1)
    else:  # a pinhole camera 1.5 units above a textured plane, pitched about 60 degrees
        px_w = max(1, int(math.sqrt(n * 16 / 9)))
        px_h = -(-n // px_w)
        turn = (float(_rand(g, 1)) - 0.5) * 0.2
        pitch = math.radians(60) + turn
        i = torch.arange(n, device=DEV)
        sx, sy = (i % px_w).double() + 0.5, torch.div(i, px_w, rounding_mode="floor").double() + 0.5

        def hit(x, y):
            nx, ny = 2 * x / px_w - 1, (1 - 2 * y / px_h) * px_h / px_w
            up = math.sin(pitch) * ny - math.cos(pitch)
            t = 1.5 / (-up).clamp_min(1e-6)
            return 0.25 * t * nx + turn, 0.25 * t * (math.sin(pitch) + math.cos(pitch) * ny)

        (u, v), (u1, v1), (u2, v2) = hit(sx, sy), hit(sx + 1, sy), hit(sx, sy + 1)
        foot = torch.maximum(torch.hypot(u1 - u, v1 - v), torch.hypot(u2 - u, v2 - v)) * side
        q = torch.stack([u % 1.0, v % 1.0, torch.log2(foot.clamp_min(1e-30)).clamp(0, mips - 1)],
                        dim=1).float()
    q[:, :2].clamp_(max=1 - 2.0 ** -24)
    return q.float().contiguous()


def _pack(idx, bits):
    """[h, w, c] indices -> uint8 [h, w, cell bytes], channel ch at bits [ch b, (ch + 1) b)."""
    h, w, c = idx.shape
    per = 8 // bits
    cb = _cell_bytes(c, bits)
    v = F.pad(idx, (0, cb * per - c)).view(h, w, cb, per)
    return (v << (bits * torch.arange(per, device=DEV, dtype=torch.int32))).sum(-1).to(torch.uint8)


def _forms(case):
    paper = case["form"] == "paper"
    return {"act": ntc.ACT_HARDGELU if paper else ntc.ACT_RELU,
            "out_act": ntc.OUT_IDENTITY if paper else ntc.OUT_SIGMOID,
            "interp0": ntc.INTERP_LEARNED if paper else ntc.INTERP_BILINEAR}


def _f8_scales(case, w):
    """Weight scales max|W| / 448 and fixed activation scales of the E4M3 form."""
    return [float(x.abs().max()) / 448.0 for x in w] + [2.0 ** -8, 2.0 ** -7, 2.0 ** -6]


def _material(case, g):
    """A compressed material as a program that loaded one has it."""
    grids0, grids1, w, b = _model(case, g, True)
    scale = None
    if case["precision"] == "f16":
        w = [x.half().contiguous() for x in w]
    elif case["precision"] == "f8":
        s = _f8_scales(case, w)
        scale = torch.tensor(s, device=DEV)
        w = [(x / scale[i]).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
             for i, x in enumerate(w)]
    return ntc.Material(case["side"], case["side"], case["channels"], case["c0"], case["c1"],
                        case["bits0"], case["bits1"], _bin(case["bits0"]), _bin(case["bits1"]),
                        [_pack(x, case["bits0"]) for x in grids0],
                        [_pack(x, case["bits1"]) for x in grids1], w, b, _k_in(case),
                        PRECISIONS[case["precision"]], scale=scale, **_forms(case))


def _texture(case, g):
    """8-bit mip chain: smooth multi-octave fields mixed across the channels."""
    side, c = case["side"], case["channels"]
    base = torch.zeros(4, side, side, device=DEV)
    for o in range(5):
        lat = _rand(g, 1, 4, min(side, 8 << o), min(side, 8 << o))
        base += 0.5 ** o * F.interpolate(lat, size=(side, side), mode="bilinear", align_corners=False)[0]
    mix = _rand(g, c, 4) + 0.05
    t = torch.einsum("cb,bhw->chw", mix / mix.sum(1, keepdim=True), base) / 2
    t = (0.9 * t + 0.1 * _rand(g, c, side, side))[None].clamp(0, 1)
    chain = []
    while True:
        chain.append((t[0] * 255).round().to(torch.uint8).permute(1, 2, 0).contiguous())
        if t.shape[-1] == 1:
            return chain
        t = F.avg_pool2d(t, 2)


def _flat(tensors):
    """Offsets of a trainer's parameter array: every tensor on 8 floats."""
    offs, n = [], 0
    for t in tensors:
        offs.append(n)
        n += (t.numel() + 7) // 8 * 8
    return offs, n


def _train_inputs(case, g):
    grids0, grids1, w, b = _model(case, g, False)
    tensors = grids0 + grids1 + [x for pair in zip(w, b) for x in pair]
    offs, n = _flat(tensors)
    # moments of a run some steps in: about the size of one batch's gradient
    size = torch.full((n,), 0.02 / (case["batch"] * case["channels"]), device=DEV)
    size[offs[len(grids0) + len(grids1)]:] = 2e-4
    m = torch.randn(n, generator=g, device=DEV) * size
    v = (size * (0.5 + _rand(g, n))) ** 2
    return grids0, grids1, w, b, m, v, _texture(case, g)


def _state(case, params, m, v):
    """The updated state of a step: parameters and both moments, the grids' and
    the MLP's part of each."""
    at = _flat([torch.empty(a * a * case["c0"], device="meta") for a, _ in _pyramid(case["side"])] +
               [torch.empty(a * a * case["c1"], device="meta") for _, a in _pyramid(case["side"])])[1]
    return {part: {"params": params[s], "m": m[s], "v": v[s]}
            for part, s in (("grids", slice(0, at)), ("mlp", slice(at, None)))}


def _trainer(case, g):
    grids0, grids1, w, b, m, v, chain = _train_inputs(case, g)
    host = lambda x: [t.cpu().numpy() for t in x]
    tr = ntc.Trainer(case["side"], case["side"], case["channels"], case["c0"], case["c1"],
                     case["bits0"], case["bits1"], _bin(case["bits0"]), _bin(case["bits1"]),
                     host(grids0), host(grids1), host(w), host(b), _k_in(case),
                     PRECISIONS[case["precision"]], total_steps=TOTAL_STEPS, **_forms(case))
    tr.adam_m.copy_(m)
    tr.adam_v.copy_(v)
    tr.step_t.fill_(START_STEP)
    return tr, ntc.Target(host(chain))


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    s = {"case": case, "seed": int(seed)}
    if kind == "decode":
        s["material"] = _material(case, g)
        s["uvl"] = _queries(case, g)
    elif kind == "decode_batched":
        parts = _parts(case)
        s["batch"] = ntc.Batch([_material(p, g) for p in parts], [p["n"] for p in parts])
        s["uvl"] = torch.cat([_queries(p, g) for p in parts])
    elif kind == "train":
        s["trainer"], s["target"] = _trainer(case, g)
        tr = s["trainer"]
        s["updated"] = _state(case, tr.params, tr.adam_m, tr.adam_v)
    elif kind == "train_batched":
        parts = _parts(case)
        pairs = [_trainer(p, g) for p in parts]
        s["batch"] = ntc.TrainBatch([t for t, _ in pairs], [t for _, t in pairs],
                                    [p["batch"] for p in parts], int(seed))
        s["updated"] = [_state(p, t.params, t.adam_m, t.adam_v) for p, (t, _) in zip(parts, pairs)]
    else:
        grids0, grids1, w, b = _model(case, g, False)
        s["grids0"], s["grids1"], s["w"], s["b"] = (
            [x.contiguous().requires_grad_() for x in v] for v in (grids0, grids1, w, b))
        s["proto"] = ntc.Material(case["side"], case["side"], case["channels"], case["c0"],
                                  case["c1"], case["bits0"], case["bits1"], _bin(case["bits0"]),
                                  _bin(case["bits1"]), grids0, grids1, w, b, _k_in(case),
                                  PRECISIONS[case["precision"]], **_forms(case))
        s["uvl"] = _queries(case, g)
        s["dout"] = torch.randn(case["n"], case["channels"], generator=g, device=DEV) / case["n"]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "decode":
        return ntc.ntc_decode(s["material"], s["uvl"], out_dtype=OUT[case["out"]],
                              filter=FILTERS[case["filter"]], noise_seed=s["seed"])
    if kind == "decode_batched":
        return ntc.ntc_decode_batched(s["batch"], s["uvl"], out_dtype=OUT[case["out"]])
    if kind == "train":
        loss = ntc.ntc_train_step(s["trainer"], s["target"], case["batch"], s["seed"],
                                  flags=ntc.FLAG_CROPS if case["crops"] else 0)
        return {"loss": loss, "updated": s["updated"]}
    if kind == "train_batched":
        loss = ntc.ntc_train_step_batched(s["batch"])
        return {"loss": loss, "updated": s["updated"]}
    leaves = s["grids0"] + s["grids1"] + s["w"] + s["b"]
    y = ntc.decode_autograd(s["proto"], s["uvl"], s["grids0"], s["grids1"], s["w"], s["b"],
                            noise=(s["seed"], START_STEP) if case["noise"] else None)
    return {"y": y, "grads": list(torch.autograd.grad(y, leaves, s["dout"]))}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
_M64 = (1 << 64) - 1


def _mix(x):
    """SplitMix64 of a Python integer."""
    z = (x + 0x9E3779B97F4A7C15) & _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _signed(x):
    return x - (1 << 64) if x >> 63 else x


def _shr(x, s):
    return (x >> s) & ((1 << (64 - s)) - 1)


def _mix_t(x):
    """SplitMix64 of an int64 tensor (the bits of unsigned values)."""
    z = x + _signed(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _key(seed, stream):
    return _signed(_mix((seed & _M64) ^ _mix(stream & _M64)))


def _side_of(case, m):
    return max(1, case["side"] >> m)


def _texels(case, seed, step, batch):
    """The training texels (x, y, mip) of a step."""
    key, mips = _key(seed, 2 * step), _mips(case)
    i = torch.arange(batch, device=DEV, dtype=torch.int64)

    def lod(c0, c1):
        h0, k = _mix_t(key ^ c0), _shr(_mix_t(key ^ c1), 40) + 1
        m = torch.zeros_like(k)
        for t in range(1, 13):
            m = torch.where(k <= 1 << (24 - 2 * t), t, m)
        return torch.where(_shr(h0, 40) < 838861, ((h0 & 0xFFFFFFFF) * mips) >> 32, m).clamp(max=mips - 1)

    if not case["crops"]:
        m, h = lod(4 * i, 4 * i + 1), _mix_t(key ^ (4 * i + 2))
        side = torch.tensor([_side_of(case, t) for t in range(mips)], device=DEV)[m]
        return ((h & 0xFFFFFFFF) * side) >> 32, (_shr(h, 32) * side) >> 32, m
    m = lod(torch.zeros_like(i), torch.ones_like(i))
    side = _side_of(case, int(m[0]))
    h = _mix_t(key ^ (4 * (i // 65536) + 2))
    return ((((h & 0xFFFFFFFF) * side) >> 32) + i % 256) % side, \
        (((_shr(h, 32) * side) >> 32) + i // 256 % 256) % side, m


def _noise(grid, key, level, which, q):
    """A grid's quantisation noise of one step."""
    h, w, c = grid.shape
    pairs = (c + 1) // 2
    cell = torch.arange(h * w, device=DEV, dtype=torch.int64)[:, None]
    ch = torch.arange(c, device=DEV, dtype=torch.int64)[None]
    d = _mix_t(key ^ (((2 * level + which) << 40) | (cell * pairs + ch // 2)))
    b = torch.where(ch % 2 == 1, _shr(d, 16) & 0xFFFFFF, _shr(d, 40))
    return ((b.double() * 2.0 ** -24 - 0.5) * q).view(h, w, c)


def _taps(x, side, gside):
    p = (x.double() + 0.5) / side * gside - 0.5
    i0 = torch.floor(p)
    f = p - i0
    i0 = i0.long()
    return i0.clamp(0, gside - 1), (i0 + 1).clamp(0, gside - 1), f


def _rows(case, grids0, grids1, x, y, m):
    """MLP input rows of texels (x, y) of mips m."""
    rows = torch.zeros(x.numel(), _k_in(case), dtype=torch.float64, device=DEV)
    mips, levels = _mips(case), len(grids0)
    tri = lambda t: 4 * (t - torch.floor(t) - 0.5).abs() - 1
    learned = case["form"] == "paper"
    w0 = case["c0"] * (4 if learned else 1)
    for mip in range(mips):
        at = torch.nonzero(m == mip).view(-1)
        if not at.numel():
            continue
        j = min(levels - 1, 0 if mip < 4 else (mip - 2) // 2)
        side = _side_of(case, mip)
        xs, ys = x[at], y[at]
        feats = []
        for k, grid in enumerate((grids0[j], grids1[j])):
            gs = grid.shape[0]
            (a0, a1, fx), (b0, b1, fy) = _taps(xs, side, gs), _taps(ys, side, gs)
            flat = grid.reshape(gs * gs, -1)
            taps = [flat[b * gs + a] for b in (b0, b1) for a in (a0, a1)]
            if learned and k == 0:
                feats += taps
            else:
                fx, fy = fx[:, None], fy[:, None]
                feats.append((taps[0] * (1 - fx) + taps[1] * fx) * (1 - fy) +
                             (taps[2] * (1 - fx) + taps[3] * fx) * fy)
        for c in (xs, ys):
            for period in (8, 4, 2):
                t = (c.double() + 0.5) / period
                feats += [tri(t - 0.25)[:, None], tri(t)[:, None]]
        feats.append(torch.full((at.numel(), 1), mip / (mips - 1) if mips > 1 else 0.0,
                                dtype=torch.float64, device=DEV))
        r = torch.cat(feats, 1)
        assert r.shape[1] == w0 + case["c1"] + 13
        rows = rows.index_put((at,), F.pad(r, (0, rows.shape[1] - r.shape[1])))
    return rows


def _mlp(case, rows, w, b, scale=None):
    act = (lambda z: z * (z / 3 + 0.5).clamp(0, 1)) if case["form"] == "paper" else torch.relu
    for i, (wi, bi) in enumerate(zip(w, b)):
        if scale is not None:  # E4M3 inputs in units of the layer's activation scale
            s = scale[3 + i]
            rows = (rows / s).float().clamp(-448, 448).to(torch.float8_e4m3fn).double() * s
        rows = rows @ wi.T + bi
        if i + 1 < len(w):
            rows = act(rows)
    return rows if case["form"] == "paper" else torch.sigmoid(rows)


def _exact_decode(case, g, seed):
    """The 64-bit decode of one material, and its queries' place in the input stream."""
    idx0, idx1, w, b = _model(case, g, True)
    deq = lambda v, bits: [(i.double() - ((1 << (bits - 1)) - 1)) * _bin(bits) for i in v]
    grids0, grids1 = deq(idx0, case["bits0"]), deq(idx1, case["bits1"])
    scale = None
    if case["precision"] == "f16":
        w = [x.half() for x in w]
    elif case["precision"] == "f8":
        scale = [float(v) for v in torch.tensor(_f8_scales(case, w))]
        s = torch.tensor(scale, device=DEV)
        w = [(x / s[i]).clamp(-448, 448).to(torch.float8_e4m3fn).double() * s[i].double()
             for i, x in enumerate(w)]
    w, b = [x.double() for x in w], [x.double() for x in b]

    def decode(uvl, first=0):
        out = []
        for at in range(0, uvl.shape[0], 1 << 19):
            out.append(_exact_chunk(case, grids0, grids1, w, b, scale, uvl[at:at + (1 << 19)],
                                    first + at, seed))
        return torch.cat(out)

    return decode


def _exact_chunk(case, grids0, grids1, w, b, scale, uvl, first, seed):
    mips = _mips(case)
    sides = torch.tensor([_side_of(case, t) for t in range(mips)], device=DEV)
    u, v, lod = uvl[:, 0], uvl[:, 1], uvl[:, 2].clamp(0, mips - 1)
    if case.get("filter", "nearest") == "nearest":
        m = torch.floor(lod).long()
        s = sides[m]
        x, y = torch.floor(u.double() * s).long(), torch.floor(v.double() * s).long()
        return _mlp(case, _rows(case, grids0, grids1, x, y, m), w, b, scale)
    if case["filter"] == "stochastic":
        i = torch.arange(first, first + uvl.shape[0], device=DEV, dtype=torch.int64)
        h = _mix_t(_key(seed, 2) ^ i)
        m = torch.floor(lod + (h & 0xFFFF).float() / 65536).long().clamp(max=mips - 1)
        s = sides[m]
        at = lambda c, bits: (torch.floor((c * s.float() - 0.5) + bits.float() * 2.0 ** -24).long() % s)
        x, y = at(u, _shr(h, 40)), at(v, _shr(h, 16) & 0xFFFFFF)
        return _mlp(case, _rows(case, grids0, grids1, x, y, m), w, b, scale)
    out = 0
    m0 = torch.floor(lod).long()
    t = lod.double() - m0
    for m, wl in ((m0, 1 - t), ((m0 + 1).clamp(max=mips - 1), t)):
        s = sides[m]
        px, py = u.double() * s - 0.5, v.double() * s - 0.5
        x0, y0 = torch.floor(px), torch.floor(py)
        fx, fy = px - x0, py - y0
        for dy in (0, 1):
            for dx in (0, 1):
                wt = wl * (fx if dx else 1 - fx) * (fy if dy else 1 - fy)
                rows = _rows(case, grids0, grids1, (x0.long() + dx) % s, (y0.long() + dy) % s, m)
                out = out + wt[:, None] * _mlp(case, rows, w, b, scale)
    return out


def _noisy(case, grids0, grids1, seed, step):
    key = _key(seed, 2 * step + 1)
    return ([v + _noise(v, key, j, 0, _bin(case["bits0"])) for j, v in enumerate(grids0)],
            [v + _noise(v, key, j, 1, _bin(case["bits1"])) for j, v in enumerate(grids1)])


def _stored(case, w):
    """The weights the forward sees."""
    return [(x.half() if case["precision"] == "f16" else x).double() for x in w]


def _exact_step(case, g, seed):
    grids0, grids1, w, b, m, v, chain = _train_inputs(case, g)
    L = len(grids0)
    leaf = lambda t: t.double().requires_grad_()
    g0, g1, wl, bl = ([leaf(t) for t in x] for x in (grids0, grids1, _stored(case, w), b))
    x, y, mip = _texels(case, seed, START_STEP, case["batch"])
    target = torch.zeros(case["batch"], case["channels"], dtype=torch.float64, device=DEV)
    for t, tex in enumerate(chain):
        at = torch.nonzero(mip == t).view(-1)
        target[at] = tex[y[at], x[at]].double() / 255
    n0, n1 = _noisy(case, g0, g1, seed, START_STEP)
    loss = ((_mlp(case, _rows(case, n0, n1, x, y, mip), wl, bl) - target) ** 2).mean()
    mlp = [t for pair in zip(wl, bl) for t in pair]
    grads = torch.autograd.grad(loss, g0 + g1 + mlp, allow_unused=True)
    tensors = grids0 + grids1 + [t for pair in zip(w, b) for t in pair]
    offs, n = _flat(tensors)
    params, m, v = torch.zeros(n, dtype=torch.float64, device=DEV), m.double(), v.double()
    decay = 0.5 * (1 + math.cos(math.pi * START_STEP / TOTAL_STEPS))
    for i, (o, t, gr) in enumerate(zip(offs, tensors, grads)):
        at = slice(o, o + t.numel())
        gr = torch.zeros_like(t.double()) if gr is None else gr
        m[at] = 0.9 * m[at] + 0.1 * gr.reshape(-1)
        v[at] = 0.999 * v[at] + 0.001 * gr.reshape(-1) ** 2
        lr = (0.01 if i < 2 * L else 0.005) * decay
        p = t.double().reshape(-1) - lr * (m[at] / (1 - 0.9 ** (START_STEP + 1))) / \
            (torch.sqrt(v[at] / (1 - 0.999 ** (START_STEP + 1))) + 1e-8)
        if i < 2 * L:
            bits = case["bits0"] if i < L else case["bits1"]
            p = p.clamp(-((1 << bits) - 1) / 2 * _bin(bits), (1 << bits) / 2 * _bin(bits))
        params[at] = p
    return {"loss": loss.detach().view(1), "updated": _state(case, params, m, v)}


def exact(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "decode":
        if case["out"] == "u8":
            return None
        decode = _exact_decode(case, g, int(seed))
        return decode(_queries(case, g))
    if kind == "decode_batched":
        if case["out"] == "u8":
            return None
        parts = _parts(case)
        decodes = [_exact_decode(p, g, int(seed)) for p in parts]
        return torch.cat([d(_queries(p, g)).view(-1) for d, p in zip(decodes, parts)])
    if kind == "train":
        return _exact_step(case, g, int(seed))
    if kind == "train_batched":
        steps = [_exact_step(p, g, int(seed) + i) for i, p in enumerate(_parts(case))]
        return {"loss": torch.cat([s["loss"] for s in steps]),
                "updated": [s["updated"] for s in steps]}
    grids0, grids1, w, b = _model(case, g, False)
    uvl = _queries(case, g)
    dout = torch.randn(case["n"], case["channels"], generator=g, device=DEV) / case["n"]
    leaf = lambda t: t.double().requires_grad_()
    g0, g1, wl, bl = ([leaf(t) for t in v] for v in (grids0, grids1, _stored(case, w), b))
    n0, n1 = _noisy(case, g0, g1, int(seed), START_STEP) if case["noise"] else (g0, g1)
    mip = torch.floor(uvl[:, 2]).long()
    side = torch.tensor([_side_of(case, t) for t in range(_mips(case))], device=DEV)[mip]
    x, y = (torch.floor(uvl[:, i].double() * side).long() for i in (0, 1))
    out = _mlp(case, _rows(case, n0, n1, x, y, mip), wl, bl)
    leaves = g0 + g1 + wl + bl
    grads = torch.autograd.grad(out, leaves, dout.double(), allow_unused=True)
    return {"y": out.detach(), "grads": [torch.zeros_like(t) if r is None else r
                                         for t, r in zip(leaves, grads)]}
