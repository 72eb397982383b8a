"""The framework's timed cases: what a user's program has it do, through the
functions of paper_2608_09388_gb300.hc on device tensors.

A case is one pass of such a program over buffers that it holds: a layer on a
new batch of masks, a layer on a mapping already built, a block with its group
norm, a whole encoder, the mask-selection steps, a training step. The sizes are
those of the repository's workloads (655- and 10475-vertex meshes, spirals of 9
and 12, 16 to 128 channels, fp32 and bf16); draw() spreads over the ranges
between and around them, ragged sizes and absent neighbours among them.

Inputs are made on the GPU from the case's seed: points uniform on the unit
sphere with each vertex's nearest vertices as its spiral, clustered or
Bernoulli contact masks, N(0, 1) features, weights N(0, 1 / sqrt(L * C_in)).
Buffers are sized for every row of the batch, as the active-row count stays on
the device.
"""
from __future__ import annotations

import math

import torch

from paper_2608_09388_gb300 import hc

ACTS = {"none": hc.HC_ACT_NONE, "elu": hc.HC_ACT_ELU, "relu": hc.HC_ACT_RELU}
LAYOUTS = {"dense": hc.HC_LAYOUT_DENSE, "compact": hc.HC_LAYOUT_COMPACT}
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
EPS = 1e-5


def listed():
    return [
        # The whole sparse layer on a batch of new contact masks: compaction,
        # Eq. 4 mapping, conv with the fused scatter. The framework's headline.
        dict(name="layer_32x10475_bf16", kind="layer", dtype="bf16", B=32, V=10475, L=12,
             C_in=64, C_out=128, act="elu", mask="clustered", density=0.05, holes=0.0),
        # One frame of the small mesh in fp32: the smallest call, all latency.
        dict(name="layer_1x655_f32", kind="layer", dtype="f32", B=1, V=655, L=9, C_in=16,
             C_out=64, act="elu", mask="uniform", density=0.1, holes=0.0),
        # An inner layer of the bf16 encoder on compact rows, mapping at hand.
        dict(name="conv_64x655_bf16", kind="conv", dtype="bf16", B=64, V=655, L=9, C_in=64,
             C_out=64, act="elu", mask="uniform", density=0.1, holes=0.0, layout="compact"),
        # The large layer with half of the mesh active: throughput.
        dict(name="conv_64x10475_bf16", kind="conv", dtype="bf16", B=64, V=10475, L=9, C_in=128,
             C_out=128, act="elu", mask="uniform", density=0.5, holes=0.0, layout="dense"),
        # A block of the encoder: conv, group norm over each frame, activation.
        dict(name="conv_gn_32x10475_bf16", kind="conv_gn", dtype="bf16", B=32, V=10475, L=12,
             C_in=64, C_out=128, act="elu", mask="clustered", density=0.05, holes=0.0,
             layout="dense", G=8),
        # Group norm of a fully active large activation (larger than L2).
        dict(name="group_norm_64x10475_bf16", kind="group_norm", dtype="bf16", B=64, V=10475,
             C=128, G=8, act="elu", density=1.0),
        # The motion encoder over 4 x 64 frames: compaction, gather, four convs
        # (a ragged 45-channel input), the 64 -> 1 head, dense logits.
        dict(name="motion_256x655_bf16", kind="encoder", dtype="bf16", B=256, V=655, L=9, C_in=45,
             C_1=64, C_2=128, C_3=128, C_4=64, C_head=1, mask="uniform", density=0.15, holes=0.0),
        # The mask-score update over the encoder's outputs for ten masks.
        dict(name="mask_score_10x41920x64_bf16", kind="mask_score", dtype="bf16", K=10, N=41920,
             D=64),
        # Serving with the best 3 of 10 masks: selection, the kept masks for
        # every sample, compaction and mapping, the gather of the active rows.
        dict(name="kappa_64x655_bf16", kind="kappa", dtype="bf16", K=10, kappa=3, B=64, V=655, L=9,
             C=16, density=0.1),
        # A training step of the headline layer: mapping, forward, transposed
        # mapping, gradients of input, weight and bias.
        dict(name="train_32x10475_bf16", kind="train", dtype="bf16", B=32, V=10475, L=12, C_in=64,
             C_out=128, act="elu", mask="clustered", density=0.05, holes=0.0, layout="dense"),
        # The same for a large inner layer: the heaviest bf16 step.
        dict(name="train_64x10475_bf16", kind="train", dtype="bf16", B=64, V=10475, L=9, C_in=128,
             C_out=128, act="elu", mask="uniform", density=0.25, holes=0.0, layout="compact"),
        # Training in fp32 (no tensor-core rounding): a motion-encoder layer.
        dict(name="train_256x655_f32", kind="train", dtype="f32", B=256, V=655, L=9, C_in=64,
             C_out=128, act="elu", mask="uniform", density=0.15, holes=0.0, layout="compact"),
    ]


# ---------------------------------------------------------------- drawn cases
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _flops_limit(dtype):
    # a forward pass's multiply-adds x 2; a drawn case costs no more than the
    # heaviest listed one (fp32 work runs at a small part of the bf16 rate)
    return 5e10 if dtype == "bf16" else 3.5e9


def _draw_mesh(rng, case, train):
    """Mesh, batch, density and channels of a conv case within the limit."""
    bf = case["dtype"] == "bf16"
    while True:
        case["V"] = rng.choice([655, 10475, _log(rng, 300, 10475)])
        case["B"] = _log(rng, 1, 64 if case["V"] > 2000 else 256)
        case["L"] = rng.choice([9, 12, rng.randint(5, 16)])
        case["mask"] = rng.choice(["uniform", "clustered"])
        case["density"] = round(math.exp(rng.uniform(math.log(0.02), math.log(1.0))), 3)
        case["holes"] = rng.choice([0.0, 0.0, 0.03])
        ci = rng.choice([16, 45, 64, 128, rng.randint(3, 16) * 8])
        co = rng.choice([64, 128, rng.randint(4, 24) * 8])
        case["C_in"], case["C_out"] = ci, co
        rows = case["B"] * case["V"] * case["density"]
        if 50 <= rows and 2 * rows * case["L"] * ci * co <= _flops_limit(case["dtype"]):
            if not (train and bf and case["B"] * case["V"] * case["L"] * ci > 8e8):
                return case


def draw(rng):
    kind = rng.choice(["layer", "layer", "conv", "conv", "conv_gn", "group_norm", "encoder",
                       "mask_score", "kappa", "train", "train"])
    c = dict(kind=kind, dtype="bf16" if rng.random() < 0.7 else "f32")
    act = rng.choice(["elu", "elu", "relu", "none"])
    if kind in ("layer", "conv", "train"):
        _draw_mesh(rng, c, kind == "train")
        c["act"] = act
        if kind != "layer":
            c["layout"] = rng.choice(["dense", "compact"])
    elif kind == "conv_gn":
        _draw_mesh(rng, c, False)
        c["C_out"] = rng.choice([64, 128])
        c.update(act=act, layout=rng.choice(["dense", "compact"]), G=rng.choice([1, 4, 8, 16]))
        limit = _flops_limit(c["dtype"]) / 2
        rows = c["B"] * c["V"] * c["density"]
        if 2 * rows * c["L"] * c["C_in"] * c["C_out"] > limit:
            c["density"] = round(c["density"] * limit / (2 * rows * c["L"] * c["C_in"] *
                                                         c["C_out"]), 4)
    elif kind == "group_norm":
        c["C"], c["G"] = rng.choice([(64, 8), (128, 8), (128, 1), (256, 32), (96, 8), (64, 16),
                                     (128, 4)])
        while True:
            c["V"] = rng.choice([655, 10475, _log(rng, 300, 10475)])
            c["B"] = _log(rng, 1, 256)
            c["density"] = round(math.exp(rng.uniform(math.log(0.03), 0.0)), 3)
            rows = c["B"] * c["V"] * c["density"]
            if 200 <= rows and rows * c["C"] * (2 if c["dtype"] == "bf16" else 4) <= 1.7e8:
                break
        c["act"] = act
    elif kind == "encoder":
        c["V"] = rng.choice([655, _log(rng, 300, 3000)])
        c["B"] = max(1, min(_log(rng, 4, 256), 170000 // c["V"]))
        c.update(L=rng.choice([9, 9, 12]), C_in=rng.choice([16, 45, 64]), C_1=64,
                 C_2=rng.choice([64, 128]), C_3=rng.choice([64, 128]), C_4=64,
                 C_head=rng.choice([1, 42]), mask=rng.choice(["uniform", "clustered"]),
                 density=round(rng.uniform(0.05, 0.3), 3), holes=0.0)
        if c["dtype"] == "f32":
            c["B"] = max(1, c["B"] // 8)
    elif kind == "mask_score":
        while True:
            c["K"] = rng.randint(2, 16)
            c["D"] = rng.choice([64, 64, 128, 96, 42, 45])
            c["N"] = _log(rng, 655, 340000)
            flops = c["N"] * float(c["K"] * c["D"]) ** 2
            if flops <= (3e11 if c["dtype"] == "bf16" else 1e10):
                break
    else:
        c["K"] = rng.randint(4, 64)
        c["kappa"] = rng.randint(1, 4)
        c["V"] = rng.choice([655, 655, 10475, _log(rng, 300, 10475)])
        c["B"] = max(1, min(_log(rng, 4, 256), 600000 // (c["V"] * c["kappa"])))
        c.update(L=rng.choice([9, 12]), C=rng.choice([16, 45, 64, 128]),
                 density=round(rng.uniform(0.03, 0.3), 3))
    return c


# ---------------------------------------------------------------- inputs
def _points(g, V):
    p = torch.randn((V, 3), generator=g, device="cuda", dtype=torch.float64)
    return p / p.norm(dim=1, keepdim=True)


def _spiral(g, pts, L, holes):
    """[V, L] int32: the vertex itself, then its nearest vertices; `holes` of
    the neighbour entries are -1 (no neighbour)."""
    V = pts.shape[0]
    parts = []
    for s in range(0, V, 2048):
        dots = pts[s:s + 2048] @ pts.T
        own = torch.arange(s, s + dots.shape[0], device="cuda")
        dots[own - s, own] = 4.0
        parts.append(dots.topk(L, dim=1).indices)
    sp = torch.cat(parts).to(torch.int32)
    if holes > 0:
        drop = torch.rand(sp.shape, generator=g, device="cuda") < holes
        drop[:, 0] = False
        sp[drop] = -1
    return sp.contiguous()


def _mask(g, pts, B, V, how, density):
    """uint8 [B, V]: Bernoulli, or eight spherical patches per frame."""
    if how == "uniform":
        return (torch.rand((B, V), generator=g, device="cuda") < density).to(torch.uint8)
    cos_r = 1.0 - 2.0 * density / 8
    centres = torch.randn((B, 8, 3), generator=g, device="cuda", dtype=torch.float64)
    centres /= centres.norm(dim=2, keepdim=True)
    out = torch.empty((B, V), dtype=torch.uint8, device="cuda")
    for b in range(B):
        out[b] = ((pts @ centres[b].T).amax(dim=1) >= cos_r).to(torch.uint8)
    return out


def _normal(g, shape, dtype, scale=1.0):
    return (torch.randn(shape, generator=g, device="cuda") * scale).to(dtype)


def _weights(g, L, ci, co, dtype):
    return _normal(g, (L * ci, co), dtype, 1.0 / math.sqrt(L * ci))


def _zeros(shape, dtype):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def _tables(s, B, V, L):
    """The buffers that compaction and the mapping write."""
    s["coords"] = _zeros((B * V, 2), torch.int32)
    s["row_of"] = _zeros((B, V), torch.int32)
    s["offsets"] = _zeros((B + 1,), torch.int32)
    s["count"] = _zeros((1,), torch.int32)
    s["rulebook"] = _zeros((L, B * V), torch.int32)


def _map(s, layout):
    hc.hc_mask_compact_rulebook(s["mask"], s["spiral"], layout, s["coords"], s["row_of"],
                                s["offsets"], s["count"], s["rulebook"])


def _conv_state(g, case):
    dt = DTYPES[case["dtype"]]
    B, V, L, ci, co = (case[k] for k in ("B", "V", "L", "C_in", "C_out"))
    s = {"act": ACTS[case["act"]], "layout": LAYOUTS[case.get("layout", "dense")]}
    pts = _points(g, V)
    s["spiral"] = _spiral(g, pts, L, case["holes"])
    s["mask"] = _mask(g, pts, B, V, case["mask"], case["density"])
    # compact inputs hold the active rows in a buffer with room for all
    s["x"] = _normal(g, (B, V, ci) if s["layout"] == hc.HC_LAYOUT_DENSE else (B * V, ci), dt)
    s["W"] = _weights(g, L, ci, co, dt)
    s["bias"] = _normal(g, (co,), torch.float32, 0.1)
    _tables(s, B, V, L)
    s["y"] = _zeros((B * V, co), dt)
    return s


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 17)
    kind, dt = case["kind"], DTYPES[case["dtype"]]
    if kind in ("layer", "conv", "conv_gn", "train"):
        s = _conv_state(g, case)
        B, V, L, ci, co = (case[k] for k in ("B", "V", "L", "C_in", "C_out"))
        if kind == "layer":
            s["out"] = _zeros((B, V, co), dt)
        elif kind == "train":
            s["dy"] = _normal(g, (B * V, co), dt)
            s["row_ptr"] = _zeros((B * V + 1,), torch.int32)
            s["taps"] = _zeros((L * B * V,), torch.int32)
            s["dx"] = torch.zeros_like(s["x"])
            s["dW"] = _zeros((L * ci, co), torch.float32)
            s["dbias"] = _zeros((co,), torch.float32)
        else:
            _map(s, s["layout"])  # the mapping serves every layer on these masks
        if kind == "conv_gn":
            s["G"] = case["G"]
            s["gamma"] = 1.0 + _normal(g, (co,), torch.float32, 0.1)
            s["beta"] = _normal(g, (co,), torch.float32, 0.1)
    elif kind == "group_norm":
        B, V, C = case["B"], case["V"], case["C"]
        s = {"act": ACTS[case["act"]], "G": case["G"]}
        rows = (torch.rand((B, V), generator=g, device="cuda") < case["density"]).sum(dim=1)
        s["offsets"] = torch.cat([rows.new_zeros(1), rows.cumsum(0)]).to(torch.int32)
        s["x"] = (_normal(g, (B * V, C), torch.float32) * 1.5 + 0.3).to(dt)
        s["gamma"] = 1.0 + _normal(g, (C,), torch.float32, 0.1)
        s["beta"] = _normal(g, (C,), torch.float32, 0.1)
        s["y"] = _zeros((B * V, C), dt)
    elif kind == "encoder":
        B, V, L = case["B"], case["V"], case["L"]
        pts = _points(g, V)
        s = {"spiral": _spiral(g, pts, L, case["holes"]),
             "mask": _mask(g, pts, B, V, case["mask"], case["density"]),
             "x": _normal(g, (B, V, case["C_in"]), dt)}
        _tables(s, B, V, L)
        ch = [case[k] for k in ("C_in", "C_1", "C_2", "C_3", "C_4")]
        s["layers"] = [(_weights(g, L, a, b, dt), _normal(g, (b,), torch.float32, 0.1))
                       for a, b in zip(ch[:-1], ch[1:])]
        s["head"] = (_weights(g, 1, ch[-1], case["C_head"], dt),
                     _normal(g, (case["C_head"],), torch.float32, 0.1))
        s["rows"] = [_zeros((B * V, c), dt) for c in ch]
        s["logits"] = _zeros((B * V, case["C_head"]), dt)
        s["out"] = _zeros((B, V, case["C_head"]), dt)
    elif kind == "mask_score":
        K, N, D = case["K"], case["N"], case["D"]
        # the outputs for one input under different masks share a part
        shared = torch.randn((1, N, D), generator=g, device="cuda")
        s = {"O": (0.7 * shared + 0.7 * torch.randn((K, N, D), generator=g, device="cuda")).to(dt),
             "alpha": _normal(g, (K,), torch.float32, 0.1)}
        s["alpha_out"], s["sim"] = _zeros((K,), torch.float32), _zeros((K, K), torch.float32)
    else:  # kappa
        B, V, L, K, kap, C = (case[k] for k in ("B", "V", "L", "K", "kappa", "C"))
        pts = _points(g, V)
        s = {"B": B, "kappa": kap, "spiral": _spiral(g, pts, L, 0.0),
             "masks": _mask(g, pts, K, V, "uniform", case["density"]),
             "alpha": _normal(g, (K,), torch.float32), "x": _normal(g, (B, V, C), dt),
             "selected": _zeros((kap,), torch.int32),
             "mask": _zeros((B * kap, V), torch.uint8)}
        _tables(s, B * kap, V, L)
        s["rows"] = _zeros((B * kap * V, C), dt)
    s["kind"] = kind
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "layer":
        _map(s, s["layout"])
        hc.hc_sparse_conv_rulebook_fwd(s["x"], s["rulebook"], s["count"], s["W"], s["bias"],
                                       s["act"], s["y"], coords=s["coords"], out=s["out"])
        return {k: s[k] for k in ("coords", "row_of", "offsets", "count", "rulebook", "y", "out")}
    if kind == "conv":
        hc.hc_sparse_conv_rulebook_fwd(s["x"], s["rulebook"], s["count"], s["W"], s["bias"],
                                       s["act"], s["y"])
        return {"y": s["y"]}
    if kind == "conv_gn":
        hc.hc_sparse_conv_gn_fwd(s["x"], s["rulebook"], s["count"], s["W"], s["bias"], s["coords"],
                                 s["offsets"], s["G"], EPS, s["gamma"], s["beta"], s["act"],
                                 s["y"])
        return {"y": s["y"]}
    if kind == "group_norm":
        hc.hc_sparse_group_norm_fwd(s["x"], s["offsets"], s["G"], EPS, s["gamma"], s["beta"],
                                    s["act"], s["y"])
        return {"y": s["y"]}
    if kind == "encoder":
        _map(s, hc.HC_LAYOUT_COMPACT)
        rows = s["rows"]
        hc.hc_gather_rows(s["x"], s["coords"], s["count"], 1, rows[0])
        for i, (W, b) in enumerate(s["layers"]):
            hc.hc_sparse_conv_rulebook_fwd(rows[i], s["rulebook"], s["count"], W, b, hc.HC_ACT_ELU,
                                           rows[i + 1])
        W, b = s["head"]
        hc.hc_sparse_linear_fwd(rows[-1], s["count"], W, b, hc.HC_ACT_NONE, s["logits"])
        B, V, _ = s["out"].shape
        hc.hc_scatter_dense(s["logits"], s["coords"], s["row_of"], s["count"], B, V, True,
                            s["out"])
        return {"coords": s["coords"], "count": s["count"], "features": rows[-1],
                "logits": s["logits"], "out": s["out"]}
    if kind == "mask_score":
        hc.hc_mask_score_update(s["O"], s["alpha"], s["alpha_out"], s["sim"])
        return {"alpha": s["alpha_out"], "sim": s["sim"]}
    if kind == "kappa":
        hc.hc_mask_select_topk(s["alpha"], s["kappa"], s["selected"])
        hc.hc_kappa_masks(s["masks"], s["selected"], s["B"], s["mask"])
        _map(s, hc.HC_LAYOUT_COMPACT)
        hc.hc_gather_rows(s["x"], s["coords"], s["count"], s["kappa"], s["rows"])
        return {k: s[k] for k in ("selected", "mask", "coords", "row_of", "offsets", "count",
                                  "rulebook", "rows")}
    _map(s, s["layout"])
    hc.hc_sparse_conv_rulebook_fwd(s["x"], s["rulebook"], s["count"], s["W"], s["bias"], s["act"],
                                   s["y"])
    x_rows = s["x"].numel() // s["x"].shape[-1]
    hc.hc_conv_rulebook_transpose(s["rulebook"], s["count"], x_rows, s["row_ptr"], s["taps"])
    hc.hc_sparse_conv_rulebook_bwd(s["x"], s["rulebook"], s["count"], s["W"], s["y"], s["dy"],
                                   s["act"], s["row_ptr"], s["taps"], s["dx"], s["dW"],
                                   s["dbias"])
    return {k: s[k] for k in ("row_ptr", "taps", "y", "dx", "dW", "dbias")}


# ---------------------------------------------------------------- the work of a pass
def work(case):
    kind = case["kind"]
    eb = 2 if case["dtype"] == "bf16" else 4
    if kind == "mask_score":
        kd = case["K"] * case["D"]
        return {"bytes": case["N"] * kd * eb + 4 * (case["K"] ** 2 + 2 * case["K"]),
                "flops": float(case["N"]) * kd * (kd + 1)}
    BV = case["B"] * case["V"]
    n = BV * case["density"]
    if kind == "group_norm":
        return {"bytes": 2 * n * case["C"] * eb + 4 * case["B"], "flops": 10.0 * n * case["C"]}
    L = case["L"]
    if kind == "kappa":
        BV, n = BV * case["kappa"], n * case["kappa"]
        return {"bytes": case["kappa"] * case["V"] + BV * (1 + 4) + n * (8 + 4 * L)
                + case["V"] * L * 4 + n * case["C"] * eb * (1 + 1.0 / case["kappa"]), "flops": 0.0}
    table = BV * (1 + 4) + n * (8 + 4 * L) + case["V"] * L * 4  # mask, row_of, coords, mapping
    if kind == "encoder":
        ch = [case[k] for k in ("C_in", "C_1", "C_2", "C_3", "C_4")]
        wide = sum(a * b for a, b in zip(ch[:-1], ch[1:]))
        weights = L * wide + ch[-1] * case["C_head"]
        return {"bytes": table + n * eb * (ch[0] + ch[-1] + case["C_head"]) + weights * eb
                + BV * case["C_head"] * eb, "flops": 2.0 * n * weights}
    ci, co = case["C_in"], case["C_out"]
    flops = 2.0 * n * L * ci * co
    # the input rows that some tap reads: the active ones (a neighbour counts
    # only where it is active)
    fwd = n * eb * (ci + co) + L * ci * co * eb + co * 4
    if kind == "layer":
        return {"bytes": table + fwd + n * co * eb, "flops": flops}
    if kind == "train":
        back = n * eb * co + BV * ci * eb + (L * ci * co + co) * 4 + 4 * BV + 4 * L * n
        return {"bytes": table + fwd + back, "flops": 3.0 * flops}
    return {"bytes": n * 4 * L + fwd, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def _act64(z, act):
    if act == hc.HC_ACT_ELU:
        return torch.where(z > 0, z, torch.expm1(z))
    return z.clamp_min(0) if act == hc.HC_ACT_RELU else z


def _compact64(mask, spiral, compact):
    """Active (frame, vertex) rows in order and, per row and slot, the input
    row of its tap (-1: absent)."""
    B, V = mask.shape
    at = mask.nonzero()
    place = torch.full((B * V,), -1, dtype=torch.int64, device="cuda")
    place[at[:, 0] * V + at[:, 1]] = torch.arange(at.shape[0], device="cuda")
    nb = spiral.long()[at[:, 1]]
    row = at[:, :1] * V + nb.clamp_min(0)
    to = place[row]
    return at, torch.where((nb >= 0) & (to >= 0), to if compact else row, -1)


def _conv64(x, taps, W, bias):
    """Rows of x [., C_in] through the taps [n, L] and W [L * C_in, C_out]."""
    z = bias.double().expand(taps.shape[0], -1).clone()
    ci = x.shape[1]
    xd, Wd = x.double(), W.double()
    for l in range(taps.shape[1]):
        for r in range(0, taps.shape[0], 1 << 17):
            t = taps[r:r + (1 << 17), l]
            z[r:r + (1 << 17)] += (xd[t.clamp_min(0)] * (t >= 0)[:, None]) @ Wd[l * ci:(l + 1) * ci]
    return z


def _norm64(x, offsets, G, gamma, beta, act):
    out = torch.empty_like(x)
    off = offsets.tolist()
    for a, b in zip(off[:-1], off[1:]):
        if b > a:
            v = x[a:b].view(b - a, G, -1)
            mu = v.mean(dim=(0, 2), keepdim=True)
            var = (v - mu).square().mean(dim=(0, 2), keepdim=True)
            out[a:b] = ((v - mu) / (var + EPS).sqrt()).reshape(b - a, -1)
    return _act64(out * gamma.double() + beta.double(), act)


def _room(rows, capacity):
    """Rows as they lie in a zeroed buffer with room for `capacity`."""
    out = torch.zeros((capacity, rows.shape[1]), dtype=torch.float64, device="cuda")
    out[:rows.shape[0]] = rows
    return out


def exact(case, seed):
    s = prepare(case, seed)
    kind = s["kind"]
    if kind == "mask_score":
        O = s["O"].double()
        K = O.shape[0]
        S = torch.stack([torch.stack([(O[i].T @ O[k]).square().sum() for k in range(K)])
                         for i in range(K)])
        norm = S.diagonal().sqrt()
        sim = S / (norm[:, None] * norm[None, :])
        off = (1 - sim).sum(dim=0) - (1 - sim).diagonal()
        alpha = s["alpha"].double()
        return {"alpha": alpha + off / (K - 1) if K > 1 else alpha, "sim": sim}
    if kind == "group_norm":
        n = int(s["offsets"][-1])
        y = _norm64(s["x"][:n].double(), s["offsets"], s["G"], s["gamma"], s["beta"], s["act"])
        return {"y": _room(y, s["x"].shape[0])}
    if kind == "kappa":
        kept = s["alpha"].topk(s["kappa"]).indices
        at = s["masks"][kept].repeat(s["B"], 1).nonzero()
        rows = s["x"][at[:, 0] // s["kappa"], at[:, 1]].double()
        return {k: None for k in ("selected", "mask", "coords", "row_of", "offsets", "count",
                                  "rulebook")} | {"rows": _room(rows, s["rows"].shape[0])}
    B, V = s["mask"].shape
    if kind == "encoder":
        at, taps = _compact64(s["mask"], s["spiral"], True)
        h = s["x"][at[:, 0], at[:, 1]].double()
        for W, b in s["layers"]:
            h = _act64(_conv64(h, taps, W, b), hc.HC_ACT_ELU)
        logits = h @ s["head"][0].double() + s["head"][1].double()
        out = torch.zeros((B, V, logits.shape[1]), dtype=torch.float64, device="cuda")
        out[at[:, 0], at[:, 1]] = logits
        return {"coords": None, "count": None, "features": _room(h, B * V),
                "logits": _room(logits, B * V), "out": out}
    at, taps = _compact64(s["mask"], s["spiral"], s["layout"] == hc.HC_LAYOUT_COMPACT)
    n = at.shape[0]
    x = s["x"].view(-1, s["x"].shape[-1])
    z = _conv64(x, taps, s["W"], s["bias"])
    if kind == "conv_gn":
        y = _norm64(z, s["offsets"], s["G"], s["gamma"], s["beta"], s["act"])
        return {"y": _room(y, B * V)}
    y = _act64(z, s["act"])
    if kind == "conv":
        return {"y": _room(y, B * V)}
    if kind == "layer":
        out = torch.zeros((B, V, y.shape[1]), dtype=torch.float64, device="cuda")
        out[at[:, 0], at[:, 1]] = y
        return {k: None for k in ("coords", "row_of", "offsets", "count", "rulebook")} | {
            "y": _room(y, B * V), "out": out}
    dz = s["dy"][:n].double()
    if s["act"] == hc.HC_ACT_ELU:
        dz = dz * torch.where(y > 0, 1.0, y + 1.0)
    elif s["act"] == hc.HC_ACT_RELU:
        dz = dz * (y > 0)
    ci = x.shape[1]
    xd, Wd = x.double(), s["W"].double()
    dx = torch.zeros_like(xd)
    dW = torch.zeros_like(Wd)
    for l in range(taps.shape[1]):
        for r in range(0, n, 1 << 17):
            t, d = taps[r:r + (1 << 17), l], dz[r:r + (1 << 17)]
            on = t >= 0
            dW[l * ci:(l + 1) * ci] += (xd[t.clamp_min(0)] * on[:, None]).T @ d
            dx.index_add_(0, t[on], (d @ Wd[l * ci:(l + 1) * ci].T)[on])
    return {"row_ptr": None, "taps": None, "y": _room(y, B * V), "dx": dx.view(s["x"].shape),
            "dW": dW, "dbias": dz.sum(dim=0)}
