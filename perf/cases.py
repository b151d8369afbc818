"""The work that programs have this library do, as cases that can be timed.

Every case is one call of a public entry point, over the range of sizes that
the repository's own configurations span: from the small latent (4 levels x 24
latitudes x 48 longitudes, width 128, the serving and ensemble size) to the
full-size one (9 x 90 x 180, width 768, the 2-degree latent of the 0.25-degree
grid) and the encoder / decoder around it (720 x 1440 fields, width 1024), in
the three precisions (FP32, BF16, BF16 with the FP8 MLP).

``listed`` names the cases, ``draw`` gives further ones of the same ranges,
``prepare`` makes inputs, weights and handles, ``run`` makes the call,
``work`` counts what the call cannot do without and ``exact`` computes its
result in float64 with plain torch.
"""
import math

import numpy as np
import torch

import paper_2503_22235_gb300 as wm

PRECISION = {"fp32": wm.WM_PREC_FP32, "bf16": wm.WM_PREC_BF16, "fp8": wm.WM_PREC_BF16_FP8MLP}
EPS = 1e-5

SMALL = {"D": 4, "H": 24, "W": 48, "C": 128, "heads": 4, "kd": 3, "kh": 5, "kw": 5, "periodic": True}
FULL = {"D": 9, "H": 90, "W": 180, "C": 768, "heads": 16, "kd": 5, "kh": 7, "kw": 7, "periodic": True}
# a regional latent: odd sizes, clamped longitude, half the full width
REGION = {"D": 5, "H": 45, "W": 91, "C": 384, "heads": 8, "kd": 3, "kh": 7, "kw": 7, "periodic": False}
# the 0.25-degree grid: 28 levels padded to 32, 4 levels x 8 x 8 pixels per token
FIELDS = {"H0": 720, "W0": 1440, "levels": 28, "level_pad": 32, "pd": 4, "p": 8, "v_atm": 5, "v_sfc_in": 8,
          "v_sfc_out": 17, "n_const": 8, "Ce": 1024, "heads": 16, "kd": 5, "kh": 7, "kw": 7, "blocks": 2,
          "C": 768, "periodic": True}


def listed():
    return [
        # one linear layer of the small latent: the smallest call, launch latency counts
        {"name": "linear_small_bf16", "kind": "linear", "precision": "bf16", "M": 4608, "N": 128, "K": 128,
         "epilogue": 0},
        # the MLP's first layer of the full-size latent, with its GELU
        {"name": "linear_full_bf16", "kind": "linear", "precision": "bf16", "M": 145800, "N": 3072, "K": 768,
         "epilogue": 1},
        # the same layer of the regional latent in the plain FP32 path: a ragged row count
        {"name": "linear_region_fp32", "kind": "linear", "precision": "fp32", "M": 20475, "N": 1536, "K": 384,
         "epilogue": 1},
        # neighborhood attention of the full-size latent: the kernel a forecast spends most time in
        {"name": "attention_full_bf16", "kind": "attention", "precision": "bf16", "batch": 1, **FULL},
        # FP32 attention of the regional latent: odd sizes, clamped longitude, two members
        {"name": "attention_region_fp32", "kind": "attention", "precision": "fp32", "batch": 2, **REGION},
        # one transformer block of the full-size latent in each precision
        {"name": "block_full_bf16", "kind": "block", "precision": "bf16", "batch": 1, "rope": False, **FULL},
        {"name": "block_full_fp8", "kind": "block", "precision": "fp8", "batch": 1, "rope": False, **FULL},
        {"name": "block_full_fp32", "kind": "block", "precision": "fp32", "batch": 1, "rope": False, **FULL},
        # a six-hour step of one small latent (8 blocks): what a serving tick runs
        {"name": "step_small_bf16", "kind": "step", "precision": "bf16", "batch": 1, "which": 0, "rope": False,
         "blocks_p6": 8, "blocks_p1": 4, **SMALL},
        # eight requests with uneven lead times advanced together to their own lead
        {"name": "rollout_small_bf16", "kind": "rollout", "precision": "bf16", "batch": 8, "max_lead": 48,
         "rope": False, "blocks_p6": 8, "blocks_p1": 4, **SMALL},
        # 0.25-degree fields to the full-size latent, and back
        {"name": "encode_full_bf16", "kind": "encode", "precision": "bf16", **FIELDS},
        {"name": "decode_full_bf16", "kind": "decode", "precision": "bf16", **FIELDS},
    ]


# The cost of the largest listed case (the full-size block in FP32) bounds what draw gives, by precision: the plain
# path runs on CUDA cores.
_RATE = {"fp32": 1.0, "bf16": 0.04, "fp8": 0.04}


def _cost(case):
    return work(case)["flops"] * _RATE[case["precision"]] + work(case)["bytes"] * 8.0


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_latent(rng, precision, batches):
    """A latent between the small and the full-size one: any grid, the widths and head sizes all paths take."""
    narrow = rng.random() < 0.4
    if narrow:   # the serving width
        c = {"C": 128, "heads": 4, "D": rng.randint(2, 8), "H": 8 * rng.randint(2, 6), "W": 16 * rng.randint(2, 8)}
        if rng.random() < 0.3:   # grids that no patch size divides
            c["H"] += rng.randint(1, 7)
            c["W"] += rng.randint(1, 15)
        k = rng.choice([3, 5])
        c.update(kd=rng.choice([1, 3]) if c["D"] >= 3 else 1, kh=k, kw=k, periodic=rng.random() < 0.8)
    else:
        C, heads = rng.choice([(256, 8), (256, 4), (384, 8), (512, 8), (768, 16), (768, 12), (1024, 16)])
        H = _log_int(rng, 16, 90)
        c = {"C": C, "heads": heads, "D": rng.randint(3, 13), "H": H, "W": min(180, 2 * H + rng.randint(-9, 9))}
        k = rng.choice([5, 7])
        c.update(kd=rng.choice([3, 5]) if c["D"] >= 5 else 3, kh=k, kw=k, periodic=rng.random() < 0.7)
    return {**c, "batch": rng.choice(batches)}


def _draw(rng):
    kind = rng.choice(["linear", "linear", "layernorm", "attention", "attention", "block", "block", "step", "rollout",
                       "hourly", "encode", "decode"])
    precision = rng.choice(["fp32", "bf16", "bf16"])
    if kind == "linear":
        C = rng.choice([128, 256, 384, 512, 768, 1024])
        n, k = rng.choice([(3, 1), (1, 1), (4, 1), (1, 4)])
        return {"kind": kind, "precision": precision, "M": _log_int(rng, 1024, 145800), "N": n * C, "K": k * C,
                "epilogue": rng.choice([0, 1, 3])}
    if kind == "layernorm":
        return {"kind": kind, "precision": precision, "M": _log_int(rng, 2048, 145800),
                "C": rng.choice([128, 256, 384, 512, 768, 1024])}
    if kind == "attention":
        return {"kind": kind, "precision": precision, **_draw_latent(rng, precision, [1, 1, 2, 4])}
    if kind in ("encode", "decode"):
        Ce, heads = rng.choice([(128, 4), (512, 8), (1024, 16)])
        k = rng.choice([5, 7])
        p = rng.choice([4, 8])
        return {"kind": kind, "precision": precision, **FIELDS, "H0": p * rng.randint(16, 90),
                "W0": p * rng.randint(32, 180), "p": p, "Ce": Ce, "heads": heads, "kh": k, "kw": k,
                "levels": rng.choice([13, 28, 30]), "C": rng.choice([128, 384, 768]),
                "periodic": rng.random() < 0.7}
    precision = rng.choice(["fp32", "bf16", "bf16", "fp8"])
    c = {"kind": kind, "precision": precision, "rope": rng.random() < 0.2,
         **_draw_latent(rng, precision, [1, 1, 2, 4, 7] if kind != "hourly" else [1])}
    if kind == "block":
        return c
    c.update(blocks_p6=rng.choice([1, 2, 8]) if c["C"] == 128 else 1, blocks_p1=rng.choice([1, 4]) if c["C"] == 128 else 1)
    if kind == "step":
        c["which"] = rng.randint(0, 1)
    elif kind == "rollout":
        c["max_lead"] = rng.randint(6, 48)
    else:
        c["max_lead"] = rng.randint(5, 20)
    return c


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= top:
            return case


# ------------------------------------------------------------------- inputs ---

def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + tag) % (1 << 62))
    return g


def _normal(shape, seed, tag):
    return torch.randn(shape, generator=_gen(seed, tag), device="cuda")


def _uniform(shape, bound, seed, tag):
    return (torch.rand(shape, generator=_gen(seed, tag), device="cuda") * 2 - 1) * bound


def _matrix(n, k, seed, tag):
    """Xavier-uniform [n, k]."""
    return _uniform((n, k), math.sqrt(6.0 / (n + k)), seed, tag)


def _block_weights(C, seed, tag):
    """One block's float32 tensors in the weight file's order: Xavier matrices, small biases, affine near one."""
    sizes = [("ln1_g", C, 0), ("ln1_b", C, 0), ("wqkv", 3 * C, C), ("bqkv", 3 * C, 0), ("wo", C, C), ("bo", C, 0),
             ("ln2_g", C, 0), ("ln2_b", C, 0), ("w1", 4 * C, C), ("b1", 4 * C, 0), ("w2", C, 4 * C), ("b2", C, 0)]
    w = {}
    for i, (name, n, k) in enumerate(sizes):
        w[name] = _matrix(n, k, seed, tag + i) if k else _uniform((n,), 0.1, seed, tag + i)
        if name.endswith("_g"):
            w[name] += 1.0
    return w


def _blocks(C, n, seed, tag):
    return [_block_weights(C, seed, tag + 100 * i) for i in range(n)]


def _pack(tensors):
    return torch.cat([t.reshape(-1) for t in tensors]).cpu().numpy()


def _leads(case, seed):
    """Lead times in hours, from 1 to the longest, uneven as requests are; the longest is always among them."""
    r = np.random.RandomState(int(seed) % (1 << 31))
    leads = r.randint(1, case["max_lead"] + 1, size=case["batch"])
    leads[r.randint(case["batch"])] = case["max_lead"]
    return [int(t) for t in leads]


def _processor(case):
    """(blocks of the six-hour, of the one-hour processor)"""
    return case.get("blocks_p6", 1), case.get("blocks_p1", 1)


def _latent(case, batch, seed):
    return _normal((batch, case["D"], case["H"], case["W"], case["C"]), seed, 1)


def _codec_tensors(case, seed):
    """The encoder's and decoder's own tensors in blob order, then their blocks."""
    k_atm = case["pd"] * case["p"] ** 2 * case["v_atm"]
    k_sfc = case["p"] ** 2 * (case["v_sfc_in"] + case["n_const"])
    n_sfc = case["p"] ** 2 * case["v_sfc_out"]
    Ce, C = case["Ce"], case["C"]
    sizes = [("embed_atm", Ce, k_atm), ("embed_sfc", Ce, k_sfc), ("enc_out", C, Ce), ("dec_in", Ce, C),
             ("unembed_atm", k_atm, Ce), ("unembed_sfc", n_sfc, Ce)]
    w = {}
    for i, (name, n, k) in enumerate(sizes):
        w[name + "_w"] = _matrix(n, k, seed, 1000 + 2 * i)
        w[name + "_b"] = _uniform((n,), 0.1, seed, 1001 + 2 * i)
    return w, _blocks(Ce, case["blocks"], seed, 2000), _blocks(Ce, case["blocks"], seed, 20000)


def _codec_grid(case):
    """(levels, latitudes, longitudes) of the latent."""
    return case["level_pad"] // case["pd"] + 1, case["H0"] // case["p"], case["W0"] // case["p"]


def _fields(case, seed):
    H0, W0 = case["H0"], case["W0"]
    return (_normal((case["levels"], H0, W0, case["v_atm"]), seed, 2), _normal((H0, W0, case["v_sfc_in"]), seed, 3),
            _normal((H0, W0, case["n_const"]), seed, 4))


def _linear_inputs(case, seed):
    A = _normal((case["M"], case["K"]), seed, 5)
    W = _matrix(case["N"], case["K"], seed, 6)
    b = _uniform((case["N"],), 0.1, seed, 7)
    if case["precision"] == "bf16":
        A, W = A.bfloat16(), W.bfloat16()
    return A, W, b


def _qkv(case, seed):
    """q, k and v of the size that the projection gives them: about unit variance."""
    x = _normal((case["batch"], case["D"], case["H"], case["W"], 3 * case["C"]), seed, 8)
    return x.bfloat16() if case["precision"] == "bf16" else x


class Handle:
    """A context or codec that is destroyed with the state that holds it."""

    def __init__(self, value, destroy):
        self.value, self.destroy = value, destroy

    def __del__(self):
        self.destroy(self.value)


def _context(case, seed, batch):
    n6, n1 = _processor(case)
    blocks = _blocks(case["C"], n6, seed, 10000) + _blocks(case["C"], n1, seed, 50000)
    cfg = wm.wm_config(case["D"], case["H"], case["W"], case["C"], case["heads"], case["kd"], case["kh"], case["kw"],
                       n6, n1, int(case["periodic"]), EPS, PRECISION[case["precision"]], batch, int(case["rope"]))
    return Handle(wm.wm_create_from_host(cfg, _pack([t for b in blocks for t in b.values()])), wm.wm_destroy)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "linear":
        s["A"], s["W"], s["bias"] = _linear_inputs(case, seed)
        wide = case["precision"] == "fp32" or case["epilogue"] == 3
        s["out"] = torch.empty(case["M"], case["N"], device="cuda", dtype=torch.float32 if wide else torch.bfloat16)
    elif kind == "layernorm":
        s["x"] = _normal((case["M"], case["C"]), seed, 9)
        s["gamma"], s["beta"] = 1 + _uniform((case["C"],), 0.1, seed, 10), _uniform((case["C"],), 0.1, seed, 11)
        s["out"] = torch.empty_like(s["x"], dtype=torch.float32 if case["precision"] == "fp32" else torch.bfloat16)
    elif kind == "attention":
        s["qkv"] = _qkv(case, seed)
        s["out"] = torch.empty((*s["qkv"].shape[:-1], case["C"]), device="cuda", dtype=s["qkv"].dtype)
    elif kind in ("encode", "decode"):
        w, enc, dec = _codec_tensors(case, seed)
        cfg = wm.wm_codec_config(case["H0"], case["W0"], case["levels"], case["level_pad"], case["pd"], case["p"],
                                 case["v_atm"], case["v_sfc_in"], case["v_sfc_out"], case["n_const"], case["Ce"],
                                 case["heads"], case["kd"], case["kh"], case["kw"], case["blocks"], case["C"],
                                 int(case["periodic"]), EPS, PRECISION[case["precision"]])
        blob = _pack([*w.values(), *(t for b in enc + dec for t in b.values())])
        s["codec"] = Handle(wm.wm_codec_create(cfg, blob), wm.wm_codec_destroy)
        if kind == "encode":
            s["fields"] = _fields(case, seed)
            s["latent"] = torch.empty(*_codec_grid(case), case["C"], device="cuda")
        else:
            s["latent"] = _normal((*_codec_grid(case), case["C"]), seed, 12)
            s["atm"] = torch.empty(case["levels"], case["H0"], case["W0"], case["v_atm"], device="cuda")
            s["sfc"] = torch.empty(case["H0"], case["W0"], case["v_sfc_out"], device="cuda")
    else:
        batch = case["batch"]
        s["ctx"] = _context(case, seed, batch)
        s["latent"] = _latent(case, batch, seed)
        if kind == "rollout":
            s["leads"] = _leads(case, seed)
            s["latents"] = list(s["latent"].unbind(0))
        elif kind == "hourly":
            s["out"] = torch.empty((case["max_lead"] + 1, *s["latent"].shape[1:]), device="cuda")
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------- run ---

def run(s):
    """One call. Blocks, steps and rollouts advance the state's latent in place, as a forecast does."""
    case = s["case"]
    kind = case["kind"]
    if kind == "linear":
        wm.wm_op_linear(s["A"], s["W"], s["bias"], s["out"], PRECISION[case["precision"]], case["epilogue"])
        return s["out"]
    if kind == "layernorm":
        wm.wm_op_layernorm(s["x"], s["gamma"], s["beta"], s["out"], EPS)
        return s["out"]
    if kind == "attention":
        wm.wm_op_neighborhood_attention(s["qkv"], s["out"], case["batch"], case["D"], case["H"], case["W"], case["C"],
                                        case["heads"], case["kd"], case["kh"], case["kw"], case["periodic"],
                                        PRECISION[case["precision"]])
        return s["out"]
    if kind == "block":
        wm.wm_block_forward(s["ctx"].value, s["latent"], wm.WM_P6, 0)
        return s["latent"]
    if kind == "step":
        wm.wm_processor_step(s["ctx"].value, s["latent"], case["which"])
        return s["latent"]
    if kind == "rollout":
        wm.wm_rollout_batch(s["ctx"].value, s["latents"], s["leads"])
        return s["latent"]
    if kind == "hourly":
        wm.wm_rollout_hourly(s["ctx"].value, s["latent"], case["max_lead"], s["out"])
        return s["out"]
    if kind == "encode":
        wm.wm_encode(s["codec"].value, *s["fields"], s["latent"])
        return s["latent"]
    wm.wm_decode(s["codec"].value, s["latent"], s["atm"], s["sfc"])
    return s["atm"], s["sfc"]


# --------------------------------------------------------------------- work ---

def _block_work(tokens, C, window, precision):
    """One block: latent in and out, weights once; 24 C^2 + 4 window C operations a token."""
    per = {"fp32": 4, "bf16": 2, "fp8": 2}[precision]
    mats = 12 * C * C * per if precision != "fp8" else 4 * C * C * 2 + 8 * C * C
    return {"bytes": 8 * tokens * C + mats + 13 * C * 4, "flops": tokens * (24 * C * C + 4 * window * C)}


def work(case):
    kind = case["kind"]
    el = 4 if case["precision"] == "fp32" else 2
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        out = 4 if case["precision"] == "fp32" or case["epilogue"] == 3 else 2
        return {"bytes": el * (M * K + N * K) + 4 * N + out * M * N, "flops": 2 * M * N * K}
    if kind == "layernorm":
        return {"bytes": case["M"] * case["C"] * (4 + el) + 8 * case["C"], "flops": 8 * case["M"] * case["C"]}
    window = case["kd"] * case["kh"] * case["kw"]
    if kind in ("encode", "decode"):
        D, H, W = _codec_grid(case)
        n = D * H * W
        b = _block_work(n, case["Ce"], window, case["precision"])
        pix = case["H0"] * case["W0"]
        sfc = case["v_sfc_in"] + case["n_const"] if kind == "encode" else case["v_sfc_out"]
        fields = 4 * pix * (case["levels"] * case["v_atm"] + sfc)
        k_atm, k_sfc = case["pd"] * case["p"] ** 2 * case["v_atm"], case["p"] ** 2 * sfc
        mats = el * case["Ce"] * (k_atm + k_sfc + case["C"])
        maps = 2 * case["Ce"] * H * W * ((D - 1) * k_atm + k_sfc) + 2 * n * case["Ce"] * case["C"]
        weights = case["blocks"] * (b["bytes"] - 8 * n * case["Ce"])
        return {"bytes": fields + 4 * n * case["C"] + mats + weights, "flops": case["blocks"] * b["flops"] + maps}
    tokens, C = case["D"] * case["H"] * case["W"], case["C"]
    if kind == "attention":
        return {"bytes": el * 4 * case["batch"] * tokens * C, "flops": 4 * window * case["batch"] * tokens * C}
    n6, n1 = _processor(case)
    one = _block_work(tokens, C, window, case["precision"])
    weights = one["bytes"] - 8 * tokens * C
    latents, blocks, mats = case["batch"], case["batch"], 1
    if kind == "step":
        mats = n6 if case["which"] == 0 else n1
        blocks *= mats
    elif kind == "rollout":   # lead times are drawn evenly from 1 to the longest
        mats = n6 + n1
        blocks = case["batch"] * (n6 * case["max_lead"] / 12 + n1 * 2.5)
    elif kind == "hourly":    # a chain of six-hour steps, one one-hour step for every other hour
        anchors = case["max_lead"] // 6
        mats = n6 + n1
        blocks = n6 * anchors + n1 * (case["max_lead"] - anchors)
        latents = (case["max_lead"] + 2) / 2
    return {"bytes": 8 * tokens * C * latents + weights * mats, "flops": blocks * one["flops"]}


# -------------------------------------------------------------------- exact ---

def _starts(n, k):
    """First key of every query's window: the full window, moved inside at the edges."""
    return [min(max(i - k // 2, 0), n - k) for i in range(n)]


def _attention64(q, k, v, case):
    """[B, D, H, W, C] float64 each; windows clamped in level and latitude, periodic or clamped in longitude."""
    B, D, H, W, C = q.shape
    h = case["heads"]
    dh, kd, kh, kw = C // h, case["kd"], case["kh"], case["kw"]
    if case["periodic"]:
        cols = [[(j - kw // 2 + e) % W for e in range(kw)] for j in range(W)]
    else:
        cols = [[s + e for e in range(kw)] for s in _starts(W, kw)]
    cols = torch.tensor(cols, device=q.device)
    out = torch.empty_like(q)
    for d, d0 in enumerate(_starts(D, kd)):
        for i, i0 in enumerate(_starts(H, kh)):
            def window(t):   # [B, W, heads, keys, dh]
                rows = t[:, d0:d0 + kd, i0:i0 + kh].reshape(B, kd * kh, W, h, dh)[:, :, cols]
                return rows.permute(0, 2, 4, 1, 3, 5).reshape(B, W, h, kd * kh * kw, dh)
            s = torch.matmul(window(k), q[:, d, i].reshape(B, W, h, dh, 1)) / math.sqrt(dh)
            p = torch.softmax(s, dim=3)
            out[:, d, i] = (window(v) * p).sum(3).reshape(B, W, C)
    return out


def _norm64(x, g, b):
    mean = x.mean(-1, keepdim=True)
    var = ((x - mean) ** 2).mean(-1, keepdim=True)
    return (x - mean) / torch.sqrt(var + EPS) * g + b


def _linear64(x, w, b):
    return torch.nn.functional.linear(x, w, b)


def _gelu64(x):
    return 0.5 * x * (1 + torch.erf(x / math.sqrt(2.0)))


def _rope64(x, case):
    """Rotates the pairs of every head of x [B, D, H, W, C] by their level, latitude and longitude angles."""
    B, D, H, W, C = x.shape
    P = C // case["heads"] // 2
    n_lon = (P + 2) // 3
    n_lat = (P - n_lon + 1) // 2
    n_lev = P - n_lon - n_lat
    angles = torch.zeros(D, H, W, P, dtype=torch.float64, device=x.device)
    for n, off, size, dim in ((n_lev, 0, D, 0), (n_lat, n_lev, H, 1), (n_lon, n_lev + n_lat, W, 2)):
        m = torch.arange(n, dtype=torch.float64, device=x.device)
        w = 10000.0 ** (-m / max(n, 1)) if dim < 2 else 2 * math.pi * (m + 1) / W
        pos = torch.arange(size, dtype=torch.float64, device=x.device).reshape([-1 if a == dim else 1 for a in range(3)])
        angles[..., off:off + n] = pos[..., None] * w
    c, s = torch.cos(angles)[:, :, :, None], torch.sin(angles)[:, :, :, None]
    x = x.reshape(B, D, H, W, case["heads"], P, 2)
    a, b = x[..., 0], x[..., 1]
    return torch.stack([a * c - b * s, a * s + b * c], -1).reshape(B, D, H, W, C)


def _block64(x, w, case):
    C = x.shape[-1]
    qkv = _linear64(_norm64(x, w["ln1_g"], w["ln1_b"]), w["wqkv"], w["bqkv"])
    q, k, v = qkv[..., :C], qkv[..., C:2 * C], qkv[..., 2 * C:]
    if case.get("rope"):
        q, k = _rope64(q, case), _rope64(k, case)
    x = x + _linear64(_attention64(q, k, v, case), w["wo"], w["bo"])
    return x + _linear64(_gelu64(_linear64(_norm64(x, w["ln2_g"], w["ln2_b"]), w["w1"], w["b1"])), w["w2"], w["b2"])


def _double(blocks):
    return [{k: t.double() for k, t in b.items()} for b in blocks]


def exact(case, seed):
    kind = case["kind"]
    if kind == "linear":
        A, W, b = (t.double() for t in _linear_inputs(case, seed))
        out = _linear64(A, W, b)
        return _gelu64(out) if case["epilogue"] == 1 else out
    if kind == "layernorm":
        s = prepare(case, seed)
        return _norm64(s["x"].double(), s["gamma"].double(), s["beta"].double())
    if kind == "attention":
        return _attention64(*_qkv(case, seed).double().chunk(3, -1), case)
    if kind in ("encode", "decode"):
        w, enc, dec = _codec_tensors(case, seed)
        w = {k: t.double() for k, t in w.items()}
        D, H, W = _codec_grid(case)
        pd, p, top = case["pd"], case["p"], case["level_pad"] - case["levels"]
        if kind == "encode":
            atm, sfc, consts = (t.double() for t in _fields(case, seed))
            atm = torch.cat([torch.zeros(top, *atm.shape[1:], dtype=atm.dtype, device=atm.device), atm])
            atm = atm.reshape(D - 1, pd, H, p, W, p, -1).permute(0, 2, 4, 1, 3, 5, 6).reshape(D - 1, H, W, -1)
            sfc = torch.cat([sfc, consts], -1).reshape(1, H, p, W, p, -1).permute(0, 1, 3, 2, 4, 5)
            x = torch.cat([_linear64(atm, w["embed_atm_w"], w["embed_atm_b"]),
                           _linear64(sfc.reshape(1, H, W, -1), w["embed_sfc_w"], w["embed_sfc_b"])])[None]
            for b in _double(enc):
                x = _block64(x, b, case)
            return _linear64(x[0], w["enc_out_w"], w["enc_out_b"])
        x = _linear64(_normal((D, H, W, case["C"]), seed, 12).double(), w["dec_in_w"], w["dec_in_b"])[None]
        for b in _double(dec):
            x = _block64(x, b, case)
        atm = _linear64(x[0, :-1], w["unembed_atm_w"], w["unembed_atm_b"])
        atm = atm.reshape(D - 1, H, W, pd, p, p, -1).permute(0, 3, 1, 4, 2, 5, 6)
        sfc = _linear64(x[0, -1], w["unembed_sfc_w"], w["unembed_sfc_b"]).reshape(H, W, p, p, -1).permute(0, 2, 1, 3, 4)
        return (atm.reshape((D - 1) * pd, case["H0"], case["W0"], -1)[top:].contiguous(),
                sfc.reshape(case["H0"], case["W0"], -1).contiguous())
    n6, n1 = _processor(case)
    p6, p1 = _double(_blocks(case["C"], n6, seed, 10000)), _double(_blocks(case["C"], n1, seed, 50000))

    def step(x, blocks):
        for b in blocks:
            x = _block64(x, b, case)
        return x

    x = _latent(case, case["batch"], seed).double()
    if kind == "block":
        return _block64(x, p6[0], case)
    if kind == "step":
        return step(x, p1 if case["which"] else p6)
    if kind == "rollout":
        leads = torch.tensor(_leads(case, seed), device=x.device)
        for k in range(case["max_lead"] // 6 + 5):
            due6, due1 = k < leads // 6, (k >= leads // 6) & (k < leads // 6 + leads % 6)
            for due, blocks in ((due6, p6), (due1, p1)):
                if bool(due.any()):
                    x[due] = step(x[due], blocks)
        return x
    out = [x]   # hourly: six-hour anchors, one-hour branches from each
    for t in range(1, case["max_lead"] + 1):
        out.append(step(out[t - 6], p6) if t % 6 == 0 else step(out[t - 1], p1))
    return torch.cat(out)
