"""Performance cases of the cached denoising path.

Each case is one call that a program using this package makes: a whole cached
sampling run (``FeatFix.sample``), one exact block on a caller's state
(``featfix_debug_block``), or one layer on caller buffers (``featfix_op_*``).
``listed()`` holds the sizes of the package's own workloads, ``draw()`` gives
others of the same ranges, ``exact()`` restates each call in plain float64
torch.  Kinds:

  sample     x_T from a seed, then every denoising step (refreshes, drafts,
             paid checks, sampler updates): what a generation service calls.
  block      the exact block of Eq. 1 on a given state, conditioning and
             modulation included: what refresh steps and paid checks run.
  attention  softmax(q k^T / sqrt(d)) v over the joint [text ; image] rows.
  gemm       a dense layer with its epilogue: bias (qkv), bias + GELU (fc1),
             bias + gate + residual (out-projection), the same with the
             history increment (fc2 of a refresh step).
  draft      the Taylor draft of a block over its refresh history.
  verify     the paid check of a site: draft, discrepancy sums and, in the
             Verify arm, the draft written over the state.
  ln         the adaLN LayerNorm-modulation in front of a dense layer.

bf16 is the mode that models are served in, f32 the mode for small models and
for checking a bf16 run.
"""

import math

import numpy as np
import torch

from paper_2607_27842_gb300 import featfix as ff, synthetic as syn

DEV = "cuda"
TD = {"f32": torch.float32, "bf16": torch.bfloat16}
EPILOGUES = ("bias", "gelu", "gated", "gated_history")


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------

def listed():
    return [
        # The smallest whole call: the 4-block fp32 class-conditional DiT, 10
        # Euler steps with refreshes at 0/3/6/9 and two sites; a chain of
        # small launches, where latency counts.
        dict(name="sample tiny f32", kind="sample", dtype="f32", blocks=4, hidden=128, heads=4, mlp=512, grid=8,
             patch=1, in_ch=4, out_ch=4, classes=10, batch=1, cfg=False, sampler="euler", steps=10, order=1, every=3,
             sites=2),
        # A whole class-conditional image batch: DiT-XL/2 shape, 8 samples with
        # guidance, 50 DDIM steps, order-2 drafts, refresh every 5, 8 sites.
        dict(name="sample DiT-XL/2 bf16", kind="sample", dtype="bf16", blocks=28, hidden=1152, heads=16, mlp=4608,
             grid=16, patch=2, in_ch=4, out_ch=8, classes=1000, batch=8, cfg=True, sampler="ddim", steps=50, order=2,
             every=5, sites=8),
        # The two-stream block of the video model at its full token count (9 x
        # 30 x 53 video + 256 text tokens, 3-D rotary): the largest layer.
        dict(name="block video dual bf16", kind="block", dtype="bf16", block="dual", hidden=2048, heads=16, mlp=8192,
             txt=256, frames=9, rows=30, cols=53, batch=1),
        # The single-stream block of the rectified-flow image model, 1024^2
        # image (4096 image + 512 text tokens, 2-D rotary).
        dict(name="block image single bf16", kind="block", dtype="bf16", block="single", hidden=3072, heads=24,
             mlp=12288, txt=512, frames=0, rows=64, cols=64, batch=1),
        # The DiT-XL/2 block in fp32 for one guided sample (2 x 256 tokens):
        # what a check of the bf16 run against fp32 evaluates block by block.
        dict(name="block DiT-XL/2 f32", kind="block", dtype="f32", block="dit", hidden=1152, heads=16, mlp=4608,
             txt=0, frames=0, rows=16, cols=16, batch=2),
        # Attention of the guided image pair at 512^2 (1024 image + 256 text
        # tokens, 24 heads): an ordinary sequence, between the 256-token and
        # the video one.
        dict(name="attention 2x1280 d128 bf16", kind="attention", dtype="bf16", batch=2, txt=256, img=1024, heads=24,
             dim=128),
        # Attention of a DiT-XL/2 step: many short sequences, head width 72.
        dict(name="attention 16x256 d72 bf16", kind="attention", dtype="bf16", batch=16, txt=0, img=256, heads=16,
             dim=72),
        # fc2 of a DiT-XL/2 refresh step: gate, residual and history increment.
        dict(name="gemm 4096x1152x4608 bf16", kind="gemm", dtype="bf16", m=4096, n=1152, k=4608, rpb=256,
             epilogue="gated_history"),
        # fc1 of the video model's image stream: 14310 rows, GELU.
        dict(name="gemm 14310x8192x2048 bf16", kind="gemm", dtype="bf16", m=14310, n=8192, k=2048, rpb=14310,
             epilogue="gelu"),
        # The draft of a DiT-XL/2 block, order 2 (three history terms).
        dict(name="draft 4.7M 3 terms bf16", kind="draft", dtype="bf16", rows=4096, width=1152, terms=3),
        # The paid check of a video block, order 1 (two history terms),
        # FeatFix arm: the sums only.
        dict(name="verify 29.8M 2 terms bf16", kind="verify", dtype="bf16", rows=14566, width=2048, terms=2,
             write=False),
        # The LayerNorm-modulation of the video model's image stream.
        dict(name="ln 14310x2048 bf16", kind="ln", dtype="bf16", rows=14310, width=2048, rpb=14310),
    ]


def _log_int(rng, lo, hi, step=1):
    """An integer spread over the logarithm of [lo, hi], a multiple of step."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step, int(round(v / step)) * step)


def draw(rng):
    kind = rng.choice(["attention", "attention", "gemm", "gemm", "gemm", "block", "block", "sample", "draft", "verify",
                       "ln"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    if kind == "attention":
        dim = rng.choice([64, 72, 128, 128])
        if dtype == "f32":
            return dict(kind=kind, dtype=dtype, batch=rng.randint(1, 4), txt=rng.choice([0, rng.randint(1, 128)]),
                        img=_log_int(rng, 64, 1024), heads=rng.randint(2, 16), dim=rng.choice([32, dim]))
        img = _log_int(rng, 64, 14310)
        txt = rng.choice([0, rng.randint(1, 512)])
        heads = rng.randint(4, 24)
        # at most the video block's attention
        most = int(4 * 14566.0 ** 2 * 16 * 128 / (4.0 * (img + txt) ** 2 * heads * dim))
        return dict(kind=kind, dtype=dtype, batch=max(1, min(rng.randint(1, 16), most)), txt=txt, img=img, heads=heads,
                    dim=dim)
    if kind == "gemm":
        if dtype == "f32":
            m, n, k = _log_int(rng, 16, 1024), _log_int(rng, 32, 4608, 4), _log_int(rng, 64, 4608, 4)
        else:
            m, n, k = _log_int(rng, 16, 14310), _log_int(rng, 32, 8192, 8), _log_int(rng, 64, 8192, 8)
        return dict(kind=kind, dtype=dtype, m=m, n=n, k=k, rpb=rng.choice([m, max(32, m // rng.randint(2, 16))]),
                    epilogue=rng.choice(EPILOGUES))
    if kind == "block":
        block = rng.choice(["dit", "dual", "single"])
        if dtype == "f32":
            heads, dim, rows, cols = rng.randint(2, 8), rng.choice([32, 64]), rng.randint(4, 12), rng.randint(4, 12)
        else:
            heads, dim, rows, cols = rng.randint(4, 16), rng.choice([64, 72, 128] if block == "dit" else [64, 128]), \
                _log_int(rng, 8, 48), _log_int(rng, 8, 48)
        if heads * dim % 32:
            heads += heads % 2 + (heads + heads % 2) % 4
        video = block != "dit" and rng.random() < 0.4
        return dict(kind=kind, dtype=dtype, block=block, hidden=heads * dim, heads=heads, mlp=4 * heads * dim,
                    txt=0 if block == "dit" else rng.randint(1, 300), frames=rng.randint(1, 3) if video else 0,
                    rows=rows, cols=cols, batch=rng.randint(1, 2))
    if kind == "sample":
        heads, dim, steps = rng.randint(2, 6), rng.choice([32, 64]), rng.choice([8, 10, 20])
        return dict(kind=kind, dtype="f32", blocks=rng.randint(2, 6), hidden=heads * dim, heads=heads,
                    mlp=4 * heads * dim, grid=rng.randint(5, 12), patch=rng.choice([1, 2]), in_ch=4, out_ch=4,
                    classes=rng.randint(2, 100), batch=rng.randint(1, 2), cfg=rng.random() < 0.5,
                    sampler=rng.choice(["euler", "ddim"]), steps=steps, order=rng.randint(0, 3),
                    every=rng.randint(2, 5), sites=rng.randint(1, 3))
    rows = _log_int(rng, 64, 14566)
    width = rng.choice([128, 256, 768, 1024, 1152, 1536, 2048, 3072])
    if kind == "ln":
        return dict(kind=kind, dtype=dtype, rows=rows, width=width, rpb=rng.choice([rows, max(32, rows // 7)]))
    case = dict(kind=kind, dtype=dtype, rows=rows, width=width, terms=rng.randint(1, 4))
    if kind == "verify":
        case["write"] = rng.random() < 0.5
    return case


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

class _Rand:
    """Seeded normal tensors made on the GPU, rounded to the case's type."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(1000003 * (seed % (1 << 40)) + 17)

    def __call__(self, dims, dtype, scale=1.0):
        return torch.randn(dims, generator=self.g, device=DEV, dtype=torch.float32).mul_(scale).to(TD[dtype])


def _shape(case):
    """The package's model description of a sample or block case."""
    if case["kind"] == "sample":
        lat = case["grid"] * case["patch"]
        return syn.reduced(syn.SHAPES["tiny"], name="case", arch="dit", n_dual=case["blocks"], hidden=case["hidden"],
                           heads=case["heads"], head_dim=case["hidden"] // case["heads"], mlp=case["mlp"],
                           in_ch=case["in_ch"], out_ch=case["out_ch"], patch=case["patch"], lat_h=lat, lat_w=lat,
                           n_classes=case["classes"], batch=case["batch"], cfg=case["cfg"], dtype=case["dtype"],
                           sampler=case["sampler"])
    dit = case["block"] == "dit"
    return syn.reduced(syn.SHAPES["dit_xl2" if dit else "flux"], name="case", n_dual=0 if case["block"] == "single" else 1,
                       n_single=1 if case["block"] == "single" else 0, hidden=case["hidden"], heads=case["heads"],
                       head_dim=case["hidden"] // case["heads"], mlp=case["mlp"], patch=2, patch_t=1,
                       lat_f=case["frames"], lat_h=2 * case["rows"], lat_w=2 * case["cols"], txt_tokens=case["txt"],
                       batch=case["batch"], cfg=False, rope_dims=0 if dit else 3 if case["frames"] else 2,
                       dtype=case["dtype"], sampler="euler")


def _schedule(case):
    refresh = tuple(range(0, case["steps"], case["every"]))
    free = [i for i in range(case["steps"]) if i not in refresh]
    n = min(case["sites"], len(free))
    sites = tuple((free[(2 * j + 1) * len(free) // (2 * n)], (2 * j + 1) * case["blocks"] // (2 * n)) for j in range(n))
    return refresh, sites


BLOCK_STEPS, BLOCK_STEP = 4, 1    # a block case evaluates its block at step 1 of a 4-step schedule


def _inputs(case, seed):
    """Everything the call reads, as tensors on the GPU."""
    r, kind, dt = _Rand(seed), case["kind"], case["dtype"]
    if kind in ("sample", "block"):
        sh = _shape(case)
        w = {name: r(dims, dt, 0.02) for name, dims in ff.weight_spec(sh)}
        d = {"w": w}
        bm = sh.batch_model
        if sh.arch == "dit":
            lab = torch.randint(0, sh.n_classes, (sh.batch,), generator=r.g, device=DEV, dtype=torch.int32)
            d["cond"] = torch.cat([lab, torch.full_like(lab, sh.n_classes)]) if sh.cfg else lab
        else:
            d["cond"] = r((bm, sh.txt_tokens, sh.hidden), "f32")
        if kind == "block":
            d["u"] = r((bm * sh.tokens, sh.hidden), dt)
        return d
    if kind == "attention":
        return {"qkv": r((case["batch"] * (case["txt"] + case["img"]), 3 * case["heads"] * case["dim"]), dt)}
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        d = {"a": r((m, k), dt), "w": r((n, k), dt, 0.02), "bias": r((n,), dt, 0.02)}
        if case["epilogue"].startswith("gated"):
            # the gate is the third of the six modulation chunks of a block
            d["gate"] = r((-(-m // case["rpb"]), 6 * n), "f32", 0.5)[:, 2 * n:3 * n]
            d["resid"] = r((m, n), dt)
        if case["epilogue"] == "gated_history":
            d["base"] = r((m, n), dt)
        return d
    n = case["rows"] * case["width"]
    if kind == "ln":
        # shift and scale are the first two of the six modulation chunks
        mod = r((-(-case["rows"] // case["rpb"]), 6 * case["width"]), "f32", 0.1)
        return {"x": r((case["rows"], case["width"]), dt, 2.0), "shift": mod[:, :case["width"]],
                "scale": mod[:, case["width"]:2 * case["width"]]}
    d = {"x": r((n,), dt), "hist": [r((n,), dt, 0.1) for _ in range(case["terms"])]}
    if kind == "verify":
        d["hf"] = (d["x"].float() + r((n,), "f32", 0.1)).to(TD[dt])
    return d


# Lagrange weights one step after the newest of refreshes three steps apart.
WEIGHTS = {1: (1.0,), 2: (4 / 3, -1 / 3), 3: (14 / 9, -7 / 9, 2 / 9), 4: (140 / 81, -35 / 27, 20 / 27, -14 / 81)}


def prepare(case, seed):
    d = _inputs(case, seed)
    kind, dt = case["kind"], case["dtype"]
    s = {"case": case, "seed": seed % (1 << 62), **d}
    if kind in ("sample", "block"):
        sh = _shape(case)
        s["model"] = ff.FeatFix(sh, d["w"])
        if kind == "sample":
            refresh, sites = _schedule(case)
            s["model"].set_schedule(case["steps"], refresh, case["order"], sites, "featfix")
            s["out"] = torch.empty(sh.latent_dims, dtype=torch.float32, device=DEV)
        else:
            s["model"].set_schedule(BLOCK_STEPS, tuple(range(BLOCK_STEPS)), 0, (), "featfix")
            s["out"] = torch.empty_like(d["u"])
    elif kind == "attention":
        s["out"] = torch.empty((d["qkv"].shape[0], case["heads"] * case["dim"]), dtype=TD[dt], device=DEV)
    elif kind == "gemm":
        s["out"] = torch.empty((case["m"], case["n"]), dtype=TD[dt], device=DEV)
        s["hist"] = torch.empty_like(s["out"]) if "base" in d else None
    elif kind == "ln":
        s["out"] = torch.empty_like(d["x"])
    elif kind == "verify":
        s["ws"] = torch.empty(ff.featfix_op_verify_workspace(d["x"].numel()), dtype=torch.uint8, device=DEV)
        s["sums"] = torch.zeros(4, dtype=torch.float64, device=DEV)
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------

def run(s):
    case = s["case"]
    kind, dt = case["kind"], case["dtype"]
    if kind == "sample":
        s["model"].sample(s["seed"], case["steps"], s["cond"], s["out"])
        return s["out"]
    if kind == "block":
        ff.featfix_debug_block(s["model"].ctx, BLOCK_STEP, 0, s["u"], s["out"], s["cond"])
        return s["out"]
    if kind == "attention":
        ff.featfix_op_attention(dt, s["qkv"], s["out"], case["batch"], case["txt"], case["img"], case["heads"],
                                case["dim"])
        return s["out"]
    if kind == "gemm":
        gated = "gate" in s
        ff.featfix_op_gemm(dt, s["a"], s["w"], s["out"], bias=s["bias"], act=int(case["epilogue"] == "gelu"),
                           gate=s.get("gate"), gate_stride=6 * case["n"] if gated else 0,
                           rows_per_batch=case["rpb"] if gated else 0, resid=s.get("resid"), hist_base=s.get("base"),
                           hist_out=s["hist"])
        return [s["out"]] if s["hist"] is None else [s["out"], s["hist"]]
    if kind == "ln":
        c = case["width"]
        ff.featfix_op_ln_modulate(dt, s["x"], s["out"], case["rows"], c, s["shift"], s["scale"], 6 * c, case["rpb"])
        return s["out"]
    w = WEIGHTS[case["terms"]]
    if kind == "draft":
        # in place, as the drafts of consecutive blocks are chained
        ff.featfix_op_draft(dt, s["x"], s["hist"], w)
        return s["x"]
    ff.featfix_op_verify(dt, s["x"], s["hist"], w, s["hf"], s["sums"], s["ws"], write_draft=case["write"])
    return [s["sums"], s["x"]] if case["write"] else [s["sums"]]


# ----------------------------------------------------------------------------
# the least work of a pass
# ----------------------------------------------------------------------------

def work(case):
    kind, b = case["kind"], 4 if case["dtype"] == "f32" else 2
    if kind == "attention":
        t = case["txt"] + case["img"]
        c = case["heads"] * case["dim"]
        return {"bytes": 4 * case["batch"] * t * c * b, "flops": 4 * case["batch"] * t * t * c}
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        extra = {"bias": 0, "gelu": 0, "gated": 1, "gated_history": 3}[case["epilogue"]]
        return {"bytes": (m * k + n * k + (1 + extra) * m * n) * b, "flops": 2 * m * n * k}
    if kind == "block":
        bm, c, mlp, txt = case["batch"], case["hidden"], case["mlp"], case["txt"]
        img = max(case["frames"], 1) * case["rows"] * case["cols"]
        t = bm * (txt + img)
        streams = 2 if case["block"] == "dual" else 1
        mods = (3 if case["block"] == "single" else 6) * c * c * streams
        weights = streams * (4 * c * c + 2 * c * mlp)
        return {"bytes": (2 * t * c + weights + mods) * b,
                "flops": 2 * t * (4 * c * c + 2 * c * mlp) + 4 * bm * (txt + img) ** 2 * c + 2 * bm * mods}
    if kind == "sample":
        refresh, sites = _schedule(case)
        c, mlp, L, p = case["hidden"], case["mlp"], case["blocks"], case["patch"] ** 2
        bm, t = case["batch"] * (2 if case["cfg"] else 1), case["grid"] ** 2
        blocks = len(refresh) * L + len(sites)
        block = 2 * bm * t * (4 * c * c + 2 * c * mlp) + 4 * bm * t * t * c
        ends = 2 * bm * t * c * p * (case["in_ch"] + case["out_ch"])
        mods = 2 * bm * (len(refresh) + len(sites)) * 6 * c * c * L
        e = bm * t * c * b
        # weights once per exact block, the history written at a refresh, and
        # each drafted step's state and history terms read once
        drafted = case["steps"] - len(refresh)
        terms = min(case["order"] + 1, len(refresh))
        return {"bytes": blocks * (4 * c * c + 2 * c * mlp) * b + 6 * c * c * L * b + len(refresh) * L * e
                + drafted * (terms + 2) * e,
                "flops": blocks * block + case["steps"] * ends + mods}
    n = case["rows"] * case["width"]
    if kind == "ln":
        return {"bytes": 2 * n * b + 8 * case["width"] * -(-case["rows"] // case["rpb"]), "flops": 0}
    if kind == "draft":
        return {"bytes": (case["terms"] + 2) * n * b, "flops": 0}
    return {"bytes": (case["terms"] + 2 + int(case["write"])) * n * b, "flops": 0}


# ----------------------------------------------------------------------------
# how far two correct implementations may be apart: about four times the
# largest distance from float64 measured over the ranges (bf16 2.3e-3 and at
# most 2e-2 of a value: the rounding of stored values; fp32 layers 1.2e-6,
# blocks 5e-8, runs 7e-7; the check's sums 1.4e-6); the whole bf16 run by
# evaluating its drafts and norms in another order (6e-3 and 1.1e-2)
# ----------------------------------------------------------------------------

def tolerance(case):
    kind = case["kind"]
    if case["dtype"] == "f32":
        return {"rel": 1e-6 if kind == "block" else 5e-6, "max": 1e-4}
    if kind == "sample":
        return {"rel": 0.03, "max": 0.2}
    if kind == "verify" and not case["write"]:
        return {"rel": 1e-5, "max": 1e-5}
    return {"rel": 1e-2, "max": 8e-2}


# ----------------------------------------------------------------------------
# the same calls in plain float64 torch
# ----------------------------------------------------------------------------

def _ln(x):
    mu = x.mean(-1, keepdim=True)
    return (x - mu) / torch.sqrt(((x - mu) ** 2).mean(-1, keepdim=True) + 1e-6)


def _gelu(x):
    return 0.5 * x * (1 + torch.tanh(math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)))


def _silu(x):
    return x / (1 + torch.exp(-x))


def _attend(q, k, v):
    """[tokens, heads, dim] of one sample."""
    out = torch.empty_like(q)
    for h in range(q.shape[1]):
        out[:, h] = torch.softmax(q[:, h] @ k[:, h].T / math.sqrt(q.shape[2]), -1) @ v[:, h]
    return out


def _samples(x, bm, txt, img):
    """Rows (all text, then all image) -> [sample, token, ...], text first."""
    t = x[:bm * txt].reshape(bm, txt, *x.shape[1:])
    i = x[bm * txt:].reshape(bm, img, *x.shape[1:])
    return torch.cat([t, i], 1)


def _rows(x, txt):
    """The inverse of _samples."""
    return torch.cat([x[:, :txt].reshape(-1, *x.shape[2:]), x[:, txt:].reshape(-1, *x.shape[2:])])


def _joint(qkv, heads):
    """Joint attention of [sample, token, 3C] (rotated already)."""
    bm, t, c3 = qkv.shape
    q, k, v = (z.reshape(bm, t, heads, -1) for z in qkv.split(c3 // 3, -1))
    return torch.stack([_attend(q[b], k[b], v[b]) for b in range(bm)]).reshape(bm, t, c3 // 3)


def _rope(qkv, heads, txt, grid):
    """Rotary positions on the image tokens' q and k of [sample, token, 3C]."""
    bm, t, c3 = qkv.shape
    d = c3 // 3 // heads
    axes = (d // 2, d // 2) if len(grid) == 2 else (d // 8, (d - d // 8) // 2, d - d // 8 - (d - d // 8) // 2)
    pos = torch.cartesian_prod(*[torch.arange(g, device=DEV, dtype=torch.float64) for g in grid])
    ang = torch.cat([pos[:, a:a + 1] * 10000.0 ** (-2.0 * torch.arange(w // 2, device=DEV, dtype=torch.float64) / w)
                     for a, w in enumerate(axes)], 1)
    cos, sin = torch.cos(ang)[None, :, None], torch.sin(ang)[None, :, None]
    x = qkv.clone().reshape(bm, t, 3, heads, d)
    for s in (0, 1):
        z = x[:, txt:, s]
        a, b = z[..., 0::2].clone(), z[..., 1::2].clone()
        z[..., 0::2] = a * cos - b * sin
        z[..., 1::2] = a * sin + b * cos
    return x.reshape(bm, t, c3)


def _lin(w, name, x):
    return x @ w[name + ".w"].T + w[name + ".b"]


def _cond(w, t, labels, bm):
    k = torch.arange(128, device=DEV, dtype=torch.float64)
    a = t * torch.exp(-math.log(10000.0) * k / 128)
    c = _lin(w, "t_fc2", _silu(_lin(w, "t_fc1", torch.cat([torch.cos(a), torch.sin(a)]))))
    c = c[None].expand(bm, -1)
    return _silu(c + w["y_emb"][labels.long()] if labels is not None else c)


def _branches(w, p, u, m, heads, attend):
    """Attention and MLP branches of a DiT block, or of one stream."""
    u1 = u + m[2][:, None] * _lin(w, p + "proj", attend)
    h = _ln(u1) * (1 + m[4][:, None]) + m[3][:, None]
    return u1 + m[5][:, None] * _lin(w, p + "fc2", _gelu(_lin(w, p + "fc1", h)))


def _dit_block(w, p, u, c, heads):
    m = _lin(w, p + "mod", c).chunk(6, -1)
    qkv = _lin(w, p + "qkv", _ln(u) * (1 + m[1][:, None]) + m[0][:, None])
    return _branches(w, p, u, m, heads, _joint(qkv, heads))


def _dual_block(w, p, u, c, heads, txt, grid):
    parts, mods, qkv = (u[:, :txt], u[:, txt:]), [], []
    for name, x in zip(("txt_", "img_"), parts):
        m = _lin(w, p + name + "mod", c).chunk(6, -1)
        mods.append(m)
        qkv.append(_lin(w, p + name + "qkv", _ln(x) * (1 + m[1][:, None]) + m[0][:, None]))
    o = _joint(_rope(torch.cat(qkv, 1), heads, txt, grid), heads)
    return torch.cat([_branches(w, p + "txt_", parts[0], mods[0], heads, o[:, :txt]),
                      _branches(w, p + "img_", parts[1], mods[1], heads, o[:, txt:])], 1)


def _single_block(w, p, u, c, heads, txt, grid):
    sh, sc, g = _lin(w, p + "mod", c).chunk(3, -1)
    y = _lin(w, p + "lin1", _ln(u) * (1 + sc[:, None]) + sh[:, None])
    width = u.shape[-1]
    o = _joint(_rope(y[..., :3 * width], heads, txt, grid), heads)
    return u + g[:, None] * _lin(w, p + "lin2", torch.cat([o, _gelu(y[..., 3 * width:])], -1))


def _normals(seed, count):
    """SplitMix64 counters to normals, as featfix_sample defines x_T."""
    n = count + count % 2
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = ((z >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    r, phi = np.sqrt(-2 * np.log(u[0::2])), 2 * np.pi * u[1::2]
    out = np.stack([r * np.cos(phi), r * np.sin(phi)], 1).reshape(-1)[:count]
    return torch.from_numpy(out.astype(np.float32).astype(np.float64)).to(DEV)


def _sample(case, w, labels, seed):
    steps, C, L, g, p, ci = (case[k] for k in ("steps", "hidden", "blocks", "grid", "patch", "in_ch"))
    refresh, sites = _schedule(case)
    bl, co = case["batch"], case["out_ch"]
    bm = bl * (2 if case["cfg"] else 1)
    x = _normals(seed, bl * ci * (g * p) ** 2).reshape(bl, ci, g * p, g * p)
    q = C // 4
    freq = 10000.0 ** (-torch.arange(q, device=DEV, dtype=torch.float64) / q)
    half = torch.arange(g, device=DEV, dtype=torch.float64)[:, None] * freq
    half = torch.cat([torch.sin(half), torch.cos(half)], 1)
    pos = torch.cat([half[:, None].expand(g, g, -1), half[None].expand(g, g, -1)], -1).reshape(g * g, C)
    ab = torch.cumprod(1 - torch.linspace(1e-4, 0.02, 1000, dtype=torch.float64), 0).tolist()
    hist = [[] for _ in range(L)]
    for i in range(steps):
        ddim = case["sampler"] == "ddim"
        t = float(1000 - 1000 // steps * (i + 1)) if ddim else 1000.0 * (1 - i / steps)
        c = _cond(w, t, labels, bm)
        y = x.reshape(bl, ci, g, p, g, p).permute(0, 2, 4, 1, 3, 5).reshape(bl, g * g, -1)
        u = _lin(w, "x_emb", torch.cat([y, y]) if case["cfg"] else y) + pos
        for l in range(L):
            if i in refresh:
                h = _dit_block(w, "blk%d." % l, u, c, case["heads"])
                hist[l] = ([(i, h - u)] + hist[l])[:case["order"] + 1]
            elif (i, l) in sites:
                h = _dit_block(w, "blk%d." % l, u, c, case["heads"])
            else:   # the polynomial through the refreshed increments, at i
                h = u
                for a, (sa, ra) in enumerate(hist[l]):
                    h = h + ra * math.prod((i - sb) / (sa - sb) for b, (sb, _) in enumerate(hist[l]) if b != a)
            u = h
        sh, sc = _lin(w, "final.mod", c).chunk(2, -1)
        y = _lin(w, "final.lin", _ln(u) * (1 + sc[:, None]) + sh[:, None])
        y = y.reshape(bm, g, g, co, p, p).permute(0, 3, 1, 4, 2, 5).reshape(bm, co, g * p, g * p)
        if case["cfg"]:
            y = y[bl:] + 4.0 * (y[:bl] - y[bl:])
        y = y[:, :ci]
        if ddim:
            at, stride = ab[int(t)], 1000 // steps
            ap = ab[int(t) - stride] if i + 1 < steps else 1.0
            x = math.sqrt(ap) * (x - math.sqrt(1 - at) * y) / math.sqrt(at) + math.sqrt(1 - ap) * y
        else:
            x = x - y / steps
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "sample" and case["dtype"] == "bf16":
        return None     # tens of TFLOP
    d = _inputs(case, seed)

    def wide(v):
        return [wide(x) for x in v] if isinstance(v, list) else v.double() if v.is_floating_point() else v

    w = {k: wide(v) for k, v in d.pop("w").items()} if kind in ("sample", "block") else None
    d = {k: wide(v) for k, v in d.items()}
    if kind == "sample":
        return _sample(case, w, d["cond"], seed % (1 << 62))
    if kind == "block":
        bm, txt = case["batch"], case["txt"]
        img = max(case["frames"], 1) * case["rows"] * case["cols"]
        grid = ((case["frames"],) if case["frames"] else ()) + (case["rows"], case["cols"])
        dit = case["block"] == "dit"
        c = _cond(w, 1000.0 * (1 - BLOCK_STEP / BLOCK_STEPS), d["cond"] if dit else None, bm)
        u = _samples(d["u"], bm, txt, img)
        if dit:
            out = _dit_block(w, "blk0.", u, c, case["heads"])
        elif case["block"] == "dual":
            out = _dual_block(w, "dual0.", u, c, case["heads"], txt, grid)
        else:
            out = _single_block(w, "single0.", u, c, case["heads"], txt, grid)
        return _rows(out, txt)
    if kind == "attention":
        return _rows(_joint(_samples(d["qkv"], case["batch"], case["txt"], case["img"]), case["heads"]), case["txt"])
    if kind == "gemm":
        y = d["a"] @ d["w"].T + d["bias"]
        if case["epilogue"] == "gelu":
            y = _gelu(y)
        if "gate" in d:
            y = d["resid"] + d["gate"][torch.arange(case["m"], device=DEV) // case["rpb"]] * y
        return [y, y - d["base"]] if "base" in d else [y]
    if kind == "ln":
        row = torch.arange(case["rows"], device=DEV) // case["rpb"]
        return _ln(d["x"]) * (1 + d["scale"][row]) + d["shift"][row]
    h = d["x"] + sum(a * r for a, r in zip(WEIGHTS[case["terms"]], d["hist"]))
    if kind == "draft":
        return h
    stored = h.to(TD[case["dtype"]]).double()     # the discrepancy is of the draft as it would be forwarded
    e = stored - d["hf"]
    sums = torch.stack([e.abs().sum(), d["hf"].abs().sum(), (e * e).sum(), (d["hf"] ** 2).sum()])
    return [sums, h] if case["write"] else [sums]
