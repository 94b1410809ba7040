"""Performance cases of the library: calls a user's program makes, with their inputs, their
least work, their tolerances and their results in 64 bits.

A case is a dict of plain values. Its ``kind`` says which entry point it calls:

  layer     one attention layer on a mask that the program built once for its prefill and keeps
            (``ris_attention_masked``): every layer of a prefill after the first call.
  call      mask and attention in one call (``ris_sparse_attention_fwd``): a single layer, or a
            program that keeps no mask.
  ensemble  one output per seed (``ris_ensemble_batch``): the independent sparse views.
  mask      the mask of a prefill, with its offsets and bitmap read back as tensors.
  step      one decode step over a rotated K/V cache (``ris_decode_step``), called directly.
  token     one generated token: a decode step per layer, captured once as a CUDA graph and
            replayed per token.

Shapes: 12 / 2 heads of 128 and 32 / 4 heads of 64 are the two grouped-query layers the
benchmark runs, 1 / 1 head of 128 its single-head layer; 8 / 8 and 16 / 1 heads are plain
multi-head and multi-query attention.
"""
from __future__ import annotations

import math

import torch

from paper_2607_21927_gb300 import ris

STOCHASTIC, STRUCTURAL, DENSE = 0, 1, 2
M32 = 0xFFFFFFFF

_DEFAULTS = dict(
    kind="layer", n=0, hq=12, hkv=2, d=128, dtype="bf16", out="bf16", lse=False, outliers=True,
    mode=STOCHASTIC, density=0.01, seeds=10, rope="yarn", theta=1e6, native=32768,
    window=1, anchors=0, per_head=False, draws=False,
    layers=1, generated=0, decode_window=1024)


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest layer: one head in fp32, 5% of the pairs; launches and latency count
        _case("layer-2k-fp32-1head", n=2048, hq=1, hkv=1, dtype="f32", out="f32", lse=True, outliers=False,
              density=0.05, seeds=1, rope="plain"),
        # the fp32 grouped-query layer: the precision of the paper's own runs
        _case("layer-6k-fp32", n=6007, dtype="f32", out="f32", outliers=False, seeds=5, rope="plain"),
        # an ordinary short prefill: ten seeds merged, about a tenth of the pairs
        _case("layer-8k", n=8192, rope="plain"),
        # head dim 64, block cliques plus global draws, positions far beyond the native window
        _case("layer-16k-hd64-blocks", n=16384, hq=32, hkv=4, d=64, out="f32", outliers=False, mode=STRUCTURAL,
              theta=1e4, native=2048),
        # the dense causal upper bound at the native window
        _case("layer-32k-dense", n=32768, mode=DENSE, density=1.0, seeds=1, rope="plain", lse=True),
        # the longest prefill, both modes: the two layers of the headline benchmark
        _case("layer-64k", n=65536),
        _case("layer-64k-blocks", n=65536, mode=STRUCTURAL),
        # one call for mask and attention at an odd length, short and sparse
        _case("call-3001", kind="call", n=3001, seeds=3, rope="plain", out="f32", lse=True),
        # independent sparse views, one output per seed
        _case("ensemble-8k", kind="ensemble", n=8192, rope="plain"),
        # the mask of a large ensemble
        _case("mask-32k-70seeds", kind="mask", n=32768, seeds=70),
        # decode: one step called directly on a short cache, and a token's layers as one graph
        _case("step-1500-hd64", kind="step", n=1500, hq=32, hkv=4, d=64, outliers=False, theta=1e4, native=2048,
              generated=20, decode_window=512),
        _case("token-64k", kind="token", n=65536, layers=28, generated=24),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["layer", "call", "ensemble", "mask", "step", "token"], [8, 3, 2, 2, 2, 1])[0]
    hq, hkv, d = rng.choices([(12, 2, 128), (32, 4, 64), (1, 1, 128), (8, 8, 128), (16, 1, 128)], [8, 4, 1, 1, 1])[0]
    c = _case(kind=kind, hq=hq, hkv=hkv, d=d, outliers=d == 128)
    c["mode"] = rng.choices([STOCHASTIC, STRUCTURAL, DENSE], [5, 4, 1 if kind in ("layer", "call") else 0])[0]
    c["density"] = 1.0 if c["mode"] == DENSE else round(math.exp(rng.uniform(math.log(0.002), math.log(0.1))), 4)
    c["seeds"] = 1 if c["mode"] == DENSE else _log_int(rng, 1, 70)
    c["rope"] = rng.choices(["none", "plain", "linear", "yarn"], [1, 3, 1, 4])[0]
    c["theta"], c["native"] = (1e4, 2048) if d == 64 else (1e6, 32768)
    c["out"] = rng.choice(["bf16", "f32"])
    c["lse"] = rng.random() < 0.3
    c["draws"] = rng.random() < 0.15
    c["per_head"] = rng.random() < 0.1
    if rng.random() < 0.2:  # a dense local window and a few initial tokens
        c["window"], c["anchors"] = rng.choice([64, 256, 1024]), 4
    if hq // hkv <= 8 and kind in ("layer", "call", "step") and rng.random() < 0.25:
        c["dtype"], c["out"], c["outliers"] = "f32", "f32", False
    if kind in ("step", "token"):
        if hq // hkv > 8:
            c["hq"] = 8 * hkv
        c["n"] = _log_int(rng, 200, 65536)
        c["generated"] = rng.randint(1, 64)
        c["layers"] = rng.randint(2, 28) if kind == "token" else 1
        c["decode_window"] = rng.choice([64, 512, 1024])
        c["window"], c["lse"] = 1, False
        if kind == "token":
            c["dtype"], c["out"] = "bf16", "bf16"
    elif kind == "mask":
        c["n"] = _log_int(rng, 500, 65536)
        c["seeds"] = min(c["seeds"], max(1, int(70 * 32768 ** 2 / c["n"] ** 2)))
        c["per_head"] = False
    elif kind == "ensemble":
        c["n"] = _log_int(rng, 300, 16000)
        c["seeds"] = max(2, min(c["seeds"], 10))
        c["density"] = min(c["density"], 0.02)
    else:
        # the most tokens that keep the pairs of all heads within the listed 64k layer's
        most = 65536 * math.sqrt(12 / max(hq, 1))
        if c["dtype"] == "f32":
            most = 8000
            c["density"] = c["density"] if c["mode"] == DENSE else min(c["density"], 0.02)
            if c["mode"] == DENSE:
                most = 3000
        c["n"] = _log_int(rng, 200, min(65536, most))
        c["seeds"] = min(c["seeds"], max(1, int(12 * 65536 ** 2 / c["n"] ** 2)))
    return c


# ---------------------------------------------------------------- inputs
def _tensor(gen, n, h, d, dtype, outliers):
    x = torch.randn(n, h * d, generator=gen, device="cuda")
    if outliers:  # a hundredth of the channels carries activations eight times as large
        m = max(1, round(0.01 * h * d))
        x[:, torch.randperm(h * d, generator=gen, device="cuda")[:m]] *= 8.0
    return x.view(n, h, d).to(dtype)


def _dtype(s):
    return torch.bfloat16 if s == "bf16" else torch.float32


def _inputs(c, seed, layer=0):
    """q, k, v of one layer; the decode kinds get one query and a whole cache of keys and values."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 64 + layer)
    decode = c["kind"] in ("step", "token")
    rows = c["n"] + c["generated"] if decode else c["n"]
    dt = _dtype(c["dtype"])
    q = _tensor(gen, 1 if decode else rows, c["hq"], c["d"], dt, c["outliers"])
    k = _tensor(gen, rows, c["hkv"], c["d"], dt, c["outliers"])
    v = _tensor(gen, rows, c["hkv"], c["d"], dt, c["outliers"])
    return q, k, v


def _mask_seeds(c, seed):
    return [(int(seed) * 1009 + i) & M32 for i in range(c["seeds"])]


def _rope(c):
    if c["rope"] == "none":
        return None
    kind = {"plain": ris.ROPE_PLAIN, "linear": ris.ROPE_LINEAR, "yarn": ris.ROPE_YARN}[c["rope"]]
    return ris.rope_cfg(kind, c["theta"], c["native"])


def _opts(c):
    return ris.mask_opts(c["window"], c["anchors"], c["per_head"],
                         sampler=ris.SAMPLER_DRAWS if c["draws"] else ris.SAMPLER_BERNOULLI)


class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.case, s.rope, s.opts, s.seeds = c, _rope(c), _opts(c), _mask_seeds(c, seed)
    s.out_dtype = _dtype(c["out"])
    if c["kind"] == "mask":
        return s
    if c["kind"] in ("step", "token"):
        s.anchor = ris.ris_decode_anchor(c["n"], c["hkv"], c["mode"], c["density"], s.seeds, s.opts)
        s.t = c["n"] + c["generated"] - 1
        s.n_ctx = c["n"] + c["generated"]
        s.layers = []
        for layer in range(c["layers"]):
            q, k, v = _inputs(c, seed, layer)
            hi, lo = ris.ris_rope_split(k, s.n_ctx, s.rope)
            s.layers.append((q[0].contiguous(), hi, lo, v))
        s.out = torch.empty(c["layers"], c["hq"], c["d"], dtype=s.out_dtype, device="cuda")
        if c["kind"] == "token":
            # the position lives on the device, so that one graph serves every token
            s.t_dev = torch.full((1,), s.t, dtype=torch.int64, device="cuda")
            _steps(s)
            torch.cuda.synchronize()
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s.graph):
                _steps(s)
        return s
    s.q, s.k, s.v = _inputs(c, seed)
    if c["kind"] == "layer":
        s.mask = ris.ris_mask_generate(c["n"], c["hkv"], c["mode"], c["density"], s.seeds, s.opts)
    return s


def _steps(s):
    c = s.case
    for layer, (q, hi, lo, v) in enumerate(s.layers):
        ris.ris_decode_step(s.anchor, q, hi, lo, v, s.t, c["decode_window"], s.n_ctx, s.rope, out=s.out[layer],
                            out_dtype=s.out_dtype, t_dev=getattr(s, "t_dev", None))


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "layer":
        return ris.ris_attention_masked(s.mask, s.q, s.k, s.v, s.rope, out_dtype=s.out_dtype, return_lse=c["lse"])
    if kind == "call":
        return ris.ris_sparse_attention_fwd(s.q, s.k, s.v, c["mode"], c["density"], s.seeds, s.rope, s.opts,
                                            out_dtype=s.out_dtype, return_lse=c["lse"])
    if kind == "ensemble":
        return ris.ris_ensemble_batch(s.q, s.k, s.v, c["mode"], c["density"], s.seeds, s.rope, s.opts,
                                      out_dtype=s.out_dtype, return_lse=c["lse"])
    if kind == "mask":
        with ris.ris_mask_generate(c["n"], c["hkv"], c["mode"], c["density"], s.seeds, s.opts) as m:
            # the bitmap is the whole mask (the key lists repeat it, and their number varies with the
            # seeds; the layer and call cases read them)
            return m.row_ptr(), m.bitmap()
    if kind == "step":
        _steps(s)
        return s.out
    s.graph.replay()
    return s.out


# ---------------------------------------------------------------- work
def _geometry(n, mode, density):
    """(block size, causal clique pairs, density of the global draws) of the Structural mode."""
    block = max(1, min(n // 10, int(math.floor(density * n + 0.5))))
    nb = n // block
    rem = n - nb * block
    clique = nb * (block * (block + 1) // 2) + rem * (rem + 1) // 2
    return block, clique, max(0.0, density - clique / (n * n))


def _hit(c, n):
    """Probability that one drawn pair is kept by one seed."""
    p = _geometry(n, c["mode"], c["density"])[2] if c["mode"] == STRUCTURAL else c["density"]
    if c["draws"]:
        return 1.0 - (1.0 - 1.0 / n) ** math.floor(p * n + 0.5)
    return p


def _pairs(c, seeds):
    """Expected kept pairs of one mask."""
    n = c["n"]
    total = n * (n + 1) / 2
    if c["mode"] == DENSE or c["density"] >= 1.0:
        return total
    w = min(c["window"], n)
    forced = w * (w + 1) / 2 + (n - w) * w
    if c["mode"] == STRUCTURAL:
        forced = max(forced, _geometry(n, c["mode"], c["density"])[1])
    forced = min(total, forced + c["anchors"] * max(0, n - w))
    return forced + (total - forced) * (1.0 - (1.0 - _hit(c, n)) ** seeds)


def _draw_ops(c, rows_pairs):
    """Integer operations of the draws: a Philox call of 10 rounds (2 wide products, 4 exclusive
    ors, 2 key additions each) and 4 comparisons per 4 words."""
    if c["mode"] == DENSE or c["density"] >= 1.0:
        return 0.0
    words = c["n"] * math.floor(_hit(c, c["n"]) * c["n"] + 0.5) if c["draws"] else rows_pairs
    return c["seeds"] * words / 4.0 * 84.0


def work(case):
    c = case
    n, hq, hkv, d = c["n"], c["hq"], c["hkv"], c["d"]
    esz, osz = (2 if c["dtype"] == "bf16" else 4), (2 if c["out"] == "bf16" else 4)
    csz = 2 if n <= 65536 else 4
    if c["kind"] == "mask":
        pairs = _pairs(c, c["seeds"])
        # the bitmap, the offsets and the key lists are written once
        return {"bytes": n * n / 16 + 8.0 * n + csz * pairs, "flops": _draw_ops(c, n * (n + 1) / 2)}
    if c["kind"] in ("step", "token"):
        lists = c["hkv"] if c["per_head"] else 1
        keys = min(n, (1.0 - (1.0 - _hit(c, n)) ** c["seeds"]) * n + c["anchors"]) + min(c["decode_window"], n)
        keys = min(keys, n + c["generated"])
        per_key = hkv * d * (3 * 2 if c["dtype"] == "bf16" else 2 * 4)
        step = keys * per_key + 4 * keys * lists + hq * d * (esz + osz)
        return {"bytes": c["layers"] * step, "flops": c["layers"] * 4.0 * d * hq * keys}
    sets = c["seeds"] if c["kind"] == "ensemble" else 1
    masks = sets * (hkv if c["per_head"] else 1)
    pairs = _pairs(c, 1 if c["kind"] == "ensemble" else c["seeds"])
    nbytes = n * d * (hq + 2 * hkv) * esz + sets * n * hq * (d * osz + (4 if c["lse"] else 0))
    flops = 4.0 * d * hq * pairs * sets
    if c["mode"] != DENSE and c["density"] < 1.0:
        nbytes += masks * min(csz * pairs + 8.0 * n, n * n / 16.0)
        if c["kind"] != "layer":
            flops += _draw_ops(c, n * (n + 1) / 2) * (hkv if c["per_head"] else 1)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    c = case
    if c["kind"] == "mask":
        return "exact"
    if c["out"] == "bf16":
        return {"rel": 7e-3, "max": 3e-2}
    if c["dtype"] == "bf16":
        return {"rel": 1e-3, "max": 2e-2}
    return {"rel": 1e-5, "max": 1e-4}


# ---------------------------------------------------------------- the same results in 64 bits
def _philox(x, y, z, w, k0, k1):
    """Philox4x32-10 of counter words x, y, z, w (int64 tensors or ints) under key (k0, k1)."""
    for _ in range(10):
        p0, p1 = x * 0xD2511F53, z * 0xCD9E8D57  # low 64 bits of the product, as int64
        x, y, z, w = ((p1 >> 32) & M32) ^ y ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ w ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x, y, z, w


def _drawn(c, seeds, r0, r1, cols, head):
    """Kept draws (i, j), r0 <= i < r1, j < cols: the union over seeds, before forced keys."""
    n, dev = c["n"], "cuda"
    kept = torch.zeros(r1 - r0, (cols + 3) // 4 * 4, dtype=torch.bool, device=dev)
    structural = c["mode"] == STRUCTURAL
    p = _geometry(n, c["mode"], c["density"])[2] if structural else c["density"]
    rows = torch.arange(r0, r1, dtype=torch.int64, device=dev)[:, None]
    stream = (1 if structural else 0) + (2 if c["draws"] else 0)
    for seed in seeds:
        if c["draws"]:
            count = int(math.floor(p * n + 0.5))
            if count == 0:
                continue
            g = torch.arange((count + 3) // 4, dtype=torch.int64, device=dev)[None, :].expand(r1 - r0, -1)
            u = torch.stack(_philox(g, rows, torch.full_like(g, stream), torch.zeros_like(g), seed, head), -1)
            j = (u.reshape(r1 - r0, -1)[:, :count] * n) >> 32
            hits = torch.zeros(r1 - r0, max(n, kept.shape[1]), dtype=torch.bool, device=dev).scatter_(1, j, True)
            kept |= hits[:, :kept.shape[1]]
        else:
            thr = min(1 << 32, int(math.floor(p * 4294967296.0 + 0.5)))
            if thr == 0:
                continue
            g = torch.arange(kept.shape[1] // 4, dtype=torch.int64, device=dev)[None, :].expand(r1 - r0, -1)
            u = torch.stack(_philox(g, rows, torch.full_like(g, stream), torch.zeros_like(g), seed, head), -1)
            kept |= u.reshape(r1 - r0, -1) < thr
    return kept[:, :cols]


def _mask_rows(c, seeds, r0, r1, cols, head):
    """Rows r0 .. r1 - 1 of the mask over keys 0 .. cols - 1."""
    i = torch.arange(r0, r1, device="cuda")[:, None]
    j = torch.arange(cols, device="cuda")[None, :]
    if c["mode"] == DENSE or c["density"] >= 1.0:
        return j <= i
    keep = _drawn(c, seeds, r0, r1, cols, head) & (j < i)
    keep |= (j > i - c["window"]) | (j < c["anchors"])
    if c["mode"] == STRUCTURAL:
        block = _geometry(c["n"], c["mode"], c["density"])[0]
        keep |= j >= i // block * block
    return keep & (j <= i)


def _rotate(c, x, positions, n_ctx):
    """RoPE of x [rows, heads, d] at the positions, in 64 bits."""
    x = x.double()
    if c["rope"] == "none":
        return x
    half = c["d"] // 2
    base = c["theta"] ** (-2.0 * torch.arange(half, dtype=torch.float64, device=x.device) / c["d"])
    s, m = max(1.0, n_ctx / c["native"]), 1.0
    if c["rope"] == "linear":
        base = base / s
    elif c["rope"] == "yarn":
        ramp = ((c["native"] * base / (2 * math.pi) - 1.0) / 31.0).clamp(0.0, 1.0)
        base = (1.0 - ramp) * base / s + ramp * base
        m = 0.1 * math.log(s) + 1.0
    ang = positions.double()[:, None, None] * base
    cos, sin = ang.cos(), ang.sin()
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * cos - b * sin, b * cos + a * sin], -1) * m


def _attend(scores, keep, v):
    """softmax over the kept keys, and its log-sum-exp: scores [h, rows, keys], v [keys, d]."""
    scores = scores.masked_fill(~keep, float("-inf"))
    lse = torch.logsumexp(scores, -1)
    return torch.matmul(torch.exp(scores - lse[..., None]), v), lse


def _exact_layer(c, seeds, q, k, v):
    n, group = c["n"], c["hq"] // c["hkv"]
    out = torch.empty(n, c["hq"], c["d"], dtype=torch.float64, device="cuda")
    lse = torch.empty(c["hq"], n, dtype=torch.float64, device="cuda")
    step = max(16, min(n, int(2 ** 28 // (n * c["hq"]))))
    for r0 in range(0, n, step):
        r1 = min(n, r0 + step)
        keep = None
        for g in range(c["hkv"]):
            if keep is None or c["per_head"]:
                keep = _mask_rows(c, seeds, r0, r1, r1, g if c["per_head"] else 0)
            hs = slice(g * group, (g + 1) * group)
            sc = torch.matmul(q[r0:r1, hs].transpose(0, 1), k[:r1, g].T) / math.sqrt(c["d"])
            o, l = _attend(sc, keep, v[:r1, g].double())
            out[r0:r1, hs] = o.transpose(0, 1)
            lse[hs, r0:r1] = l
    return out, lse


def exact(case, seed):
    c = case
    if c["kind"] == "mask":
        return None  # whole numbers, compared as they are
    seeds = _mask_seeds(c, seed)
    if c["kind"] in ("step", "token"):
        t, n_ctx = c["n"] + c["generated"] - 1, c["n"] + c["generated"]
        group, outs, keeps = c["hq"] // c["hkv"], [], []
        row = dict(c, window=0)  # row n of the prefill's mask, without its local window
        for g in range(c["hkv"]):
            keep = torch.zeros(n_ctx, dtype=torch.bool, device="cuda")
            keep[:c["n"]] = _mask_rows(row, seeds, c["n"], c["n"] + 1, c["n"], g if c["per_head"] else 0)[0]
            keep[max(0, t - c["decode_window"] + 1):] = True
            keeps.append(keep.nonzero()[:, 0])
        for layer in range(c["layers"]):
            q, k, v = _inputs(c, seed, layer)
            qr = _rotate(c, q, torch.tensor([t], device="cuda"), n_ctx)[0]
            o = torch.empty(c["hq"], c["d"], dtype=torch.float64, device="cuda")
            for g in range(c["hkv"]):
                idx = keeps[g]
                hs = slice(g * group, (g + 1) * group)
                kr = _rotate(c, k[idx, g:g + 1], idx, n_ctx)[:, 0]
                p = torch.softmax(qr[hs] @ kr.T / math.sqrt(c["d"]), -1)
                o[hs] = p @ v[idx, g].double()
            outs.append(o)
        return torch.stack(outs)
    n, sets = c["n"], (c["seeds"] if c["kind"] == "ensemble" else 1)
    if 4.0 * c["d"] * c["hq"] * n * n / 2 * sets > 4e12 or c["seeds"] * float(n) ** 2 > 4e10:
        return None  # too long in 64 bits
    q, k, v = _inputs(c, seed)
    pos = torch.arange(n, device="cuda")
    q, k = _rotate(c, q, pos, n), _rotate(c, k, pos, n)
    if c["kind"] == "ensemble":
        parts = [_exact_layer(c, [s], q, k, v) for s in seeds]
        out, lse = torch.stack([p[0] for p in parts]), torch.stack([p[1] for p in parts])
    else:
        out, lse = _exact_layer(c, seeds, q, k, v)
    return (out, lse) if c["lse"] else out
