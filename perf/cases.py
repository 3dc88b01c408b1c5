"""What a user of the framework has it do, as timed cases.

Three kinds of call, each through the package's public entry points:

* ``compress``: one post-prefill compression of a request's KV cache
  (gracekv.Compressor on device tensors, or gracekv_compress_host on pinned
  host tensors); the outputs are the whole packed cache, the slots and the
  curvature.
* ``decode``: one decoding step on a packed cache (gracekv.Decoder), either
  one attention launch over every layer or append + attention layer by layer,
  the way a model runs.
* ``sensitivity``: the per-(layer, KV head) sensitivity from the output
  projections (gracekv.gracekv_head_sensitivity).

Inputs follow the recipe of synth.py (piecewise segments whose means follow an
AR(1) walk, outlier channels, RoPE-rotated keys, N(0, 1) queries), drawn on
the GPU in fp32 so that a whole 128K-token cache takes well under a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_07001_gb300 import gracekv as gk
from paper_2608_07001_gb300 import synth

DEV = "cuda"
TDT = {"bf16": torch.bfloat16, "f32": torch.float32}


def _compress(name, L, G, Hq, d, T, W, ratio, *, dtype="bf16", base=5.0e5, outliers=3, scale=10.0,
              prefix=0, suffix=0, alpha=0.0, lam=0.0, omega=False, surprisal=False, skew=False, host=False):
    c = dict(kind="compress", L=L, G=G, Hq=Hq, d=d, T=T, W=W, ratio=ratio, dtype=dtype, base=base,
             outliers=outliers, scale=scale, prefix=prefix, suffix=suffix, alpha=alpha, lam=lam,
             omega=omega, surprisal=surprisal, skew=skew, host=host)
    return dict(c, name=name) if name else c


def _decode(name, L, G, Hq, d, rows, n_app, *, dtype="bf16", by_layer=False):
    c = dict(kind="decode", L=L, G=G, Hq=Hq, d=d, rows=rows, n_app=n_app, dtype=dtype, by_layer=by_layer)
    return dict(c, name=name) if name else c


def _sensitivity(name, L, G, Hq, d, D, U):
    c = dict(kind="sensitivity", L=L, G=G, Hq=Hq, d=d, D=D, U=U)
    return dict(c, name=name) if name else c


def listed():
    return [
        # One layer of a short fp32 request: launches, host waits and latency are all of it.
        _compress("pr1_f32_8x", 1, 2, 2, 128, 1024, 32, 8, dtype="f32", base=1.0e4, outliers=4, scale=8.0),
        # A small model's chat-length request, mild compression: most trees are built deep.
        _compress("small_8x", 16, 8, 32, 64, 8192, 64, 8, base=1.0e4, outliers=4, scale=8.0),
        # The same model from an offloading engine: inputs and cache in pinned host memory.
        _compress("small_host_16x", 16, 8, 32, 64, 8192, 64, 16, base=1.0e4, outliers=4, scale=8.0, host=True),
        # Every option at once on a ragged length: system prompt and suffix kept, singleton floor,
        # multi-hop relevance, head sensitivity, surprisal.
        _compress("options_16x", 8, 4, 16, 128, 12347, 48, 16, prefix=19, suffix=7, alpha=0.6, lam=0.3,
                  omega=True, surprisal=True),
        # An 8B-shaped model's document-length request.
        _compress("llama32k_32x", 32, 8, 32, 128, 32768, 64, 32),
        # The long-context request the method is made for, at its two budgets.
        _compress("llama128k_32x", 32, 8, 32, 128, 131072, 64, 32),
        _compress("llama128k_128x", 32, 8, 32, 128, 131072, 64, 128),
        # A caller's own partition with single-token and multi-thousand-token slots, and
        # queries that look at three regions only.
        _compress("skew64k_32x", 32, 8, 32, 128, 65536, 64, 32, skew=True),
        # One decoding step over all layers of a 128K-token cache packed 32x (4096 rows a head).
        _decode("decode_128k_32x", 32, 8, 32, 128, 4096, 65),
        # One decoding step as a model takes it, layer by layer, on a 32K-token cache packed 32x.
        _decode("decode_layers_32k_32x", 32, 8, 32, 128, 1024, 64, by_layer=True),
        # The smallest call: one fp32 layer's attention over a few hundred rows.
        _decode("decode_f32_small", 1, 2, 2, 128, 160, 3, dtype="f32"),
        # Once per model load: the output projections of an 8B-shaped model.
        _sensitivity("sensitivity_8b", 32, 8, 32, 128, 4096, 32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    G = rng.choice([1, 2, 4, 8])
    gq = rng.choice([1, 2, 4, 4, 8])
    d = rng.choice([64, 128, 128])
    if u < 0.2:
        L = _log_int(rng, 1, 32)
        f32 = rng.random() < 0.3
        rows = _log_int(rng, 64, 4096)
        return _decode("", L, G, G * gq, d, max(64, min(rows, 600_000 // (L * G))) if f32 else rows,
                       rng.randint(0, 128), dtype="f32" if f32 else "bf16", by_layer=rng.random() < 0.5)
    if u < 0.3:
        return _sensitivity("", _log_int(rng, 1, 32), G, G * gq, d, 8 * _log_int(rng, 32, 512), rng.randint(1, 64))
    # a compression: token-heads (L G T) bounded so that no drawn one costs more than the largest
    # listed; a mild ratio builds its trees deeper, so it gets fewer
    f32 = rng.random() < 0.15
    host = not f32 and rng.random() < 0.1
    skew = not f32 and not host and rng.random() < 0.15
    ratio = rng.choice([4, 8, 12, 16, 32, 32, 64, 100, 128])
    lo = max(600, 64 * ratio, 6000 if skew else 0)
    T = _log_int(rng, lo, max(lo + 1, 4096 if f32 else 131072))
    cap = 600_000 if f32 else 2_000_000 if host else (16_000_000 if skew else 33_000_000) * min(1.0, ratio / 40)
    L = max(1, min(_log_int(rng, 1, 32), int(cap / (G * T))))
    T = min(T, int(cap / (G * L)))
    opts = not f32 and not host and not skew and rng.random() < 0.25
    return _compress("", L, G, G * gq, d, T, rng.choice([32, 64, 64, rng.randint(8, 64)]), ratio,
                     dtype="f32" if f32 else "bf16", base=rng.choice([1.0e4, 5.0e5]),
                     outliers=rng.choice([3, 4]), scale=rng.choice([8.0, 10.0]),
                     prefix=rng.randint(0, 40) if opts else 0, suffix=rng.randint(0, 20) if opts else 0,
                     alpha=rng.choice([0.0, 0.6]) if opts else 0.0, lam=rng.choice([0.0, 0.3]) if opts else 0.0,
                     omega=opts, surprisal=opts and rng.random() < 0.5, skew=skew, host=host)


# ---- inputs -----------------------------------------------------------------

def _segments(rng, T):
    """Segment id of every token: lognormal(ln 200, 0.5) lengths, clamped to [16, 2000]."""
    n = np.clip(np.rint(rng.lognormal(math.log(200.0), 0.5, size=T // 16 + 2)), 16, 2000).astype(np.int64)
    return torch.as_tensor(np.repeat(np.arange(len(n)), n)[:T], device=DEV)


def _walk(gen, n_seg, *shape):
    """Stationary AR(1) segment means [n_seg, *shape]."""
    xi = torch.randn(n_seg, *shape, generator=gen, device=DEV)
    for s in range(1, n_seg):
        xi[s] = 0.8 * xi[s - 1] + 0.6 * xi[s]
    return xi


def _rotate(x, cos, sin):
    h = x.shape[-1] // 2
    a, b = x[..., :h], x[..., h:]
    return torch.cat([a * cos - b * sin, a * sin + b * cos], dim=-1)


def _angles(T, d, base):
    inv = torch.pow(torch.tensor(base, dtype=torch.float64, device=DEV),
                    -2.0 * torch.arange(d // 2, dtype=torch.float64, device=DEV) / d)
    ang = torch.arange(T, dtype=torch.float64, device=DEV)[:, None] * inv
    return torch.cos(ang).float(), torch.sin(ang).float()


def _slots(rng, N):
    """A caller's partition: a long slot (4097..8192 tokens) per 8192 tokens of context, 1% of
    the others a single token, the rest U{16..128}."""
    lens, left = [], N
    n_long = max(1, N // 8192 - 1)
    for _ in range(n_long):
        n = int(rng.integers(4097, 8193))
        if left - n < N // 4:
            break
        lens.append(n)
        left -= n
    while left > 0:
        n = min(left, 1 if rng.random() < 0.01 else int(rng.integers(16, 129)))
        lens.append(n)
        left -= n
    rng.shuffle(lens)
    return torch.as_tensor(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32), device=DEV)


def _cache_inputs(c, seed):
    """K, V [L, G, T, d] and Q [L, Hq, W, d] on the GPU."""
    L, G, Hq, T, d, W = c["L"], c["G"], c["Hq"], c["T"], c["d"], c["W"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    tdt = TDT[c["dtype"]]
    seg = _segments(rng, T)
    mu = _walk(gen, int(seg[-1]) + 1, 2, L, G, d)
    gain = torch.ones(2, L, G, d, device=DEV)
    gain.scatter_(3, torch.rand(2, L, G, d, generator=gen, device=DEV).topk(c["outliers"], dim=3).indices, c["scale"])
    gain /= math.sqrt(2.0)
    cos, sin = _angles(T, d, c["base"])
    K = torch.empty(L, G, T, d, dtype=tdt, device=DEV)
    V = torch.empty_like(K)
    Q = torch.randn(L, Hq, W, d, generator=gen, device=DEV)
    for l in range(L):
        for g in range(G):
            for k, out in enumerate((K, V)):
                x = torch.randn(T, d, generator=gen, device=DEV).add_(mu[:, k, l, g][seg]).mul_(gain[k, l, g])
                out[l, g] = (x if k else _rotate(x, cos, sin)).to(tdt)
    if c["skew"]:   # three 512-token regions whose keys the queries point at
        at = np.sort(rng.integers(0, T - 32 - 3 * 512 + 1, size=3)) + 512 * np.arange(3)
        dirs = torch.nn.functional.normalize(torch.randn(L, G, 3, d, generator=gen, device=DEV), dim=-1)
        for r, a in enumerate(at):
            e = torch.nn.functional.normalize(torch.randn(L, G, 512, d, generator=gen, device=DEV), dim=-1)
            K[:, :, a:a + 512] = (math.sqrt(d) * (0.95 * dirs[:, :, r, None] + 0.312 * e)).to(tdt)
        aim = dirs.repeat_interleave(Hq // G, dim=1)[:, :, torch.arange(W, device=DEV) % 3]
        Q = math.sqrt(d) * (0.95 * aim + 0.312 * torch.nn.functional.normalize(Q, dim=-1))
    return K, V, Q.to(tdt), rng, gen


def _prepare_compress(c, seed):
    K, V, Q, rng, gen = _cache_inputs(c, seed)
    L, G, T, d = K.shape
    p = gk.make_params(L, G, c["Hq"], T, d, c["W"], dtype=K.dtype, rope_base=c["base"],
                       budget=gk.gracekv_budget_for_ratio(L, G, T - c["prefix"] - c["suffix"], c["ratio"]),
                       ctx_start=c["prefix"], ctx_end=T - c["suffix"], alpha_floor=c["alpha"], lambda_graph=c["lam"])
    if c["host"]:
        ctx = gk.Context(p)
        K, V, Q = (t.cpu().pin_memory() for t in (K, V, Q))
        return dict(c=c, ctx=ctx, K=K, V=V, Q=Q, cache=gk.Cache.empty_host(p.budget + 8, d, L * G, K.dtype))
    comp = gk.Compressor(p)
    comp.slots.fill_(-1)   # its tail past the last slot stays as it is here
    more = {}
    if c["omega"]:
        more["omega"] = torch.rand(L, G, generator=gen, device=DEV) + 0.5
    if c["surprisal"]:
        more["surprisal"] = -torch.log(torch.rand(T, generator=gen, device=DEV).clamp_min(1e-6))
    if c["lam"] > 0:   # queries of every position at the graph layers, rotated like the keys
        cos, sin = _angles(T, d, c["base"])
        layers = gk.graph_layers(L)
        more["Qg"] = torch.empty(len(layers), c["Hq"], T, d, dtype=K.dtype, device=DEV)
        for i in range(len(layers)):
            more["Qg"][i] = _rotate(torch.randn(c["Hq"], T, d, generator=gen, device=DEV), cos, sin).to(K.dtype)
    if c["skew"]:
        more["slot_starts"] = _slots(rng, comp.ctx.n_c)
    return dict(c=c, comp=comp, K=K, V=V, Q=Q, more=more)


def _prepare_decode(c, seed):
    w = synth.Workload("decode", c["L"], c["G"], c["Hq"], c["d"], c["rows"], 64, c["dtype"], "lognormal", 3, 10.0,
                       5.0e5, (1,), seed)
    x = synth.make_decode_cache(w, 1, n_app=c["n_app"], app_cap=c["n_app"] + 1, device=DEV, seed=seed)
    dec = gk.Decoder(x.K, x.V, x.log_m, x.offsets, L=w.L, G=w.G, Hq=w.Hq, app_cap=c["n_app"] + 1)
    dec.K_app.copy_(x.K_app)
    dec.V_app.copy_(x.V_app)
    dec.n_app = c["n_app"]
    # the new token's row of every (l, g) is the last one drawn
    return dict(c=c, dec=dec, x=x, k_new=x.K_app[:, :, -1].contiguous(), v_new=x.V_app[:, :, -1].contiguous(),
                out=torch.empty(w.L, w.Hq, w.d, device=DEV))


def _prepare_sensitivity(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    W = torch.empty(c["L"], c["D"], c["Hq"] * c["d"], dtype=torch.bfloat16, device=DEV)
    for l in range(c["L"]):
        W[l] = torch.randn(c["D"], c["Hq"] * c["d"], generator=gen, device=DEV) / c["d"] ** 0.5
    o = torch.randn(c["L"], c["Hq"], c["U"], c["d"], generator=gen, device=DEV).to(torch.bfloat16)
    return dict(c=c, W=W, o=o)


def prepare(case, seed):
    return {"compress": _prepare_compress, "decode": _prepare_decode,
            "sensitivity": _prepare_sensitivity}[case["kind"]](case, int(seed))


# ---- one pass ---------------------------------------------------------------

def _cache_dict(cache, E):
    return dict(K=cache.K[:E], V=cache.V[:E], pos=cache.pos[:E], log_m=cache.log_m[:E],
                src_lo=cache.src_lo[:E], src_hi=cache.src_hi[:E], offsets=cache.offsets)


def run(s):
    c = s["c"]
    if c["kind"] == "sensitivity":
        return gk.gracekv_head_sensitivity(s["W"], s["o"], c["G"])
    if c["kind"] == "decode":
        dec, x, out = s["dec"], s["x"], s["out"]
        if not c["by_layer"]:
            dec.n_app = c["n_app"]
            return dec.attention(x.q, out=out)
        for l in range(c["L"]):
            dec.n_app = c["n_app"]
            dec.append(s["k_new"][l:l + 1], s["v_new"][l:l + 1], l0=l)
            dec.n_app = c["n_app"] + 1
            dec.attention(x.q[l:l + 1], l0=l, out=out[l:l + 1])
        return dict(out=out, k_row=dec.K_app[:, :, c["n_app"]], v_row=dec.V_app[:, :, c["n_app"]])
    if c["host"]:
        E = s["ctx"].gracekv_compress_host(s["K"], s["V"], s["Q"], s["cache"])
        return _cache_dict(s["cache"], E)
    comp = s["comp"]
    cache = comp(s["K"], s["V"], s["Q"], **s["more"])
    return dict(_cache_dict(cache, comp.n_entries), slots=comp.slots, kappa=comp.kappa)


def work(case):
    """The bytes and operations no implementation can leave out: for a
    compression, K and V read once, the cache written once, the query x key
    contraction, and every slot's probe statistics from both ends (2 x 2 W d
    per token and KV head); the candidates' distortions come on top of that
    and depend on the data."""
    c = case
    L, G, Hq, d = c["L"], c["G"], c["Hq"], c["d"]
    if c["kind"] == "sensitivity":
        return dict(bytes=2 * L * Hq * d * (c["D"] + c["U"]) + 4 * L * G, flops=2 * L * c["D"] * Hq * d * c["U"])
    es = 2 if c["dtype"] == "bf16" else 4
    if c["kind"] == "decode":
        n = c["n_app"] + int(c["by_layer"])
        rows = L * G * (c["rows"] + n)
        return dict(bytes=rows * 2 * d * es + L * G * c["rows"] * 4 + (L * G + 1) * 8 + L * Hq * d * (es + 4)
                    + (4 * L * G * d * es if c["by_layer"] else 0), flops=4 * rows * d * (Hq // G))
    T, W = c["T"], c["W"]
    E = L * G * ((T - c["prefix"] - c["suffix"]) // c["ratio"] + c["prefix"] + c["suffix"])
    n_graph = len(gk.graph_layers(L)) if c["lam"] > 0 else 0
    return dict(bytes=L * G * T * 2 * d * es + L * Hq * W * d * es + E * (2 * d * es + 16) + (4 * T if c["surprisal"] else 0)
                + n_graph * Hq * 64 * d * es,
                flops=2 * L * Hq * W * T * d + 4 * L * G * T * W * d + n_graph * 2 * 2 * Hq * 64 * T * d)


# ---- the same values in 64 bits -----------------------------------------------

def _exact_decode(c, s):
    x, L, G, d = s["x"], c["L"], c["G"], c["d"]
    gq = c["Hq"] // G
    n = c["n_app"] + int(c["by_layer"])
    off = x.offsets.tolist()
    out = torch.empty(L, c["Hq"], d, dtype=torch.float64, device=DEV)
    for l in range(L):
        for g in range(G):
            a, b = off[l * G + g], off[l * G + g + 1]
            K = torch.cat([x.K[a:b], x.K_app[l, g, :n]]).double()
            V = torch.cat([x.V[a:b], x.V_app[l, g, :n]]).double()
            bias = torch.cat([x.log_m[a:b].double(), torch.zeros(n, dtype=torch.float64, device=DEV)])
            q = x.q[l, g * gq:(g + 1) * gq].double()
            out[l, g * gq:(g + 1) * gq] = torch.softmax(q @ K.T / math.sqrt(d) + bias, dim=-1) @ V
    return dict(out=out, k_row=s["k_new"].double(), v_row=s["v_new"].double()) if c["by_layer"] else out


def _exact_sensitivity(c, s):
    L, G, d = c["L"], c["G"], c["d"]
    n = c["Hq"] // G * d
    raw = torch.empty(L, G, dtype=torch.float64, device=DEV)
    for l in range(L):
        for g in range(G):
            W = s["W"][l, :, g * n:(g + 1) * n].double()
            X = s["o"][l, g * (n // d):(g + 1) * (n // d)].double().transpose(0, 1).reshape(c["U"], n)
            raw[l, g] = torch.sqrt(W.norm() * (W @ X.T).norm(dim=0).mean())
    return raw / (raw.mean() + 1e-6)


def _exact_kappa(c, V):
    """The stabilised curvature of the trajectory of the segmentation layers' values."""
    L, G, T, d = V.shape
    layers = sorted({min(int(math.floor(r * L)), L - 1) for r in (0.33, 0.50, 0.67)})
    ks = []
    for l in layers:
        h = V[l].transpose(0, 1).reshape(T, G * d).double()
        h = h / h.norm(dim=1, keepdim=True).clamp_min(1e-6)
        for w in (4, 8, 16):
            k = torch.zeros(T, dtype=torch.float64, device=DEV)
            if T > 2 * w:
                mid = slice(w, T - w)
                hi = h[mid]
                before = sum(h[w - t:T - w - t] for t in range(w)) / w
                after = sum(h[w + t:T - w + t] for t in range(1, w + 1)) / w
                dm, dp = hi - before, after - hi
                k[mid] = 1.0 - (dm * dp).sum(1) / (dm.norm(dim=1).clamp_min(1e-6) * dp.norm(dim=1).clamp_min(1e-6))
            ks.append(k)
    ks = torch.stack(ks)
    return ks.mean(0) - 0.25 * ks.std(0, unbiased=False)


def exact(case, seed):
    """Decoding, sensitivity and the curvature have a closed form; the packed
    prototypes follow from the selection, whose whole numbers stay equal."""
    c = case
    if c["kind"] == "decode":
        return _exact_decode(c, _prepare_decode(c, int(seed)))
    if c["kind"] == "sensitivity":
        return _exact_sensitivity(c, _prepare_sensitivity(c, int(seed)))
    if c["host"]:
        return None
    V = _cache_inputs(c, int(seed))[1]
    return dict(K=None, V=None, pos=None, log_m=None, src_lo=None, src_hi=None, offsets=None, slots=None,
                kappa=_exact_kappa(c, V))
