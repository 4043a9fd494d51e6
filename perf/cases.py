"""Performance cases of the classify path: what a program that uses this library
has it do, through the public entry points.

A case is one call (the recursive ones: one call that runs k layer passes) of
sp_classify, sp_classify_host, sp_classify_hidden, sp_classify_hidden_host,
sp_attend or sp_project.  Layer shapes are those of the workloads module (the
4B-, 8B- and 27B-class draft heads) or generic ones; values follow its recipe
(weights, soft prompts and rows N(0, 0.02), gains 1 + N(0, 0.02), cached keys
and values N(0, 1), hidden states N(0, 1)), drawn on the GPU from the seed.
Calls go to one side stream, as a monitor beside a decoding loop has it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl

# layer shapes: d_model, query heads, kv heads, head_dim, d_ff
LAYERS = {
    "tiny": (128, 4, 2, 32, 256),
    "0.6b": (1024, 16, 8, 128, 3072),
    "4b": (2560, 32, 8, 128, 9728),
    "8b": (4096, 32, 8, 128, 12288),
    "27b": (5120, 40, 8, 128, 17408),
}


def _case(name, entry, layer, B, lo, hi, k, C=2, page=16, rows=True, T=1, pool="mean",
          lm_head=False, fp32=False):
    """entry: the call; B sequences of lo..hi cached tokens; k soft-prompt rows;
    page: tokens per page, 0 = contiguous caches; rows: per-sequence input rows
    (else the handle's shared soft prompt); T tasks; fp32: weights and caches."""
    c = {"entry": entry, "layer": layer, "B": B, "lo": lo, "hi": hi, "k": k, "C": C, "page": page,
         "rows": rows, "T": T, "pool": pool, "lm_head": lm_head, "fp32": fp32}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the fp32 layer of the tiny configuration, one
        # sequence (launch latency, the CUDA-core kernels)
        _case("tiny_fp32", "classify", "tiny", 1, 64, 64, 4, fp32=True, page=0),
        # one request monitored while it decodes: shared soft prompt, every
        # weight read for four rows
        _case("one_request", "classify", "8b", 1, 2048, 2048, 4, C=16, rows=False),
        # the 4B-class configuration: ragged batch, contiguous caches
        _case("4b_ragged", "classify", "4b", 16, 256, 2048, 8),
        # single-step probing of a decode batch end to end: base hidden states
        # from host memory through the input fusion, logits back to the host
        _case("4b_hidden_host", "hidden_host", "4b", 16, 256, 2048, 8, C=8, lm_head=True),
        # the paper's recursive probing SP-8 over the same batch
        _case("4b_recursive", "recursive", "4b", 16, 256, 2048, 8, C=8, page=0),
        # several classifiers sharing one pass over the cache, last-row pooling
        _case("8b_tasks", "classify", "8b", 24, 700, 3000, 2, C=4, page=32, rows=False, T=4,
              pool="last"),
        # a large moderation batch of short texts, shared soft prompt
        _case("8b_short_batch", "classify", "8b", 128, 384, 640, 4, rows=False),
        # the 8B/9B-class paged configuration
        _case("8b_paged", "classify", "8b", 64, 1024, 8192, 16, C=4),
        # the 27B-class long-context configuration
        _case("27b_long", "classify", "27b", 8, 32768, 32768, 16),
        # the serving sweep's largest batch, bulk classification
        _case("8b_bulk", "classify", "8b", 256, 1536, 2560, 16),
        # the attention step alone, for a caller with its own projections
        # (odd batch and row count, empty to long caches, fp32 output)
        _case("attend_ragged", "attend", "8b", 37, 0, 6000, 5, page=0),
        # the projection step alone, a ragged number of rows
        {"name": "project_300", "entry": "project", "M": 300, "N": 6144, "K": 4096},
    ]


def _cost(case):
    """A rough time of a call, to bound the drawn ones (recursion: k layer passes)."""
    w = work(case)
    return (w["bytes"] / 5e12 + w["flops"] / 1e15) * (case["k"] if case["entry"] == "recursive" else 1)


def draw(rng):
    """One more call of the same ranges: B 1..256, L 0..32768, every entry."""
    most = _cost(listed()[9])
    while True:
        entry = rng.choice(["classify"] * 5 + ["host", "hidden", "hidden_host", "recursive", "attend",
                                               "attend", "project"])
        if entry == "project":
            c = {"entry": entry, "M": int(round(2 ** rng.uniform(0, 11))),
                 "N": 128 * int(round(2 ** rng.uniform(2, 8))), "K": 64 * int(round(2 ** rng.uniform(2, 8)))}
        else:
            layer = rng.choice(["0.6b", "4b", "4b", "8b", "8b", "27b"])
            G = LAYERS[layer][1] // LAYERS[layer][2]
            T = rng.choice([1, 1, 1, 2, 4]) if entry == "classify" else 1
            k = min(int(round(2 ** rng.uniform(0, 5))), 128 // (G * T))
            if entry == "recursive":
                k = min(k, 6)
            B = int(round(2 ** rng.uniform(0, 8)))
            mid = 2 ** rng.uniform(5, 15)
            spread = rng.choice([0.0, 0.25, 0.8])
            c = _case("", entry, layer, B, int(mid * (1 - spread)), min(32768, int(mid * (1 + spread)) + 1),
                      k, C=rng.choice([2, 4, 16]), page=rng.choice([0, 0, 16, 16, 16, 32, 64]),
                      rows=rng.choice([True, False]), T=T, pool=rng.choice(["mean", "mean", "last"]),
                      lm_head=rng.random() < 0.25)
        if _cost(c) <= most:
            return c


# --------------------------------------------------------------------------- #
# inputs
# --------------------------------------------------------------------------- #
_STREAM = None


def _stream():
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    return g


def _normal(g, shape, std, dtype, mean=0.0):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    if std != 1.0:
        x *= std
    if mean:
        x += mean
    return x.to(dtype)


def _draw_weights(case, g):
    d, hq, hkv, dh, f = LAYERS[case["layer"]]
    k, T, C = case["k"], case["T"], case["C"]
    dt = torch.float32 if case["fp32"] else torch.bfloat16
    f32 = torch.float32
    w = {"w_q": _normal(g, (hq * dh, d), 0.02, dt), "w_k": _normal(g, (hkv * dh, d), 0.02, dt),
         "w_v": _normal(g, (hkv * dh, d), 0.02, dt), "w_o": _normal(g, (d, hq * dh), 0.02, dt),
         "w_gate": _normal(g, (f, d), 0.02, dt), "w_up": _normal(g, (f, d), 0.02, dt),
         "w_down": _normal(g, (d, f), 0.02, dt), "g_in": _normal(g, (d,), 0.02, f32, 1.0),
         "g_post": _normal(g, (d,), 0.02, f32, 1.0), "soft_prompt": _normal(g, (T * k, d), 0.02, dt),
         "head_w": _normal(g, (T * C, d), 0.02, f32), "head_b": _normal(g, (T * C,), 0.02, f32)}
    if case["entry"] in ("hidden", "hidden_host", "recursive"):
        w["w_fc"] = _normal(g, (d, 2 * d), 0.02, dt)
        w["g_h"] = _normal(g, (d,), 0.02, f32, 1.0)
        w["g_e"] = _normal(g, (d,), 0.02, f32, 1.0)
    if case["lm_head"]:
        w["g_final"] = _normal(g, (d,), 0.02, f32, 1.0)
        w["head_b"] = None
    return w


def _lengths(case, seed):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, case["B"]])
    return rng.integers(case["lo"], case["hi"], size=case["B"], endpoint=True).astype(np.int32)


def _draw_cache(case, g, lens, seed):
    """Token-major keys and values of all sequences (contiguous), or a pool with
    a random page table.  K and V as [slots][Hkv][dh] or [page][Hkv][P][dh]."""
    _, _, hkv, dh, _ = LAYERS[case["layer"]]
    dt = torch.float32 if case["fp32"] else torch.bfloat16
    P = case["page"]
    if not P:
        shape = (max(int(lens.sum()), 1), hkv, dh)
        table = None
    else:
        pages = (lens.astype(np.int64) + P - 1) // P
        perm = np.random.default_rng([int(seed) & 0x7FFFFFFF, 7]).permutation(int(pages.sum())).astype(np.int32)
        table = np.full((len(lens), max(1, int(pages.max()))), -1, dtype=np.int32)
        at = 0
        for b, n in enumerate(pages):
            table[b, :n] = perm[at:at + n]
            at += n
        shape = (max(at, 1), hkv, P, dh)
    return _normal(g, shape, 1.0, dt), _normal(g, shape, 1.0, dt), table


def _draw_all(case, seed):
    g = _generator(seed)
    if case["entry"] == "project":
        return {"x": _normal(g, (case["M"], case["K"]), 1.0, torch.float32),
                "w": _normal(g, (case["N"], case["K"]), 0.02, torch.bfloat16)}
    d, hq, hkv, dh, _ = LAYERS[case["layer"]]
    B, k, T = case["B"], case["k"], case["T"]
    lens = _lengths(case, seed)
    s = {"lens": lens}
    s["K"], s["V"], s["table"] = _draw_cache(case, g, lens, seed)
    dt = torch.float32 if case["fp32"] else torch.bfloat16
    if case["entry"] == "attend":
        # rotated queries and keys of a projection: standard deviation 0.02 sqrt(d)
        s["q"] = _normal(g, (B, k, hq, dh), 0.02 * math.sqrt(d), torch.float32)
        s["k_new"] = _normal(g, (B, k, hkv, dh), 0.02 * math.sqrt(d), torch.float32)
        s["v_new"] = _normal(g, (B, k, hkv, dh), 0.02 * math.sqrt(d), torch.float32)
        return s
    s["weights"] = _draw_weights(case, g)
    if case["entry"] in ("hidden", "hidden_host", "recursive"):
        s["hidden"] = _normal(g, (B, d), 1.0, dt)
    elif case["rows"]:
        s["rows"] = _normal(g, (B, T * k, d), 0.02, dt)
    return s


def _host(t):
    """A host array in the library's storage form (bf16 as 16-bit patterns)."""
    if t is None:
        return None
    return t.view(torch.int16).cpu().numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.cpu().numpy()


def _descriptor(case, s):
    _, _, hkv, dh, _ = LAYERS[case["layer"]]
    if case["page"]:
        s["table_d"] = torch.from_numpy(s["table"]).cuda()
        return sp.sp_kv_cache(sp.SP_KV_PAGED, None, None, s["K"].data_ptr(), s["V"].data_ptr(),
                              s["table_d"].data_ptr(), case["page"], s["K"].shape[0],
                              s["table"].shape[1], case["B"])
    step = hkv * dh * s["K"].element_size()
    at = (np.cumsum(s["lens"], dtype=np.int64) - s["lens"]) * step
    s["k_ptr"] = torch.from_numpy(s["K"].data_ptr() + at).cuda()
    s["v_ptr"] = torch.from_numpy(s["V"].data_ptr() + at).cuda()
    return sp.sp_kv_cache(sp.SP_KV_CONTIGUOUS, s["k_ptr"].data_ptr(), s["v_ptr"].data_ptr(), None, None,
                          None, 16, 0, 0, case["B"])


def prepare(case, seed):
    s = _draw_all(case, seed)
    s["case"] = case
    entry = case["entry"]
    if entry == "project":
        M, N, K = case["M"], case["N"], case["K"]
        s["y"] = torch.empty((M, N), device="cuda")
        s["ws_bytes"] = sp.sp_project_workspace_bytes(M, N, K)
        s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        return s
    _, hq, hkv, dh, _ = LAYERS[case["layer"]]
    B, k, T, C = case["B"], case["k"], case["T"], case["C"]
    s["lens_d"] = torch.from_numpy(s["lens"]).cuda()
    s["kv"] = _descriptor(case, s)
    max_len = int(case["hi"])
    if entry == "attend":
        s["dims"] = sp.sp_attn_dims(hq, hkv, dh, k, sp.SP_F32 if case["fp32"] else sp.SP_BF16, max_len, 0, 0)
        s["out"] = torch.empty((B, k, hq, dh), device="cuda")
        s["ws_bytes"] = sp.sp_attend_workspace_bytes(s["dims"], B)
        s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        return s
    d, _, _, _, f = LAYERS[case["layer"]]
    dt = wl.F32 if case["fp32"] else wl.BF16
    shape = wl.Shape(d, hq, hkv, dh, f, k, C, w_dtype=dt, kv_dtype=dt,
                     pool=wl.POOL_LAST if case["pool"] == "last" else wl.POOL_MEAN,
                     page_size=case["page"] or 16, n_tasks=T)
    weights = wl.Weights(**{n: _host(t) for n, t in s.pop("weights").items()})
    s["model"] = sp.Model(shape, weights, B, max_len)
    if entry == "recursive":
        sp.sp_set_option(s["model"].handle, sp.SP_OPT_RECURSIVE, 1)
    if entry in ("host", "hidden_host"):
        s["h_lens"] = torch.from_numpy(s["lens"]).pin_memory()
        for n in ("rows", "hidden"):
            if n in s:
                s["h_" + n] = s.pop(n).cpu().pin_memory()
        s["logits"] = torch.empty((B, T, C)).pin_memory()
    else:
        s["logits"] = torch.empty((B, T, C), device="cuda")
    torch.cuda.synchronize()
    return s


# --------------------------------------------------------------------------- #
# one pass
# --------------------------------------------------------------------------- #
def run(s):
    case, st = s["case"], _stream()
    entry = case["entry"]
    if entry == "project":
        sp.sp_project(st, case["M"], case["N"], case["K"], s["x"], s["w"], s["y"], 0, s["ws"], s["ws_bytes"])
        return s["y"]
    if entry == "attend":
        sp.sp_attend(st, s["dims"], case["B"], None, s["lens_d"], s["kv"], s["q"], s["k_new"], s["v_new"],
                     s["out"], sp.SP_F32, s["ws"], s["ws_bytes"])
        return s["out"]
    h = s["model"].handle
    if entry == "classify":
        sp.sp_classify(h, st, case["B"], None, s["lens_d"], s["kv"], s.get("rows"), s["logits"])
    elif entry == "host":
        sp.sp_classify_host(h, st, case["B"], None, s["h_lens"], s["kv"], s.get("h_rows"), s["logits"])
    elif entry == "hidden_host":
        sp.sp_classify_hidden_host(h, st, case["B"], None, s["h_lens"], s["kv"], s["h_hidden"], s["logits"])
    else:
        sp.sp_classify_hidden(h, st, case["B"], None, s["lens_d"], s["kv"], s["hidden"], s["logits"])
    return s["logits"]


def work(case):
    """Each input read once and each output written once; the soft prompt's own
    projections are part of the handle, so a call that uses it skips Q/K/V."""
    if case["entry"] == "project":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4.0 * M * K + 2.0 * N * K + 4.0 * M * N, "flops": 2.0 * M * N * K}
    d, hq, hkv, dh, f = LAYERS[case["layer"]]
    B, k, T, C = case["B"], case["k"], case["T"], case["C"]
    es = 4 if case["fp32"] else 2
    tokens = B * (case["lo"] + case["hi"]) / 2.0
    rows = B * k * T
    kv = 2.0 * es * tokens * hkv * dh
    attn = 4.0 * dh * hq * k * T * tokens
    if case["entry"] == "attend":
        return {"bytes": kv + 4.0 * rows * dh * (2 * hq + 2 * hkv), "flops": attn}
    mats = d * hq * dh + 3 * d * f
    fused = case["entry"] in ("hidden", "hidden_host", "recursive")
    if fused or case["rows"]:
        mats += d * (hq + 2 * hkv) * dh
    flops = 2.0 * rows * mats
    if fused:
        mats += d * d
        flops += 2.0 * (rows if case["entry"] == "recursive" else B) * d * d
    inputs = es * d * (B if fused else rows if case["rows"] else T * k)
    return {"bytes": kv + es * mats + inputs + 4.0 * T * C * (d + B),
            "flops": flops + attn + 2.0 * B * T * C * d}


def tolerance(case):
    """About four times the largest distance from exact() measured over the listed
    and 40 drawn cases: 1e-5 (projection: 16-bit mantissa inputs, fp32 sums over
    up to 16384 terms), 1e-7 (fp32 layer), 2e-3 (attention alone: bf16 probabilities and new
    keys), 3e-3 (the layer with hi + lo projection inputs) and 4e-3 (plain bf16
    MLP inputs, from 8 mean-pooled rows on); the logits of one call can be few."""
    if case["entry"] == "project":
        return {"rel": 4e-5}
    if case["fp32"]:
        return {"rel": 2e-6}
    if case["entry"] == "attend":
        return {"rel": 8e-3, "max": 0.1}
    return {"rel": 1.6e-2 if case["pool"] == "mean" and case["k"] >= 8 else 1.2e-2, "max": 0.1}


# --------------------------------------------------------------------------- #
# the same in 64 bits
# --------------------------------------------------------------------------- #
def _norm(x, gain, eps=1e-6):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * gain


def _rotate(x, pos):
    """Rotate-half form, theta 1e4; x [rows][heads][dh] at positions pos [rows]."""
    half = x.shape[-1] // 2
    freq = 1.0e4 ** (-2.0 * torch.arange(half, dtype=torch.float64, device=x.device) / x.shape[-1])
    ang = pos.to(torch.float64)[:, None, None] * freq
    c, sn = torch.cos(ang), torch.sin(ang)
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * sn, b * c + a * sn], dim=-1)


def _cached(case, s, b):
    L = int(s["lens"][b])
    if case["page"]:
        n = -(-L // case["page"])
        at = torch.from_numpy(s["table"][b, :n].astype(np.int64)).cuda()
        pick = lambda t: t[at].transpose(1, 2).reshape(-1, t.shape[1], t.shape[3])[:L]  # noqa: E731
    else:
        o = int(s["lens"][:b].sum())
        pick = lambda t: t[o:o + L]  # noqa: E731
    return pick(s["K"]).double(), pick(s["V"]).double()


def _attention(case, s, b, q, kn, vn, sees):
    """q [rows][Hq][dh] over the cache of sequence b and the new keys that
    sees [rows][new] allows."""
    _, hq, hkv, dh, _ = LAYERS[case["layer"]]
    K, V = _cached(case, s, b)
    L, rows = K.shape[0], q.shape[0]
    K, V = torch.cat([K, kn]), torch.cat([V, vn])
    qg = q.view(rows, hkv, hq // hkv, dh).permute(1, 2, 0, 3).reshape(hkv, -1, dh)
    sc = torch.matmul(qg, K.permute(1, 2, 0)) / math.sqrt(dh)
    mask = torch.cat([torch.ones((rows, L), dtype=torch.bool, device=q.device), sees], dim=1)
    sc = sc.view(hkv, hq // hkv, rows, -1).masked_fill(~mask, -math.inf)
    p = torch.softmax(sc, dim=-1).view(hkv, -1, L + kn.shape[0])
    o = torch.matmul(p, V.permute(1, 0, 2)).view(hkv, hq // hkv, rows, dh)
    return o.permute(2, 0, 1, 3).reshape(rows, hq * dh)


def _after_attention(w, x, o):
    h1 = x + o @ w["w_o"].T
    n = _norm(h1, w["g_post"])
    return h1 + (torch.nn.functional.silu(n @ w["w_gate"].T) * (n @ w["w_up"].T)) @ w["w_down"].T


def _qkv(case, w, x, pos):
    _, hq, hkv, dh, _ = LAYERS[case["layer"]]
    xn = _norm(x, w["g_in"])
    return (_rotate((xn @ w["w_q"].T).view(-1, hq, dh), pos),
            _rotate((xn @ w["w_k"].T).view(-1, hkv, dh), pos), (xn @ w["w_v"].T).view(-1, hkv, dh))


def exact(case, seed):
    s = _draw_all(case, seed)
    if case["entry"] == "project":
        return s["x"].double() @ s["w"].double().T
    d, hq, hkv, dh, _ = LAYERS[case["layer"]]
    B, k, T, C = case["B"], case["k"], case["T"], case["C"]
    causal = torch.ones((k, k), dtype=torch.bool, device="cuda").tril()
    if case["entry"] == "attend":
        q, kn, vn = (s[n].double() for n in ("q", "k_new", "v_new"))
        return torch.stack([_attention(case, s, b, q[b], kn[b], vn[b], causal) for b in range(B)]
                           ).view(B, k, hq, dh)
    w = {n: None if t is None else t.double() for n, t in s["weights"].items()}
    R = T * k
    lens = torch.from_numpy(s["lens"].astype(np.int64)).cuda()
    prompt = w["soft_prompt"]
    if case["entry"] == "recursive":
        prev, outs = s["hidden"].double(), []
        kn = torch.zeros((B, k, hkv, dh), dtype=torch.float64, device="cuda")
        vn = torch.zeros_like(kn)
        for i in range(k):
            e = _norm(prompt[i], w["g_e"]).expand(B, d)
            x = torch.cat([_norm(prev, w["g_h"]), e], dim=1) @ w["w_fc"].T
            q, kn[:, i], vn[:, i] = _qkv(case, w, x, lens + i)
            o = torch.cat([_attention(case, s, b, q[b:b + 1], kn[b], vn[b], causal[i:i + 1]) for b in range(B)])
            prev = _after_attention(w, x, o)
            outs.append(prev)
        h2 = torch.stack(outs, dim=1)
    else:
        if case["entry"] in ("hidden", "hidden_host"):
            hn = _norm(s["hidden"].double(), w["g_h"])[:, None].expand(B, R, d)
            e = _norm(prompt, w["g_e"])[None].expand(B, R, d)
            x = (torch.cat([hn, e], dim=2) @ w["w_fc"].T).reshape(B * R, d)
        elif case["rows"]:
            x = s["rows"].double().reshape(B * R, d)
        else:
            x = prompt[None].expand(B, R, d).reshape(B * R, d)
        pos = (lens[:, None] + (torch.arange(R, device="cuda") % k)[None]).reshape(-1)
        q, kn, vn = (t.view(B, R, -1, dh) for t in _qkv(case, w, x, pos))
        sees = torch.block_diag(*[causal] * T)
        o = torch.cat([_attention(case, s, b, q[b], kn[b], vn[b], sees) for b in range(B)])
        h2 = torch.cat([_after_attention(w, x[i:i + 512], o[i:i + 512]) for i in range(0, B * R, 512)])
    h2 = h2.view(B, T, k, d)
    p = h2[:, :, -1] if case["pool"] == "last" else h2.mean(2)
    if w.get("g_final") is not None:
        p = _norm(p, w["g_final"])
    z = torch.einsum("btd,tcd->btc", p, w["head_w"].view(T, C, d))
    return z if w["head_b"] is None else z + w["head_b"].view(T, C)
