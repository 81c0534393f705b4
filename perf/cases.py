"""The calls that a user of the library makes, at the sizes where they are made: eviction of a layer's cache after
prefill (from Q, K, V or from the prefill's own attention statistics), eviction again while decoding, and decode steps
over full and compacted caches.

The attention geometry is that of the repository's workloads (32 query heads over 8 KV heads, head_dim 128, window 32,
bf16; the tiny fp32 workload has 8 over 2 heads of 64).  A case is a dict of plain values:

  call        "evict" | "evict_from_lse" | "decode"
  batch, n    sequences, and scored prefix rows of each (for "decode": rows of the cache)
  tail        0, or 32: K and V also carry the window tokens' own rows (always kept)
  budget      rows kept per head
  width       pooling width (the fixed kernel; in the adaptive window its base width)
  window      "fixed" | "adaptive" (Eq. 10-12)
  d_model     0, or the model width: the norm of Eq. 7 is taken behind an output projection of this width
  dtype       "bf16" | "f32"
"""
import math

import numpy as np
import torch

from paper_2605_08840_b200 import binding as rk

WINDOW = 32
DECAY = 0.9
BETA = 2000.0
DEVICE = "cuda"


def _case(call, batch, n, tail=0, budget=0, width=7, window="fixed", d_model=0, dtype="bf16", name=None):
    c = {"call": call, "batch": batch, "n": n, "tail": tail, "budget": budget, "width": width, "window": window,
         "d_model": d_model, "dtype": dtype}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one decode step over a compacted cache that has grown by some tokens: the call made most often of all, once
        # per layer and generated token, and the smallest
        _case("decode", 1, 2085, name="decode_compacted"),
        # the same for a batch of sequences
        _case("decode", 8, 2176, name="decode_compacted_batch"),
        # one decode step over a cache that was not evicted
        _case("decode", 1, 131072, name="decode_full"),
        # the tiny single-precision workload
        _case("evict", 1, 1024, 0, 128, 7, dtype="f32", name="evict_f32_tiny"),
        # a short prompt, window tokens in the cache
        _case("evict", 1, 3000, 32, 1024, 5, name="evict_short_prompt"),
        # the 8B-shaped layer
        _case("evict", 1, 16384, 0, 1024, 7, name="evict_16k"),
        # the long context that the benchmark is quoted on
        _case("evict", 1, 131072, 0, 2048, 7, name="evict_128k"),
        # a batch of sequences
        _case("evict", 8, 32768, 0, 2048, 7, name="evict_32k_batch"),
        # eviction again during decoding: budget + 128 rows back to the budget, the statistics known from the decode steps
        _case("evict_from_lse", 1, 2144, 32, 2048, 7, name="reevict"),
        # a prompt whose prefill has left the window rows' outputs and normalisers, of a length that fits nothing
        _case("evict_from_lse", 1, 50021, 32, 2048, 7, name="evict_from_prefill_50021"),
        # the adaptive window
        _case("evict", 1, 20011, 32, 1024, 5, window="adaptive", name="evict_adaptive_20011"),
        # the norm of Eq. 7 as printed, behind the layer's output projection
        _case("evict", 1, 32768, 0, 2048, 7, d_model=4096, name="evict_projected_32k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "evict", "evict", "evict", "from_lse", "from_lse", "adaptive", "projected", "f32"])
    if kind == "decode":
        batch = rng.choice([1, 1, 2, 4, 8])
        return _case("decode", batch, _log(rng, 1024, 131072 // batch))
    tail, width = rng.choice([0, WINDOW]), rng.choice([5, 7])
    if kind == "f32":
        n = _log(rng, 512, 4096)
        return _case("evict", 1, n, tail, tail + min(rng.randint(64, 512), n // 3), width, dtype="f32")
    batch = rng.choice([1, 1, 1, 2, 4, 8]) if kind in ("evict", "from_lse") else 1
    longest = min(131072, 262144 // batch) if kind in ("evict", "from_lse") else 32768
    n = _log(rng, 2048, longest)
    budget = tail + min(rng.choice([256, 512, 1024, 2048]), n // 2)
    if kind == "from_lse":
        return _case("evict_from_lse", batch, n, tail, budget, width)
    return _case("evict", batch, n, tail, budget, width, window="adaptive" if kind == "adaptive" else "fixed",
                 d_model=4096 if kind == "projected" else 0)


def _geometry(case):
    """(query heads, KV heads, head_dim, element type)"""
    return (8, 2, 64, torch.float32) if case["dtype"] == "f32" else (32, 8, 128, torch.bfloat16)


def _spans(rng, n, salient):
    """A mask of `salient` of n rows in spans of some dozens of rows, the first of them at row 0, that lie apart."""
    rest = n - salient
    count = max(1, min(salient // 24, rest // 16))
    lengths = 16 + rng.multinomial(salient - 16 * count, np.full(count, 1.0 / count))
    gaps = 12 + rng.multinomial(rest - 12 * count, np.full(count, 1.0 / count))
    return np.repeat(np.tile([True, False], count), np.stack([lengths, gaps], 1).reshape(-1))


def _inputs(case, seed):
    """Q [b, Hq, w, d] and K, V [b, Hkv, n + tail, d] as a prompt leaves them: Gaussian rows, a few passages (as many rows
    as the budget keeps) whose keys the window queries lean on, and a first row that draws a fifth of the attention
    through an outlier channel, as the first token of a prompt does.  The rows of V are
    Gaussian directions of one length, so that the passages' scores stay well apart from the rest."""
    Hq, Hkv, d, dtype = _geometry(case)
    b, n, tail = case["batch"], case["n"], case["tail"]
    g = torch.Generator(DEVICE).manual_seed(seed)
    rng = np.random.RandomState(seed % (1 << 32))

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=DEVICE)

    salient = case["budget"] - tail
    s = randn(b, Hkv, 1, d)
    s[..., 0] = 0
    s *= math.sqrt(d) / s.norm(dim=-1, keepdim=True)
    q = randn(b, Hq, WINDOW, d) + (4.0 / math.sqrt(d)) * s.repeat_interleave(Hq // Hkv, dim=1)
    q[..., 0] = 8.0
    mask = torch.from_numpy(np.stack([_spans(rng, n, salient) for _ in range(b * Hkv)])).to(DEVICE).view(b, Hkv, n, 1)
    K = torch.empty(b, Hkv, n + tail, d, dtype=dtype, device=DEVICE)
    V = torch.empty_like(K)
    sink = (math.log(0.25 * (1.65 * n + 20.0 * salient)) * math.sqrt(d) / 8.0)
    for i in range(b):      # one sequence at a time: the single-precision draws are twice the size of the cache
        k = randn(Hkv, n + tail, d)
        k[:, :n] = torch.where(mask[i], 0.1 * k[:, :n] + 0.75 * s[i], k[:, :n])
        k[:, 0] -= 0.75 * s[i, :, 0]
        k[..., 0] *= 0.05
        k[:, 0, 0] = sink
        K[i] = k
        v = randn(Hkv, n + tail, d)
        V[i] = v.mul_(math.sqrt(d) / v.norm(dim=-1, keepdim=True))
    return q.to(dtype), K, V


def _window_statistics(Q, K, V, tail):
    """The window rows' attention outputs and natural-log normalisers, as the prefill or the decode steps left them."""
    b, Hq, w, d = Q.shape
    Hkv, n_kv = K.shape[1], K.shape[2]
    O = torch.empty(b, Hq, w, d, device=Q.device)
    L = torch.empty(b, Hq, w, device=Q.device)
    G = Hq // Hkv
    future = torch.zeros(G * w, n_kv, dtype=torch.bool, device=Q.device)
    if tail:
        i = torch.arange(w, device=Q.device).repeat(G)[:, None]
        future[:, n_kv - tail:] = torch.arange(tail, device=Q.device)[None] > i
    for x in range(b):
        for h in range(Hkv):
            s = (Q[x, h * G:(h + 1) * G].float().reshape(G * w, d) @ K[x, h].float().T) / math.sqrt(d)
            s.masked_fill_(future, float("-inf"))
            lse = torch.logsumexp(s, dim=-1)
            O[x, h * G:(h + 1) * G] = (torch.exp(s - lse[:, None]) @ V[x, h].float()).view(G, w, d)
            L[x, h * G:(h + 1) * G] = lse.view(G, w)
    return O, L


def prepare(case, seed):
    Hq, Hkv, d, dtype = _geometry(case)
    b, n_kv = case["batch"], case["n"] + case["tail"]
    st = {"case": case, "handle": rk.Handle()}
    h = st["handle"]
    st["shape"] = rk.make_shape(b, Hq, Hkv, d, n_kv, WINDOW, case["tail"], rk.F32 if case["dtype"] == "f32" else rk.BF16)
    if case["call"] == "decode":
        g = torch.Generator(DEVICE).manual_seed(seed)
        st["q"] = torch.randn(b, Hq, d, generator=g, device=DEVICE).to(dtype)
        st["K"] = torch.randn(b, Hkv, n_kv, d, generator=g, device=DEVICE, dtype=dtype)
        st["V"] = torch.randn(b, Hkv, n_kv, d, generator=g, device=DEVICE, dtype=dtype)
        st["out"] = torch.empty(b, Hq, d, device=DEVICE)
        st["lse"] = torch.empty(b, Hq, device=DEVICE)
        st["workspace"] = torch.empty(h.workspace_bytes(st["shape"], 0), dtype=torch.uint8, device=DEVICE)
        return st
    st["Q"], st["K"], st["V"] = _inputs(case, seed)
    if case["call"] == "evict_from_lse":
        st["O"], st["L"] = _window_statistics(st["Q"], st["K"], st["V"], case["tail"])
    if case["d_model"]:
        g = torch.Generator(DEVICE).manual_seed(seed + 1)
        W_O = torch.randn(Hq * d, case["d_model"], generator=g, device=DEVICE).div_(math.sqrt(case["d_model"])).to(dtype)
        st["factor"] = torch.empty(h.output_projection_bytes(Hq, d), dtype=torch.uint8, device=DEVICE)
        h.prepare_output_projection(Hq, d, case["d_model"], rk.BF16, W_O, st["factor"])
        h.set_output_projection(st["factor"], Hq, d)
    adaptive = case["window"] == "adaptive"
    budget = min(case["budget"], n_kv)
    st["pool"] = rk.adaptive_pool(BETA, case["width"], budget) if adaptive else rk.fixed_pool(case["width"])
    st["scores"] = torch.empty(b, Hkv, n_kv, device=DEVICE)
    st["indices"] = torch.empty(b, Hkv, budget, dtype=torch.int32, device=DEVICE)
    st["K_out"] = torch.empty(b, Hkv, budget, d, dtype=dtype, device=DEVICE)
    st["V_out"] = torch.empty_like(st["K_out"])
    st["workspace"] = torch.empty(h.workspace_bytes(st["shape"], budget, adaptive=adaptive), dtype=torch.uint8, device=DEVICE)
    return st


def run(st):
    h, case = st["handle"], st["case"]
    if case["call"] == "decode":
        h.decode(st["shape"], st["q"], st["K"], st["V"], case["n"], st["out"], st["workspace"], lse=st["lse"])
        return {"out": st["out"], "lse": st["lse"]}
    if case["call"] == "evict_from_lse":
        h.evict_from_lse(st["shape"], st["Q"], st["K"], st["V"], st["O"], st["L"], DECAY, st["pool"], case["budget"],
                         st["indices"], st["K_out"], st["V_out"], st["workspace"], scores_out=st["scores"])
    else:
        h.evict(st["shape"], st["Q"], st["K"], st["V"], DECAY, st["pool"], case["budget"], st["indices"], st["K_out"],
                st["V_out"], st["workspace"], scores_out=st["scores"])
    return {"scores": st["scores"], "indices": st["indices"], "K": st["K_out"], "V": st["V_out"]}


def work(case):
    """K and V read once, the other inputs read and the outputs written once; the contractions of Eq. 3 (Q K^T, P V) and
    Eq. 7 (O V^T, and V W W^T V with a projection, as V L for a factor L of W W^T)."""
    Hq, Hkv, d, dtype = _geometry(case)
    b, n_kv, es = case["batch"], case["n"] + case["tail"], 4 if case["dtype"] == "f32" else 2
    rows = b * Hkv * n_kv
    kv = 2 * rows * d * es
    if case["call"] == "decode":
        return {"bytes": kv + b * Hq * (d * es + d * 4 + 4), "flops": 4 * b * Hq * n_kv * d}
    products = 2 if case["call"] == "evict_from_lse" else 3
    flops = products * 2 * b * Hq * WINDOW * n_kv * d
    size = kv + b * Hq * WINDOW * d * es + rows * 4 + b * Hkv * case["budget"] * (2 * d * es + 4)
    if case["call"] == "evict_from_lse":
        size += b * Hq * WINDOW * (d + 1) * 4
    if case["d_model"]:
        flops += 2 * b * Hq * n_kv * d * d
        size += Hq * d * d * 4
    return {"bytes": size, "flops": flops}


def tolerance(case):
    # Single precision: sums of 32-bit products.  bf16: the softmax weights meet V, and the outputs O meet V again, rounded to
    # bf16 (2^-8 each, random in sign), everything else is 32-bit.  The kept rows are those of the passages, well apart
    # from the others, so indices and copied rows have no reason to differ but for a tie.
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    if case["call"] == "decode":
        return {"rel": 3e-3, "max": 2e-2}
    return {"rel": 2e-3, "max": 1e-2, "differ": 1e-3}
