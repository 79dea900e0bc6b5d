"""The calls that a video generator makes on a Forcing-KV cache, as cases to be timed and compared.

A case is a plain dict.  `kind` says which call sequence one pass is:

  step      one autoregressive step: append_chunk on every layer, compress, attend on every layer;
            with `denoise` > 1 the further denoising steps (set_current, attend) follow.  Each pass
            appends the next chunk of a small pool, as a generator does, to a window that is full.
  denoise   one later denoising step of a chunk: set_current, attend (the most frequent call).
  prefill   a history of `window` frames is loaded at once (append_frames), then the chunk is set,
            compressed and attended: the start of a video from given frames.
  profile   one offline head-profiling pass (Eq. 1) over a whole attention window.

Sizes are those of this repository's workloads (480P: 1560 tokens a frame, 1080P: 8160, 12 heads of
128 channels, chunks of 3 frames, the 30-layer stack, the rolling window, the comparison rules, FP8)
and generic ragged ones; `draw` spreads the same options over the whole range.
"""
import math

import numpy as np
import torch

from paper_2605_09681_gb300 import ForcingKVCache, head_profile

POOL = 2                                     # chunks that the passes of one state take in turn

_BASE = {"kind": "step", "layers": 1, "heads": 12, "dim": 128, "tokens": 1560, "chunk": 3, "sinks": 1,
         "window": 18, "segments": 6, "keep": 700, "static": 0.5, "scope": "per_frame",
         "source": "per_head", "incremental": False, "selection": "similarity", "drop_anchor": False,
         "precision": "bf16", "denoise": 1}


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # the smallest call: a test-sized model (60 tokens a frame, D = 64); launches and latency
        _case("prefill_tiny", kind="prefill", heads=4, dim=64, tokens=60, sinks=0, window=7, segments=1,
              keep=500, scope="pooled"),
        # a preview-sized two-layer model with ragged sizes (404 tokens a frame, 808 queries)
        _case("step_preview", layers=2, heads=6, tokens=404, chunk=2, sinks=2, window=5, segments=4,
              keep=600, denoise=2),
        # what a generator calls most: one of a chunk's later denoising steps, 480P
        _case("denoise_480p", kind="denoise"),
        # one 480P autoregressive step, the whole window rescored
        _case("step_480p"),
        # long videos: a rolling 12-frame window, scored and compacted incrementally
        _case("step_rolling", window=12, keep=600, incremental=True),
        # a whole model's step: 30 layers, the first layer's keys score for all of them
        _case("step_stack", layers=30, source="layer0_pooled", incremental=True),
        # the largest: 1080P, 24480 queries
        _case("step_1080p", tokens=8160, window=9),
        # FP8 attention on the compressed cache, Q K^T only and both products
        _case("step_fp8qk", precision="fp8_qk"),
        _case("denoise_fp8", kind="denoise", precision="fp8"),
        # comparison rules: StreamingLLM's 3 sinks and 4 recent frames on every head (equal lengths),
        # and random token pruning (one-token segments)
        _case("step_streaming", sinks=3, window=4, selection="all", static=0.0),
        _case("step_tokens", segments=1560, selection="random"),
        # offline profiling of one 480P layer over its full window
        {"name": "profile_480p", "kind": "profile", "heads": 12, "dim": 128, "tokens": 1560, "chunk": 3,
         "sinks": 1, "window": 18},
    ]


_MOST_FLOPS, _MOST_BYTES = 9.0e12, 3.0e9


def draw(rng):
    while True:
        kind = rng.choice(["step"] * 9 + ["denoise"] * 4 + ["prefill"] * 3 + ["profile"] * 4)
        tokens = math.exp(rng.uniform(math.log(48), math.log(8160)))
        c = {"kind": kind, "heads": rng.choice([1, 2, 3, 4, 6, 8, 12, 12, 12, 16]),
             "dim": rng.choice([64, 128, 128, 128]), "chunk": rng.choice([1, 2, 3, 3, 3, 4]),
             "sinks": rng.choice([0, 1, 1, 2, 3]), "window": rng.randint(2, 18)}
        if kind == "profile":
            c["tokens"] = int(tokens)
        else:
            c["selection"] = rng.choice(["similarity"] * 8 + ["all", rng.choice(["uniform", "random"])])
            if kind == "prefill" and c["selection"] == "random":
                c["selection"] = "uniform"
            c["segments"] = rng.choice([1, 2, 3, 4, 6, 6, 6, 8])
            if c["selection"] in ("uniform", "random"):       # token pruning: one-token segments
                tokens = min(tokens, 2048)
                c["segments"] = int(tokens)
            c["tokens"] = max(4 if c["segments"] < 48 else 1, round(tokens / c["segments"])) * c["segments"]
            c["keep"] = rng.randint(200, 1000)
            c["scope"] = "pooled" if c["selection"] == "similarity" and rng.random() < 0.25 else "per_frame"
            c["static"] = 0.0 if c["selection"] == "all" else rng.choice([0.0, 0.25, 0.5, 0.5, 0.5, 0.75])
            c["drop_anchor"] = False
            if c["selection"] == "all" and rng.random() < 0.5:
                c.update(static=0.5, drop_anchor=True)
            c["incremental"] = rng.random() < 0.5
            c["precision"] = "bf16" if c["dim"] == 64 else rng.choice(["bf16", "bf16", "bf16", "fp8_qk", "fp8"])
            c["layers"] = rng.randint(2, 30) if kind == "step" and rng.random() < 0.3 else 1
            c["source"] = "layer0_pooled" if c["layers"] > 1 and rng.random() < 0.5 else "per_head"
            c["denoise"] = rng.choice([1, 1, 2, 4]) if kind == "step" else 1
        w = work(c)
        if w["flops"] <= _MOST_FLOPS and w["bytes"] <= _MOST_BYTES:
            return c


# ------------------------------------------------------------------ sizes
def _queries(c):
    return c["chunk"] * c["tokens"]


def _head_map(c):
    """[layers, heads], 1 = static: a layer's share of static heads, in an order of its own."""
    m = np.zeros((c["layers"], c["heads"]), np.uint8)
    for l in range(c["layers"]):
        m[l, np.random.RandomState(100 + l).permutation(c["heads"])[:int(c["static"] * c["heads"])]] = 1
    return m


def _history(c):
    """(history frames, first window frame, anchor frame) that the first pass attends over."""
    nh = c["sinks"] + c["window"] + (c["chunk"] if c["kind"] == "step" else 0)
    return nh, max(c["sinks"], nh - c["window"]), nh - 1


def _keep_count(c):
    _, lo, anchor = _history(c)
    t, n = anchor - lo, c["segments"]
    if c["selection"] == "all":
        return t * n
    return t * (c["keep"] * n // 1000) if c["scope"] == "per_frame" else c["keep"] * t * n // 1000


def _key_counts(c):
    """Keys of a static and of a dynamic head."""
    F = c["tokens"]
    base = _queries(c) + c["sinks"] * F
    return base + (0 if c["drop_anchor"] else F), base + F + _keep_count(c) * (F // c["segments"])


def work(case):
    c = case
    F, H, D, nq = c["tokens"], c["heads"], c["dim"], _queries(c)
    if c["kind"] == "profile":
        nk = nq + (c["sinks"] + c["window"]) * F
        return {"bytes": 2.0 * (nq + nk) * H * D + 32 * H, "flops": 2.0 * nq * nk * H * D}
    ns, nd = _key_counts(c)
    m = _head_map(c)
    heads_s, heads_d = int(m.sum()), int((1 - m).sum())
    keys = heads_s * ns + heads_d * nd                       # attended in one pass over the layers
    cached = keys - c["layers"] * H * nq                     # of them, not the current chunk's
    row = 2.0 * D                                            # bytes of one bf16 row
    chunk = c["layers"] * H * nq * row
    n = c["denoise"]
    moved = n * (2 * chunk + 2 * chunk) + n * 2 * cached * row          # K, V, Q, O; cached K, V
    if c["kind"] == "step":                                  # the retired chunk joins the history
        moved += 2 * chunk * heads_d / (c["layers"] * H)
    if c["kind"] == "prefill":                               # the frames are read, and kept for scoring
        moved += 2.0 * c["window"] * F * row * (H + heads_d)
    return {"bytes": moved, "flops": n * 4.0 * nq * keys * D}


# ------------------------------------------------------------------ inputs
def _generator(*tags):
    s = 0x51ED2701
    for t in tags:
        s = (s * 1000003 + int(t) + 1) & 0x7FFFFFFFFFFF
    return torch.Generator(device="cuda").manual_seed(s)


def _ar1(g, frames, shape, rho):
    """`frames` frames [F, H, D] of x_f = rho x_{f-1} + sqrt(1 - rho^2) e_f, unit variance."""
    out = torch.empty((frames,) + shape, dtype=torch.float32, device="cuda")
    for f in range(frames):
        e = torch.randn(shape, generator=g, device="cuda")
        out[f] = e if f == 0 else rho * out[f - 1] + math.sqrt(1 - rho * rho) * e
    return out


def _layer_inputs(c, seed, layer):
    """Keys, values of the history and of the chunks that follow it, and queries, of one layer:
    neighbouring frames are correlated (0.9), each head's keys have a scale of their own."""
    F, H, D, C = c["tokens"], c["heads"], c["dim"], c["chunk"]
    nh = c["sinks"] + c["window"]
    n_chunks = {"step": 1 + POOL, "denoise": 2, "prefill": 1}[c["kind"]]
    g = _generator(seed, layer)
    scale = 0.5 + 1.5 * torch.rand((H, 1), generator=g, device="cuda")
    K = (_ar1(g, nh + n_chunks * C, (F, H, D), 0.9) * scale).to(torch.bfloat16)
    V = _ar1(g, nh + n_chunks * C, (F, H, D), 0.9).to(torch.bfloat16)
    q = [torch.randn((C * F, H, D), generator=g, device="cuda").to(torch.bfloat16) for _ in range(POOL)]

    def span(x, a, b):
        return x[a:b].reshape(-1, H, D).clone()

    chunks = [(span(K, nh + i * C, nh + (i + 1) * C), span(V, nh + i * C, nh + (i + 1) * C))
              for i in range(n_chunks)]
    return {"hist": (span(K, 0, nh), span(V, 0, nh)), "chunks": chunks, "q": q}


def _profile_inputs(c, seed):
    """One layer's window of keys [generated | sinks | other | transition] and its queries; heads
    range from attending to their own chunk to attending across the window."""
    F, H, D, nq = c["tokens"], c["heads"], c["dim"], _queries(c)
    nk = nq + (c["sinks"] + c["window"]) * F
    g = _generator(seed, 7)
    K = torch.randn((nk, H, D), generator=g, device="cuda")
    K[nk - F:] = 0.7 * K[nq - F:nq] + 0.7 * K[nk - F:]
    beta = 1.4 * torch.rand((H, 1), generator=g, device="cuda")
    Q = beta * K[:nq] + torch.randn((nq, H, D), generator=g, device="cuda")
    return Q.to(torch.bfloat16), K.to(torch.bfloat16), (nq, c["sinks"] * F, F)


class _State:
    """A cache with its history loaded, and the tensors of the passes."""

    def __init__(self, c, seed):
        self.c, self.i = c, 0
        self.cache = ForcingKVCache(
            n_layers=c["layers"], n_heads=c["heads"], head_dim=c["dim"], tokens_per_frame=c["tokens"],
            frames_per_chunk=c["chunk"], n_sink_frames=c["sinks"], window_frames=c["window"],
            n_segments=c["segments"], keep_budget_permille=c["keep"], head_is_static=_head_map(c),
            select_scope=c["scope"], score_source=c["source"], incremental=c["incremental"],
            max_history_frames=c["sinks"] + c["window"], selection=c["selection"], select_seed=7,
            static_drop_anchor=c["drop_anchor"], attn_precision=c["precision"])
        self.x = []
        for l in range(c["layers"]):
            x = _layer_inputs(c, seed, l)
            k, v = x.pop("hist")
            if c["kind"] == "prefill":           # the sinks are there; a pass loads the window
                n = c["sinks"] * c["tokens"]
                if n:
                    self.cache.append_frames(l, k[:n].clone(), v[:n].clone())
                x["hist"] = (k[n:].clone(), v[n:].clone())
            else:
                self.cache.append_frames(l, k, v)
                self.cache.set_current(l, *x["chunks"][0])
            self.x.append(x)
        if c["kind"] != "prefill":
            self.cache.compress()
        torch.cuda.synchronize()


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "profile":
        return {"c": c, "in": _profile_inputs(c, seed)}
    return _State(c, seed)


# ------------------------------------------------------------------ one pass
def run(state):
    if isinstance(state, dict):
        Q, K, (n_gen, n_sink, n_trans) = state["in"]
        mass, _ = head_profile(Q, K, n_gen, n_sink, n_trans)
        return mass
    c, cache, x = state.c, state.cache, state.x
    if c["kind"] == "denoise":
        cache.set_current(0, *x[0]["chunks"][1])
        return cache.attend(0, x[0]["q"][0])
    if c["kind"] == "prefill":
        cache.append_frames(0, *x[0]["hist"])
        cache.set_current(0, *x[0]["chunks"][0])
        cache.compress()
        return cache.attend(0, x[0]["q"][0])
    i = state.i % POOL
    state.i += 1
    L = c["layers"]
    out = torch.empty((c["denoise"], L) + tuple(x[0]["q"][0].shape), dtype=torch.bfloat16, device="cuda")
    for d in range(c["denoise"]):
        for l in range(L):
            if d == 0:
                cache.append_chunk(l, *x[l]["chunks"][1 + i])
            else:
                cache.set_current(l, *x[l]["chunks"][1 + (i + d) % POOL])
        if d == 0:
            cache.compress()
        for l in range(L):
            cache.attend(l, x[l]["q"][(i + d) % POOL], out[d, l])
    return out


# ------------------------------------------------------------------ comparison
def tolerance(case):
    if case["kind"] == "profile":
        return {"rel": 1e-5, "max": 1e-4}        # fp32 sums of exponentials, bf16 products exact in fp32
    if case["precision"] == "fp8":
        return {"rel": 2e-2, "max": 0.3}         # softmax numerators rounded to E4M3
    return {"rel": 1e-2, "max": 0.1}             # softmax numerators and outputs rounded to bf16


def _e4m3(x):
    return x.clamp(-448, 448).to(torch.float8_e4m3fn).to(torch.float64)


def _softmax_rows(q, k):
    s = torch.matmul(q, k.t()).mul_(1.0 / math.sqrt(q.shape[1]))
    s.sub_(s.amax(1, keepdim=True)).exp_()
    return s.div_(s.sum(1, keepdim=True))


def _attend64(c, q, k, v):
    """One head in 64 bits; under FP8 on the operands as the definition rounds them."""
    q, k, v = q.double(), k.double(), v.double()
    if c["precision"] != "bf16":
        e = torch.ceil(torch.log2(q.abs().amax(1, keepdim=True).clamp_min(1e-30) / 448))
        q, k = _e4m3(q * torch.exp2(-e)) * torch.exp2(e), _e4m3(k)
    if c["precision"] == "fp8":
        v = _e4m3(v)
    out = torch.empty_like(q)
    rows = max(1, int(2.5e8 // k.shape[0]))
    for a in range(0, q.shape[0], rows):
        out[a:a + rows] = torch.matmul(_softmax_rows(q[a:a + rows], k), v)
    return out


def _splitmix64(z):
    with np.errstate(over="ignore"):
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _kept(c, hist):
    """[T, n] per scored set: which segments of the window's scoreable frames are kept.  hist:
    [frames, F, heads, D] keys in 64 bits of the heads that score together."""
    _, lo, anchor = _history(c)
    T, n = anchor - lo, c["segments"]
    k = n if c["selection"] == "all" else c["keep"] * n // 1000
    j = np.arange(n)
    if c["selection"] == "all":
        s = np.zeros((T, n))
    elif c["selection"] == "uniform":
        s = np.ones((T, n))
        s[:, [i * n // k for i in range(k)]] = 0
    elif c["selection"] == "random":
        t = np.arange(lo, anchor)[:, None].astype(np.uint64)
        key = (np.uint64(7) << np.uint64(40)) ^ (t << np.uint64(20)) ^ j.astype(np.uint64)
        s = (_splitmix64(key) >> np.uint64(40)).astype(np.float64)
    else:
        x = hist[lo:anchor + 1].reshape(T + 1, n, -1)
        norm = x.square().sum(2)
        s = ((x[:-1] * x[1:]).sum(2) / (norm[:-1] * norm[1:]).sqrt()).cpu().numpy()
    keep = np.zeros((T, n), bool)
    if c["scope"] == "per_frame":
        for t in range(T):
            keep[t, np.argsort(s[t], kind="stable")[:k]] = True
    else:
        keep.reshape(-1)[np.argsort(s.reshape(-1), kind="stable")[:_keep_count(c)]] = True
    return keep


def _exact_profile(c, seed):
    Q, K, (n_gen, n_sink, n_trans) = _profile_inputs(c, seed)
    mass = torch.zeros((c["heads"], 4), dtype=torch.float64, device="cuda")
    nq, nk = Q.shape[0], K.shape[0]
    rows = max(1, int(2.5e8 // nk))
    for h in range(c["heads"]):
        k = K[:, h].double()
        for a in range(0, nq, rows):
            p = _softmax_rows(Q[a:a + rows, h].double(), k)
            mass[h] += torch.stack([torch.tensor(float(p.shape[0]), dtype=torch.float64, device="cuda"),
                                    p[:, :n_gen].sum(), p[:, nk - n_trans:].sum(),
                                    p[:, n_gen:n_gen + n_sink].sum()])
    return mass


def exact(case, seed):
    c = case
    if c["kind"] == "profile":
        return _exact_profile(c, seed)
    if work(c)["flops"] > 1.0e13:
        return None                              # over 20 seconds in 64 bits
    F, H, D, n = c["tokens"], c["heads"], c["dim"], c["segments"]
    nh, lo, anchor = _history(c)
    static = _head_map(c)
    step = c["kind"] == "step"
    out = torch.empty((c["denoise"], c["layers"], _queries(c), H, D), dtype=torch.float64, device="cuda")
    shared = None
    for l in range(c["layers"]):
        x = _layer_inputs(c, seed, l)
        hk, hv = x["hist"]
        if step:                                 # the pass retires the chunk that was current
            hk, hv = (torch.cat([a, b]) for a, b in zip((hk, hv), x["chunks"][0]))
        if c["source"] == "layer0_pooled" and l == 0:
            shared = _kept(c, hk.view(nh, F, H, D).double())
        first = 0 if c["kind"] == "prefill" else 1
        for h in range(H):
            rows = [torch.arange(c["sinks"] * F)]
            if not (static[l, h] and c["drop_anchor"]):
                rows.append(torch.arange(anchor * F, (anchor + 1) * F))
            if not static[l, h]:
                keep = shared if shared is not None else _kept(c, hk.view(nh, F, H, D)[:, :, h:h + 1].double())
                mask = torch.from_numpy(np.repeat(keep, F // n, axis=1).reshape(-1))
                rows.append(lo * F + torch.nonzero(mask).flatten())
            rows = torch.cat(rows).cuda()
            for d in range(c["denoise"]):
                ck, cv = x["chunks"][first + (d % POOL if step else 0)]
                out[d, l, :, h] = _attend64(c, x["q"][d % POOL][:, h], torch.cat([ck[:, h], hk[rows, h]]),
                                            torch.cat([cv[:, h], hv[rows, h]]))
    return out if step else out[0, 0]
