"""Attention: the running maximum raised in either part of a key tile (keys 0-95 and 96-127 are
handed to the tensor cores separately), in the first, a middle and the ragged last tile; every launch
plan (query tiles per CTA, key splits) by itself."""
import numpy as np
import pytest

import workloads as W
from fkharness import run_snapshot

pytestmark = pytest.mark.gpu


def _spiked(w, spikes, seed):
    """Snapshot inputs whose queries share a direction u, and keys a * u at the given positions of
    the head's key set [current chunk | sink | anchor]: logits of about 22.6 a (D = 128)."""
    rng = np.random.default_rng(seed)
    F, H, D = w.tokens_per_frame, w.n_heads, w.head_dim
    u = rng.choice([-1.0, 1.0], size=D)
    K = rng.standard_normal((3 * F, H, D))
    V = rng.standard_normal((3 * F, H, D))
    for pos, a in spikes:
        K[pos] = a * u
    q = rng.standard_normal((F, H, D)) + 2.0 * u
    b = W.to_bf16_bits
    return b(K[F:]), b(V[F:]), b(K[:F]), b(V[:F]), b(q)


PRECISIONS = [(64, "bf16"), (128, "bf16"), (128, "fp8_qk"), (128, "fp8")]
# (query tiles per CTA, key splits); None: the library's own choice
PLANS = [(t, k) for t in (2, 1) for k in range(1, 9)]


@pytest.mark.parametrize("dim,precision", PRECISIONS)
@pytest.mark.parametrize("tokens", [384, 404, 418])       # last tile full, 60 keys, 102 keys
@pytest.mark.parametrize("plan", [None, (2, 1), (1, 1), (2, 2)])
def test_maximum_raised_in_either_part(dim, precision, tokens, plan):
    """9 or 10 key tiles: all of them in one warpgroup's turn (2, 1), every other one (1, 1), half (2, 2)."""
    w = W.TINY_PER_FRAME.with_(name="parts", n_heads=2, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=1, n_history_frames=2, n_segments=2, static_heads=(0, 1),
                               attn_precision=precision)
    nk = 3 * tokens
    last = (nk - 1) // 128 * 128
    # part 2 of the first tile, part 1 and part 2 of middle tiles, both parts of one tile, the
    # last tile; each above the one before (0.25 is ~8 in log2 units)
    spikes = [(100, 0.25), (128 + 40, 0.5), (256 + 120, 0.75), (512 + 3, 1.0), (512 + 127, 1.5),
              (last + 5, 2.0), (nk - 1, 2.5)]
    for n in range(len(spikes) + 1):           # the maximum stays at each of them once
        run_snapshot(w, inputs=_spiked(w, spikes[:n], seed=n), plan=plan)


@pytest.mark.parametrize("dim,precision", PRECISIONS)
@pytest.mark.parametrize("plan", PLANS)
def test_plans(dim, precision, plan):
    """Every plan: one or two query tiles per CTA, 1 to 8 key splits, over 71 key tiles (each warpgroup gets
    at least 4), the last one of 88 keys, with the maximum raised in early and late tiles of each range."""
    F, frames = 312, 29                                      # 2 or 3 query tiles, 9048 keys
    w = W.TINY_PER_FRAME.with_(name="plans", n_heads=2, head_dim=dim, tokens_per_frame=F, frames_per_chunk=1,
                               n_sink_frames=frames - 2, n_history_frames=frames - 1, n_segments=1,
                               static_heads=(0, 1), attn_precision=precision)
    rng = np.random.default_rng(7)
    nk, b = frames * F, W.to_bf16_bits
    u = rng.choice([-1.0, 1.0], size=dim)
    K, V = rng.standard_normal((nk, 2, dim)), rng.standard_normal((nk, 2, dim))
    rise = np.linspace(0.1, 2.5, 24)                         # 24 keys, each above the ones before it
    K[np.linspace(300, nk - 20, 24).astype(int)] = rise[:, None, None] * u
    q = rng.standard_normal((F, 2, dim)) + 2.0 * u * (rng.random((F, 1, 1)) < 0.5)   # half of the rows follow u
    rows = np.unique(np.r_[np.linspace(0, F - 1, 60).astype(int), 127, 128, 255, 256])
    inputs = (b(K[F:]), b(V[F:]), b(K[:F]), b(V[:F]), b(q))
    run_snapshot(w, rows=rows, inputs=inputs, plan=plan)


@pytest.mark.parametrize("dim,precision", PRECISIONS)
@pytest.mark.parametrize("heads,tokens,sinks", [(1, 341, 1), (1, 345, 1), (40, 225, 3)])
@pytest.mark.parametrize("plan", PLANS)
def test_plans_of_short_heads(dim, precision, heads, tokens, sinks, plan):
    """8 or 9 key tiles, the last one of 127, 11 or 101 keys: ranges of one or two tiles, uneven over most splits,
    key sets of one tile or none, query tiles of 89 to 256 rows."""
    w = W.TINY_PER_FRAME.with_(name="short", n_heads=heads, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=sinks, n_history_frames=sinks + 1, n_segments=1,
                               static_heads=tuple(range(heads)), attn_precision=precision, seed=heads + tokens)
    run_snapshot(w, rows=np.arange(0, tokens, 1 if heads == 1 else 9), plan=plan)


def test_plans_that_do_not_fit():
    """More splits than a head has key tiles are refused by the call, and the cache goes on as before."""
    import torch

    from fkharness import to_dev
    from paper_2605_09681_gb300 import ForcingKVCache
    from paper_2605_09681_gb300._lib import FkError
    w = W.TINY_PER_FRAME.with_(name="fit", n_heads=1, tokens_per_frame=120, frames_per_chunk=1, n_sink_frames=1,
                               n_history_frames=2, static_heads=(0,))
    hk, hv, ck, cv, q = W.snapshot_inputs(w)
    with ForcingKVCache.from_workload(w, W.head_map(w)) as cache:
        cache.append_frames(0, to_dev(hk), to_dev(hv))
        cache.set_current(0, to_dev(ck), to_dev(cv))
        cache.compress()
        want = cache.attend(0, to_dev(q))
        for bad in ((3, 1), (0, 1), (1, 0), (2, 9), (-1, -1)):
            with pytest.raises(FkError):
                cache.force_attention_plan(*bad)
        cache.force_attention_plan(2, 4)                     # 360 keys: three key tiles
        with pytest.raises(FkError):
            cache.attend(0, to_dev(q))
        cache.force_attention_plan()
        assert torch.equal(cache.attend(0, to_dev(q)), want)


@pytest.mark.parametrize("dim,precision", PRECISIONS)
@pytest.mark.parametrize("heads,tokens,sinks", [(1, 171, 1), (1, 256, 1), (1, 277, 1), (1, 341, 1), (2, 170, 1),
                                                (40, 225, 3), (70, 225, 3), (1, 1040, 1)])
def test_key_splits(dim, precision, heads, tokens, sinks):
    """Grids whose heads have 4 to 9 (and 25) key tiles, the last one of 1 to 128 keys, as the library splits them
    (one query tile per CTA, up to 8 splits)."""
    w = W.TINY_PER_FRAME.with_(name="splits", n_heads=heads, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=sinks, n_history_frames=sinks + 1, n_segments=1,
                               static_heads=tuple(range(heads)), attn_precision=precision, seed=heads + tokens)
    run_snapshot(w)


@pytest.mark.parametrize("dim,precision", PRECISIONS)
@pytest.mark.parametrize("heads,tokens,history", [(1, 20, 2), (3, 43, 2), (2, 86, 2), (1, 127, 4), (2, 129, 5), (1, 300, 6)])
def test_one_query_tile(dim, precision, heads, tokens, history):
    """Small grids, one query tile per CTA over two sets of key tiles: 1 key tile (the second set is
    empty), 2 and 3, up to 17; query tiles of 1 to 128 rows; a larger key late in either set."""
    w = W.TINY_PER_FRAME.with_(name="one", n_heads=heads, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=history - 1, n_history_frames=history, n_segments=1,
                               static_heads=tuple(range(heads)), attn_precision=precision, seed=heads + tokens)
    hk, hv, ck, cv, q = W.snapshot_inputs(w)
    for plan in (None, (1, 1)):
        run_snapshot(w, inputs=(hk, hv, ck, cv, q), plan=plan)
        for frac in (0.6, 0.95):                  # a key well above the rest, in an even or an odd tile
            big = W.bf16_bits_to_f32(hk).copy()
            big[int(frac * len(big))] *= 4.0
            run_snapshot(w, inputs=(W.to_bf16_bits(big), hv, ck, cv, q), plan=plan)


@pytest.mark.parametrize("dim", [64, 128])
def test_key_splits_on_two_streams(dim):
    """Layers attended on two streams at once give what one stream gives, over many rounds."""
    import torch

    from paper_2605_09681_gb300 import ForcingKVCache
    g = torch.Generator(device="cuda").manual_seed(dim)
    L, H, F = 4, 3, 300
    with ForcingKVCache(n_layers=L, n_heads=H, head_dim=dim, tokens_per_frame=F, frames_per_chunk=2, n_sink_frames=1,
                        window_frames=6, n_segments=3, keep_budget_permille=700,
                        head_is_static=np.zeros((L, H), np.uint8)) as cache:
        def rand(n):
            return torch.randn((n, H, dim), generator=g, device="cuda").to(torch.bfloat16)
        for l in range(L):
            cache.append_frames(l, rand(7 * F), rand(7 * F))
            cache.set_current(l, rand(2 * F), rand(2 * F))
        cache.compress()
        q = [rand(2 * F) for _ in range(L)]
        want = [cache.attend(l, q[l]) for l in range(L)]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        for _ in range(20):
            outs = [torch.empty_like(x) for x in q]
            torch.cuda.synchronize()
            for l in range(L):
                cache.attend(l, q[l], outs[l], stream=streams[l % 2])
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(outs, want))
        assert cache.sync_status() == 0


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("g,s,t,nk", [(300, 100, 90, 1000), (512, 0, 128, 1024), (33, 7, 1, 2090), (0, 0, 480, 700)])
@pytest.mark.parametrize("heads,queries", [(3, 200), (8, 1000), (12, 1000)])
def test_profile_maximum_raised(dim, g, s, t, nk, heads, queries):
    """Head profiling: keys that raise the running maximum in tiles of one class, of two classes and
    in the last one; 6 or 8 key ranges per query tile of 1 to 3 tiles each (3 heads), 4 ranges of 1 to 5 (8), and
    2 of 3 to 9 (12), where both sets of statistics warps get tiles after their first."""
    import torch

    import oracle as O
    from fkharness import to_dev
    from paper_2605_09681_gb300 import head_profile
    rng = np.random.default_rng(nk + dim)
    u = rng.choice([-1.0, 1.0], size=dim)
    q = rng.standard_normal((queries, heads, dim)) + 2.0 * u
    for n in range(6):
        k = rng.standard_normal((nk, heads, dim))
        for pos, a in ((20, 0.25), (nk // 3, 0.5), (nk // 2, 1.0), (nk // 2 + 1, 1.5), (nk - 1, 2.0))[:n]:
            k[pos] = a * u
        qb, kb = W.to_bf16_bits(q), W.to_bf16_bits(k)
        mass, status = head_profile(to_dev(qb), to_dev(kb), g, s, t)
        torch.cuda.synchronize()
        qf, kf = W.bf16_bits_to_f32(qb), W.bf16_bits_to_f32(kb)
        check = sorted({0, heads // 2, heads - 1})
        ref = np.stack([O.head_attention_mass(qf[:, h], kf[:, h], g, s, t) for h in check])
        assert int(status.item()) == 0
        assert np.abs(mass.cpu().numpy()[check] - ref).max() <= 1e-4 * queries      # fp32 exponentials and sums
