"""Attention: the running maximum raised in either part of a key tile (keys 0-95 and 96-127 are
handed to the tensor cores separately), in the first, a middle and the ragged last tile."""
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


@pytest.mark.parametrize("dim,precision", [(64, "bf16"), (128, "bf16"), (128, "fp8_qk"), (128, "fp8")])
@pytest.mark.parametrize("tokens", [384, 404, 418])       # last tile full, 60 keys, 102 keys
def test_maximum_raised_in_either_part(dim, precision, tokens):
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
        run_snapshot(w, inputs=_spiked(w, spikes[:n], seed=n))


@pytest.mark.parametrize("dim,precision", [(64, "bf16"), (128, "bf16"), (128, "fp8_qk"), (128, "fp8")])
@pytest.mark.parametrize("heads,tokens,sinks", [(1, 171, 1), (1, 256, 1), (1, 277, 1), (1, 341, 1), (2, 170, 1),
                                                (40, 225, 3), (70, 225, 3), (1, 1040, 1)])
def test_key_splits(dim, precision, heads, tokens, sinks):
    """Grids whose heads have 4 to 9 (and 25) key tiles, the last one of 1 to 128 keys: 2 to 8 key
    splits with uneven ranges, query tiles of 1 to 256 rows."""
    w = W.TINY_PER_FRAME.with_(name="splits", n_heads=heads, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=sinks, n_history_frames=sinks + 1, n_segments=1,
                               static_heads=tuple(range(heads)), attn_precision=precision, seed=heads + tokens)
    run_snapshot(w)


@pytest.mark.parametrize("dim,precision", [(64, "bf16"), (128, "bf16"), (128, "fp8_qk"), (128, "fp8")])
@pytest.mark.parametrize("heads,tokens,history", [(1, 20, 2), (3, 43, 2), (2, 86, 2), (1, 127, 4), (2, 129, 5), (1, 300, 6)])
def test_one_query_tile(dim, precision, heads, tokens, history):
    """Small grids, one query tile per CTA over two sets of key tiles: 1 key tile (the second set is
    empty), 2 and 3, up to 14, over 1 to 8 splits; query tiles of 1 to 128 rows; the maximum raised late in either set."""
    w = W.TINY_PER_FRAME.with_(name="one", n_heads=heads, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=history - 1, n_history_frames=history, n_segments=1,
                               static_heads=tuple(range(heads)), attn_precision=precision, seed=heads + tokens)
    hk, hv, ck, cv, q = W.snapshot_inputs(w)
    run_snapshot(w, inputs=(hk, hv, ck, cv, q))
    for frac in (0.6, 0.95):                      # a key well above the rest, in an even or an odd tile
        big = W.bf16_bits_to_f32(hk).copy()
        big[int(frac * len(big))] *= 4.0
        run_snapshot(w, inputs=(W.to_bf16_bits(big), hv, ck, cv, q))


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
@pytest.mark.parametrize("g,s,t,nk", [(300, 100, 90, 1000), (512, 0, 128, 1024), (33, 7, 1, 2090), (0, 0, 0, 700)])
def test_profile_maximum_raised(dim, g, s, t, nk):
    """Head profiling: keys that raise the running maximum in tiles of one class, of two classes and
    in the last one, over 2 to 8 key ranges per query tile."""
    import torch

    import oracle as O
    from fkharness import to_dev
    from paper_2605_09681_gb300 import head_profile
    rng = np.random.default_rng(nk + dim)
    u = rng.choice([-1.0, 1.0], size=dim)
    q = rng.standard_normal((200, 3, dim)) + 2.0 * u
    for n in range(6):
        k = rng.standard_normal((nk, 3, dim))
        for pos, a in ((20, 0.25), (nk // 3, 0.5), (nk // 2, 1.0), (nk // 2 + 1, 1.5), (nk - 1, 2.0))[:n]:
            k[pos] = a * u
        qb, kb = W.to_bf16_bits(q), W.to_bf16_bits(k)
        mass, status = head_profile(to_dev(qb), to_dev(kb), g, s, t)
        torch.cuda.synchronize()
        qf, kf = W.bf16_bits_to_f32(qb), W.bf16_bits_to_f32(kb)
        ref = np.stack([O.head_attention_mass(qf[:, h], kf[:, h], g, s, t) for h in range(3)])
        assert int(status.item()) == 0
        assert np.abs(mass.cpu().numpy() - ref).max() <= 1e-4 * 200      # fp32 exponentials and sums
