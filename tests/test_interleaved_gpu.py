"""Steps of two caches queued behind one another on one stream, nothing waiting between them: each
gives what it gives alone, over many new caches.  And compressions with nothing but chained launches
between them and the launch that wrote the frames."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "fp8_qk"])
def test_steps_of_two_caches(precision):
    import torch

    from paper_2605_09681_gb300 import ForcingKVCache
    H, D, F, C, W = 12, 128, 1560, 3, 18
    static = np.zeros((1, H), np.uint8)
    static[0, [1, 2, 4, 5, 6, 9]] = 1
    g = torch.Generator(device="cuda").manual_seed(5)

    def frames(n):
        return torch.randn((n * F, H, D), generator=g, device="cuda").to(torch.bfloat16)

    data = [{"hist": (frames(1 + W), frames(1 + W)), "chunks": [(frames(C), frames(C)) for _ in range(3)],
             "q": frames(C)} for _ in range(2)]

    def make(d):
        cache = ForcingKVCache(n_layers=1, n_heads=H, head_dim=D, tokens_per_frame=F, frames_per_chunk=C,
                               n_sink_frames=1, window_frames=W, n_segments=6, keep_budget_permille=700,
                               head_is_static=static, attn_precision=precision)
        cache.append_frames(0, *d["hist"])
        cache.set_current(0, *d["chunks"][0])
        return cache

    def step(cache, d, i):
        cache.append_chunk(0, *d["chunks"][i])
        cache.compress()
        return cache.attend(0, d["q"])

    want = []
    for d in data:
        with make(d) as cache:
            outs = []
            for i in (1, 2):
                outs.append(step(cache, d, i))
                torch.cuda.synchronize()
            want.append(outs)
    for _ in range(100):
        with make(data[0]) as a, make(data[1]) as b:
            torch.cuda.synchronize()
            first, other, second = step(a, data[0], 1), step(b, data[1], 1), step(a, data[0], 2)
            torch.cuda.synchronize()
            assert torch.equal(first, want[0][0])
            assert torch.equal(other, want[1][0])
            assert torch.equal(second, want[0][1])


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("incremental", [False, True])
def test_compress_straight_after_frames(dim, incremental):
    """append_frames, then compress with no set_current between, and a second compress after an append of
    no frames: nothing but chained launches behind the one that wrote the frames.  Scores, kept sets and
    outputs over many new caches, queued behind one another, are the oracle's."""
    import torch

    import oracle as O
    import workloads as W
    from fkharness import compare_layer, to_dev
    from paper_2605_09681_gb300 import ForcingKVCache
    w = W.TINY_PER_FRAME.with_(name="straight", n_heads=8, head_dim=dim, tokens_per_frame=240, frames_per_chunk=2,
                               n_sink_frames=1, window_frames=9, n_segments=6, keep_budget_permille=500,
                               n_history_frames=14, static_heads=(3,), incremental=incremental)
    hm = W.head_map(w)
    hk, hv, ck, cv, q = W.snapshot_inputs(w)
    cut = 9 * w.tokens_per_frame
    parts = [(hk[:cut], hv[:cut]), (hk[cut:], hv[cut:]), (hk[:0], hv[:0])]
    orc = O.ForcingKVOracle.from_workload(w, hm)
    for k, v in parts:
        orc.append_frames(0, k, v)
    orc.set_current(0, ck, cv)
    dev = [(to_dev(k), to_dev(v)) for k, v in parts]
    cur, qd = (to_dev(ck), to_dev(cv)), to_dev(q)
    first = None
    for _ in range(50):
        caches = [ForcingKVCache.from_workload(w, hm) for _ in range(4)]
        torch.cuda.synchronize()
        outs = []
        for cache in caches:
            for k, v in dev:
                cache.append_frames(0, k, v)
                cache.compress()
            cache.set_current(0, *cur)
            outs.append(cache.attend(0, qd))
        torch.cuda.synchronize()
        for cache, out in zip(caches, outs):
            if first is None:
                first = out
                compare_layer(cache, orc, 0, q, out, label=w.name)
            assert torch.equal(out, first)
            for h in range(w.n_heads):
                assert cache.kept(0, h) == (orc.kept(0, h) if not hm[0, h] else [])
            assert cache.sync_status() == 0
            cache.close()
