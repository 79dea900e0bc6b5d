"""Steps of two caches queued behind one another on one stream, nothing waiting between them: each
gives what it gives alone, over many new caches."""
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
