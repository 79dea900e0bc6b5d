"""Keys whose logits lie below the float range (-inf) take no part in the softmax, wherever they lie: the
first keys of a head, a whole key split or every key tile of one warpgroup, or the first keys of a
profiled window."""
import numpy as np
import pytest

import workloads as W
from fkharness import run_snapshot, to_dev

pytestmark = pytest.mark.gpu

LOWEST = -3.3895e38                           # the lowest bf16 value


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("heads,tokens", [(1, 341), (2, 700), (12, 1560)])   # one and two query tiles per CTA
@pytest.mark.parametrize("span", [(0, 32), (0, 130), (0, 1), "sink", "odd", "even"])
def test_keys_below_the_range(dim, heads, tokens, span):
    w = W.TINY_PER_FRAME.with_(name="below", n_heads=heads, head_dim=dim, tokens_per_frame=tokens, frames_per_chunk=1,
                               n_sink_frames=1, n_history_frames=2, n_segments=1, static_heads=tuple(range(heads)),
                               seed=heads + dim)
    rng = np.random.default_rng(dim)
    K = rng.standard_normal((3 * tokens, heads, dim))   # the view: current chunk, sink, anchor
    tile = np.arange(3 * tokens) // 128
    hit = {"sink": (np.arange(3 * tokens) // tokens) == 1, "odd": tile % 2 == 1, "even": tile % 2 == 0}.get(span)
    K[hit if hit is not None else slice(*span)] = LOWEST
    V = rng.standard_normal((3 * tokens, heads, dim))
    q = np.abs(rng.standard_normal((tokens, heads, dim))) + 0.1      # every product with LOWEST is negative
    b = W.to_bf16_bits
    rows = np.unique(np.linspace(0, tokens - 1, 40).astype(int))
    run_snapshot(w, rows=rows, inputs=(b(K[tokens:]), b(V[tokens:]), b(K[:tokens]), b(V[:tokens]), b(q)))


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("nk", [130, 1000, 2090])
@pytest.mark.parametrize("first", [1, 32, 64, 129])
def test_profiled_keys_below_the_range(dim, nk, first):
    import torch

    import oracle as O
    from paper_2605_09681_gb300 import head_profile
    rng = np.random.default_rng(nk + first)
    k = rng.standard_normal((nk, 3, dim))
    k[:first] = LOWEST
    k[nk // 2: nk // 2 + first // 2] = LOWEST
    q = np.abs(rng.standard_normal((200, 3, dim))) + 0.1
    qb, kb = W.to_bf16_bits(q), W.to_bf16_bits(k)
    g, s, t = 60, 20, 50
    mass, status = head_profile(to_dev(qb), to_dev(kb), g, s, t)
    torch.cuda.synchronize()
    qf, kf = W.bf16_bits_to_f32(qb), W.bf16_bits_to_f32(kb)
    ref = np.stack([O.head_attention_mass(qf[:, h], kf[:, h], g, s, t) for h in range(3)])
    assert int(status.item()) == 0
    assert np.abs(mass.cpu().numpy() - ref).max() <= 1e-4 * 200      # fp32 exponentials and sums
