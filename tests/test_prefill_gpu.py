"""Prefill of history frames in one launch per push: batches of frames, pushes that straddle the
sinks or exceed the window, and every kind of destination, against the oracle."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from fkharness import compare_layer, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,precision", [(64, "bf16"), (128, "bf16"), (128, "fp8")])
@pytest.mark.parametrize("sinks,window,pushes", [(0, 3, (1, 1)), (2, 4, (1, 3, 1)), (1, 4, (4, 5)), (3, 2, (9,)),
                                                 (1, 0, (2, 6, 1)), (2, 8, (5, 0, 8)), (0, 16, (13,))])
@pytest.mark.parametrize("drop", [False, True])
def test_prefill_pushes(dim, precision, sinks, window, pushes, drop):
    from paper_2605_09681_gb300 import ForcingKVCache
    w = W.TINY_PER_FRAME.with_(name="prefill", n_heads=3, head_dim=dim, tokens_per_frame=33, frames_per_chunk=2,
                               n_sink_frames=sinks, window_frames=window, n_segments=3, keep_budget_permille=700,
                               n_history_frames=sum(pushes), static_heads=(1,), attn_precision=precision,
                               static_drop_anchor=drop, seed=sum(pushes))
    hm = W.head_map(w)
    hk, hv, ck, cv, q = W.snapshot_inputs(w)
    F = w.tokens_per_frame
    orc = O.ForcingKVOracle.from_workload(w, hm)
    with ForcingKVCache.from_workload(w, hm) as cache:
        f = 0
        for n in pushes:
            for dst, conv in ((cache, to_dev), (orc, lambda a: a)):
                dst.append_frames(0, conv(hk[f * F:(f + n) * F]), conv(hv[f * F:(f + n) * F]))
            f += n
        cache.set_current(0, to_dev(ck), to_dev(cv))
        orc.set_current(0, ck, cv)
        cache.compress()
        compare_layer(cache, orc, 0, q, cache.attend(0, to_dev(q)), label=str((sinks, window, pushes)))
        assert cache.sync_status() == 0
