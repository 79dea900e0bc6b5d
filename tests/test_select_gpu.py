"""Selection with many segments per frame (radix select): sizes around the thread count, budgets from
none to all, ties, and every rule, against the oracle."""
import numpy as np
import pytest

import workloads as W
from fkharness import run_snapshot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,keep", [(65, 500), (65, 1000), (100, 9), (255, 700), (256, 0), (257, 996), (600, 333),
                                    (1023, 700)])
@pytest.mark.parametrize("rule", ["similarity", "random", "uniform", "all"])
def test_many_segments(n, keep, rule):
    w = W.TINY_PER_FRAME.with_(name="segments", n_heads=2, head_dim=64, tokens_per_frame=n, frames_per_chunk=1,
                               n_segments=n, keep_budget_permille=keep, n_history_frames=4, static_heads=(1,),
                               selection=rule, select_seed=n, seed=n)
    hk, hv, ck, cv, q = W.snapshot_inputs(w)
    run_snapshot(w, inputs=(hk, hv, ck, cv, q))
    if rule == "similarity":                     # few distinct scores: ties at every boundary
        hk = hk.reshape(4, n, 2, 64).copy()
        hk[:, 7:] = hk[:, np.arange(n - 7) % 7]
        hk[2, : n // 2] = hk[3, : n // 2]        # and scores of exactly 1
        run_snapshot(w, inputs=(hk.reshape(4 * n, 2, 64), hv, ck, cv, q))
