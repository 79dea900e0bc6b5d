"""Selection with many segments per frame (radix select): sizes around the thread count, budgets from
none to all, ties, and every rule, against the oracle; configurations at the limits of shared memory."""
import os
import subprocess
import sys

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


# Values staged and n_segments whose shared memory lies at the limit of a launch without a request (48 KB),
# with the most a frame may have, and at the most that is accepted (227 KB).
LIMITS = [dict(n=1000, window=9, rule="similarity"), dict(n=1000, window=9, rule="random", scope="pooled"),
          dict(n=64, window=190, rule="similarity"), dict(n=64, window=192, rule="random"),
          dict(n=12, window=1023, rule="similarity"), dict(n=4096, window=3, rule="random"),
          dict(n=8192, window=3, rule="uniform"), dict(n=8192, window=3, rule="all"),
          dict(n=8400, window=2, rule="random"), dict(n=64, window=907, rule="random", scope="pooled"),
          dict(n=64, window=907, rule="random")]


@pytest.mark.parametrize("case", LIMITS, ids=lambda c: "-".join(map(str, c.values())))
def test_shared_memory_limits(case):
    """Each in a process of its own: a handle raises the limit for those that follow."""
    here = os.path.dirname(os.path.abspath(__file__))
    code = ("import sys; sys.path[:0] = [%r, %r]; import test_select_gpu as t; t.at_limit(**%r)"
            % (here, os.path.dirname(here), case))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-1500:]


def at_limit(n, window, rule, scope="per_frame"):
    w = W.TINY_PER_FRAME.with_(name="limit", n_heads=2, head_dim=64, tokens_per_frame=n, frames_per_chunk=1,
                               n_segments=n, keep_budget_permille=300, n_history_frames=window, static_heads=(1,),
                               selection=rule, select_scope=scope, select_seed=n, seed=n)
    run_snapshot(w, rows=np.arange(2), window_frames=window)


def test_shared_memory_refusals():
    """One past the most that is accepted is refused when the cache is made."""
    from paper_2605_09681_gb300 import ForcingKVCache
    from paper_2605_09681_gb300._lib import FkError
    for n, window in ((64, 909), (8500, 2), (16384, 2), (1560, 35)):
        w = W.TINY_PER_FRAME.with_(name="past", n_heads=1, head_dim=64, tokens_per_frame=n, frames_per_chunk=1,
                                   n_segments=n, n_history_frames=2, static_heads=(), selection="random")
        with pytest.raises(FkError):
            ForcingKVCache.from_workload(w, W.head_map(w), window_frames=window)
