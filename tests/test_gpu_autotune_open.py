"""The autotuners time the library's own launch shape (every knob 0) beside the explicit ones, so that their
choice is never slower than not tuning by more than the timing's noise, and a plan that holds it runs it."""
import numpy as np
import pytest
import torch

from gpu_util import t
from test_gpu_block_search import _setup

pytestmark = pytest.mark.gpu


def _open(row):
    return row["queries_per_warp"] == row["warps_per_block"] == row["hash_slots"] == 0


def test_autotune_times_the_library_choice():
    import paper_2312_16335_gb300 as lv
    idx, Q, P = _setup(lv, 6000, 96, 48, 8, 64, 0, 100, seed=2)
    tune = lv.autotune(idx, Q, P, k=10, L=160, rerank=160, width=2, reps=1)
    assert sum(_open(r) for r in tune["table"]) == 1
    assert tune["best"]["ms"] <= next(r["ms"] for r in tune["table"] if _open(r))
    assert not any(_open(r) for r in lv.autotune(idx, Q, P, k=10, L=64, queries_per_warp=(2,), reps=1)["table"])


def test_uneven_plans_time_and_run_the_library_choice():
    import paper_2312_16335_gb300 as lv
    idx, Q, P = _setup(lv, 6000, 96, 48, 8, 64, 0, 100, seed=3)
    rng = np.random.default_rng(4)
    L = rng.integers(10, 260, 100)
    k = np.minimum(L, 10)
    desc = t(np.stack([k, L, L, np.zeros(100, int)], 1).astype(np.int32))
    want = idx.search(Q, P, k=10, L=int(L.max()), rerank=int(L.max()), desc=desc, ldo=10, width=2, queries_per_warp=1)
    tuned = lv.autotune_uneven(idx, Q, P, desc, ldo=10, width=2, bounds=(64, 128, 320), reps=1)
    for name, launches in tuned["plan_launches"].items():
        rows = [r for r in tuned["table"] if r["plan"] == name and _open(r)]
        assert len(rows) == len(launches)
        for c, r in zip(launches, rows):
            assert c["ms"] <= r["ms"]
        plan = {"order": tuned["plan_orders"][name],
                "classes": [dict(c, queries_per_warp=0, warps_per_block=0, hash_slots=0) for c in launches]}
        g = lv.UnevenGraph(idx, Q, P, desc, plan, ldo=10, width=2)
        assert all(kw["warps_per_query"] == 0 for _, kw in g.calls)
        ids, sc = g.replay()
        torch.cuda.synchronize()
        assert torch.equal(g.unsorted(ids), want[0]) and torch.equal(g.unsorted(sc), want[1])
    assert not any(_open(r) for r in lv.autotune_uneven(idx, Q, P, desc, ldo=10, teams=(2,), reps=1)["table"])
