"""The default split of decode batches of few rows, as ts_plan_step shows it: with units of `keys` keys on SMs that stream 70 GB/s
and 2 us per unit, no batch takes longer than with the split it would have without the rule (an SM's share, at least 512 keys)."""
import heapq

import numpy as np
import pytest

from paper_2512_03416_b200 import binding as B

SMS = 148                # assumed by the planner where there is no device


def make_ctx(Hq, Hkv, D, split=0):
    rc, h = B.ts_create(B.ts_config(Hq, Hkv, D, 16, 400000, 160, 2100, 0, 0, split, 0, 0.0, 0, 0, None, 0, None, 0))
    assert rc == B.TS_OK
    for r in range(160):
        rc, slot = B.ts_request_add(h, r, 1, 1)
        assert rc == B.TS_OK and slot == r and B.ts_alloc_pages(h, slot, 2000 * 16 + 1, 0) == B.TS_OK
    return h


def plan(h, keys):
    """Keys of every unit of a decode batch whose rows see `keys` keys, longest first."""
    for r, n in enumerate(keys):
        assert B.ts_request_set_len(h, r, n - 1) == B.TS_OK
    rc, items = B.ts_plan_step(h, B.make_step(list(range(len(keys))), [1] * len(keys), [n - 1 for n in keys])[0])
    assert rc == B.TS_OK
    return [i[5] - i[4] for i in items]


def makespan(items, Hkv, D):
    """us until the last SM is done: units in the order of the plan, each to the SM that is free first."""
    free = [0.0] * SMS
    for n in items:
        for _ in range(Hkv):
            heapq.heapreplace(free, free[0] + n * 4 * D / 70e3 + 2.0)
    return max(free)


@pytest.mark.parametrize("Hq,Hkv,D", [(32, 8, 128), (64, 8, 128), (8, 1, 128), (8, 2, 64), (16, 16, 128)], ids=lambda v: str(v))
def test_no_small_batch_is_planned_longer(Hq, Hkv, D):
    rng = np.random.default_rng(Hq + D)
    h = make_ctx(Hq, Hkv, D)
    fixed = {}
    batches = [[3042, 4371, 751], [5314, 1094, 638], [1880, 1441, 3387, 326], [7104]] + [[n] for n in range(500, 9000, 37)]
    for _ in range(700):
        rows = int(rng.integers(1, min(150, SMS // Hkv + 3)))
        batches.append(rng.integers(1, int(rng.choice([600, 1500, 5000, 30000])), rows).tolist())
    changed = 0
    for keys in batches:
        share = sum(keys) * Hkv // SMS
        base = -(-min(max(share, 512), 4096) // 64) * 64
        if base not in fixed:
            fixed[base] = make_ctx(Hq, Hkv, D, base)
        now, before = plan(h, keys), plan(fixed[base], keys)
        assert sum(now) == sum(before) == sum(keys)
        if len(keys) * Hkv > SMS or max(keys) <= 512 * 128 // D:
            assert now == before, keys
        if now != before:
            changed += 1
        assert makespan(now, Hkv, D) <= makespan(before, Hkv, D) * (1 + 1e-9), keys
    assert changed > 50
