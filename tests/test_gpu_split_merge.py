"""GPU parity of decode steps around the size from which the decode launch merges split rows itself."""
import numpy as np
import pytest
import torch

from paper_2512_03416_b200 import workloads as wl
from tests.helpers import GpuRun, assert_parity, oracle_step

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def check(b, launches, **kw):
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, **kw)
    for i in range(3):                                     # the counters are back at zero after a step
        before = run.dec.velocity()["kernel_launches"]
        assert_parity(run.step(keep_len=True), want, "peaked", f"step {i}")
        if i > 0:                                          # the first one may bring block-table entries along
            assert run.dec.velocity()["kernel_launches"] - before == launches
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("shape", [wl.Shape(32, 8, 128), wl.Shape(8, 1, 128), wl.Shape(3, 1, 128), wl.Shape(12, 1, 128), wl.Shape(16, 8, 64)],
                         ids=["32-8", "8-1", "3-1", "12-1", "d64"])
@pytest.mark.parametrize("over", [0, 1, 2])
def test_split_rows_are_merged_by_the_decode_launch(shape, over):
    """Rows in 2 to 18 splits of 64 keys; units on two thirds of the SMs (merged by a launch of its own), one item more, and
    more units than SMs."""
    n, ctx = (2 * sms() // (3 * shape.Hkv), 2 * sms() // (3 * shape.Hkv) + 1, sms() // shape.Hkv + 1)[over], []
    for pieces in [18, 9, 5, 4] + [2] * n:
        left = n - sum(-(-(c + 1) // 64) for c in ctx)
        if left <= 0:
            break
        ctx.append(64 * min(pieces, left) - 3)
    b = wl.make_batch("merge", shape, ctx, [1] * len(ctx), seed=over + shape.Hq, profile="peaked")
    check(b, 1 if over else 2, decode_split_tokens=64)


@pytest.mark.parametrize("rows,units,longest", [([521], 40, 128), ([2157], 96, 192), ([900] * 4 + [100], 136, 256), ([2000, 1500, 1100, 600], 144, 320),
                                                ([5400, 30, 4000, 300], 152, 576), ([2300] * 8, 128, 1152), ([970] * 12, 96, 971),
                                                ([3041, 4370, 750], 136, 512), ([16000] + [200] * 17, 256, 1088)],
                         ids=lambda r: f"{len(r)}x{r[0]}" if isinstance(r, list) else str(r))
def test_default_splits_of_steps_around_one_unit_per_SM(rows, units, longest):
    """The planned units and the longest one's keys on 148 SMs (of the last batch no split fits: an SM's share), who merges, and
    parity."""
    b = wl.make_batch("few", wl.LLAMA8B, rows, [1] * len(rows), seed=len(rows), profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    items = run.dec.plan_step(run.slots, [1] * len(rows), rows)
    if sms() == 148:
        assert (8 * len(items), max(i[5] - i[4] for i in items)) == (units, longest)
    for i in range(3):
        before = run.dec.velocity()["kernel_launches"]
        assert_parity(run.step(keep_len=True), want, "peaked", f"{rows}, step {i}")
        if i > 0:
            own_merge = len(items) > len(rows) and 3 * 8 * len(items) <= 2 * sms()
            assert run.dec.velocity()["kernel_launches"] - before == 1 + own_merge
    assert np.array_equal(run.pool(), pool_want)


def test_many_units_of_split_rows():
    """Most units are finished, counted and merged while their thread block streams on."""
    b = wl.make_batch("many", wl.Shape(32, 8, 128), [1000 + 37 * i for i in range(24)], [1] * 24, seed=5, profile="peaked")
    check(b, 1, decode_split_tokens=128)


@pytest.mark.parametrize("shape", [wl.Shape(8, 2, 128), wl.Shape(16, 2, 128), wl.Shape(32, 2, 128), wl.Shape(8, 2, 64)], ids=["G4", "G8", "G16", "d64"])
def test_a_rows_bits_do_not_depend_on_who_merges_it(shape):
    """200 rows of 5 to 18 splits, merged inside the decode launch by whichever warps finish a row's last split, and one by
    one, merged by a launch of their own: the same bits every time."""
    ctx = [64 * (5 + i % 14) - 1 - i % 60 for i in range(200)]
    b = wl.make_batch("bits", shape, ctx, [1] * 200, seed=shape.Hq, profile="peaked")
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    first = run.step(keep_len=True)
    for i in range(6):
        before = run.dec.velocity()["kernel_launches"]
        assert np.array_equal(run.step(keep_len=True), first), f"step {i}"
        assert run.dec.velocity()["kernel_launches"] - before == 1, "not merged inside the decode launch"
    lb, before = run.lb, run.dec.velocity()["kernel_launches"]
    for r in range(200):
        run.dec.mixed_step([lb.slots[r]], [1], [ctx[r]], lb.q[r:r + 1], lb.k_new[r:r + 1], lb.v_new[r:r + 1], lb.out[r:r + 1], keep_len=True)
    assert run.dec.velocity()["kernel_launches"] - before == 400, "not merged by a launch of their own"
    alone = lb.output()
    differ = np.flatnonzero((alone != first).any(axis=(1, 2)))
    assert differ.size == 0, f"rows {differ[:8]} differ, {int((alone != first).sum())} of {alone.size} values"


@pytest.mark.parametrize("shape", [wl.Shape(32, 2, 64), wl.Shape(32, 2, 128)], ids=["d64", "G16"])
def test_host_step_in_pieces_whose_rows_are_merged_elsewhere(shape):
    """Shapes whose decode rows never ride along with the tiles: the first piece's three rows are merged by a launch of their
    own, in the whole step by the decode launch. Bit for bit the same."""
    ctx = [1000, 990, 980, 0] + [64 * (5 + i % 14) - 9 for i in range(60)] + [0]
    ql = [1, 1, 1, 1400] + [1] * 60 + [1400]
    b = wl.make_batch("pieces", shape, ctx, ql, seed=shape.D, profile="peaked", chunk_size=sum(ql))
    one, two = GpuRun(b, decode_split_tokens=64), GpuRun(b, decode_split_tokens=64)
    want = one.step()
    host = [torch.from_numpy(a.view(np.int16)).pin_memory() for a in (b.q, b.k_new, b.v_new)]
    out = torch.full(host[0].shape, 0x7FC0, dtype=torch.int16).pin_memory()
    two.dec.mixed_step_host(two.slots, ql, ctx, *host, out)
    assert two.dec.velocity()["kernel_launches"] > one.dec.velocity()["kernel_launches"] + 2, "it went in one piece"
    assert np.array_equal(wl.bf16_bits_to_f32(out.numpy().view(np.uint16)), want)
    assert np.array_equal(two.pool(), one.pool())
    assert two.dec.device_status() == 0


@pytest.mark.parametrize("items,launches", [(152, 1), (153, 2), (266, 2), (267, 1)])
def test_who_merges_short_units_of_head_dim_64(items, launches):
    """One wave of units and four more, a second one of up to 1.8 units per SM, and more, on 148 SMs: the first and last are merged by the
    decode launch."""
    if sms() != 148:
        pytest.skip("sizes are those of 148 SMs")
    ctx = [64 * 3 - 5] * (items // 3) + [64 * (items % 3) - 7] * (items % 3 > 0)
    b = wl.make_batch("wave", wl.Shape(4, 1, 64), ctx, [1] * len(ctx), seed=items, profile="peaked")
    check(b, launches, decode_split_tokens=64)
