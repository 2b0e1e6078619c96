"""GPU parity: ts_mixed_step / ts_kv_append through the C ABI against the CPU oracle."""
import math

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


@pytest.mark.parametrize("profile", ["paper", "peaked", "needle"])
def test_config1_tiny_mixed(profile):
    b = wl.config1(profile=profile)
    want, pool_want = oracle_step(b)
    run = GpuRun(b)
    got = run.step()
    assert_parity(got, want, profile, f"config1/{profile}")
    assert np.array_equal(run.pool(), pool_want), "pool differs after append"


@pytest.mark.parametrize("profile", ["paper", "peaked", "needle"])
def test_config2_decode_8b(profile):
    b = wl.config2(profile=profile)
    want, pool_want = oracle_step(b)
    run = GpuRun(b)
    got = run.step()
    assert_parity(got, want, profile, f"config2/{profile}")
    assert np.array_equal(run.pool(), pool_want)


CASES = [
    # (Hq, Hkv, D, ctx list, q_len list)
    (4, 2, 64, [1, 15, 16, 17], [1, 1, 1, 1]),
    (8, 1, 128, [255, 256, 257, 0], [1, 1, 1, 1]),
    (8, 8, 64, [0, 3], [2, 17]),
    (16, 2, 128, [0, 31, 100], [64, 130, 1]),
    (6, 2, 64, [5, 77], [33, 1]),
    (32, 8, 128, [700, 0, 1300], [1, 200, 1]),
    (64, 8, 128, [513, 64], [1, 96]),
    (2, 2, 128, [0], [1]),
    (12, 4, 64, [19], [300]),
    (16, 1, 64, [40, 41], [1, 5]),
    # head_dim 128 with group sizes that do not divide 128 (query tiles of 126, 125, 126, 120 packed rows)
    (24, 8, 128, [300, 0, 77], [1, 200, 1]),
    (40, 8, 128, [33, 5], [1, 150]),
    (48, 8, 128, [129, 600, 18], [140, 1, 1]),
    (7, 1, 128, [0, 260], [90, 1]),
    (12, 1, 128, [70, 15, 0], [1, 1, 75]),
    # sixteen query heads per KV head at head_dim 128: 8-token query tiles, the decode rows in a
    # launch of their own (two head groups per unit) followed by the split merge
    (16, 1, 128, [900, 0, 4500, 31], [1, 70, 1, 1]),
    (32, 2, 128, [257, 5000, 12], [1, 1, 100]),
    (32, 2, 128, [255, 256, 4700, 0], [1, 1, 1, 1]),
    (16, 1, 128, [4200, 63], [1, 1]),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}-{c[1]}-{c[2]}-{i}" for i, c in enumerate(CASES)])
@pytest.mark.parametrize("profile", ["peaked", "needle"])
def test_shape_sweep(case, profile):
    Hq, Hkv, D, ctx, ql = case
    b = wl.make_batch("sweep", wl.Shape(Hq, Hkv, D), ctx, ql, seed=hash(case[:3]) % 1000 + len(ctx), profile=profile)
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    got = run.step()
    assert_parity(got, want, profile, f"sweep {case}")
    assert np.array_equal(run.pool(), pool_want)


def test_empty_step_launches_nothing():
    b = wl.make_batch("e", wl.TINY, [3], [1], seed=3)
    run = GpuRun(b)
    before = run.dec.velocity()
    run.dec.mixed_step([], [], [], None, None, None, None)
    after = run.dec.velocity()
    assert after["kernel_launches"] == before["kernel_launches"] and after["steps"] == before["steps"]


@pytest.mark.parametrize("split", [64, 128, 192, 1024, 1 << 20])
def test_split_count_invariance(split):
    b = wl.make_batch("s", wl.LLAMA8B, [1000, 63, 64, 4095], [1, 1, 1, 1], seed=9, profile="peaked")
    want, _ = oracle_step(b)
    got = GpuRun(b, decode_split_tokens=split).step()
    assert_parity(got, want, "peaked", f"split {split}")


@pytest.mark.parametrize("profile", ["paper", "peaked", "needle"])
def test_config3_burst_8b(profile):
    b = wl.config3(profile=profile)
    want, pool_want = oracle_step(b)
    run = GpuRun(b)
    got = run.step()
    assert_parity(got, want, profile, f"config3/{profile}")
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("profile", ["paper", "peaked", "needle"])
def test_config4_chunked_8b(profile):
    b = wl.config4(profile=profile)
    want, pool_want = oracle_step(b)
    run = GpuRun(b)
    got = run.step()
    assert_parity(got, want, profile, f"config4/{profile}")
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("prefill_ctas", [-1, 0, 1, 3, 100, 1000])
def test_mixed_launch_split_invariance(prefill_ctas):
    """The result does not depend on how the attention launch divides its CTAs between prefill
    tiles and decode rows: two launches (-1), the cost model (0), one or three prefill CTAs (the
    decode CTAs then take most tiles from the queue, many work units per CTA), or more prefill
    CTAs than there are SMs (clamped)."""
    b = wl.make_batch("mix", wl.LLAMA8B, [700, 50, 1300, 3000, 9, 0, 200], [1, 1, 1, 1, 1, 600, 130], seed=21,
                      profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, mixed_prefill_ctas=prefill_ctas)
    got = run.step()
    assert_parity(got, want, "peaked", f"mixed launch, prefill_ctas={prefill_ctas}")
    assert np.array_equal(run.pool(), pool_want)


def test_prefill_only_many_units_per_cta():
    """A prefill-only step with more work units (tile pairs x KV heads) than SMs: every CTA of the
    persistent kernel walks through several units, and the units differ in length."""
    b = wl.make_batch("pf", wl.LLAMA8B, [37, 0], [1300, 75], seed=22, profile="needle")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    got = run.step()
    assert_parity(got, want, "needle", "prefill-only, many units")
    assert np.array_equal(run.pool(), pool_want)


def test_mixed_70b_shape_group8():
    """Eight query heads per KV head (the 70B-shaped layer): 16-token query tiles, decode rows in the same launch."""
    b = wl.make_batch("m70", wl.LLAMA70B, [900, 17, 2500, 0], [1, 1, 1, 200], seed=23, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    got = run.step()
    assert_parity(got, want, "peaked", "70B-shaped mixed step")
    assert np.array_equal(run.pool(), pool_want)


def test_maximum_sizes_sampled():
    """The largest shapes the workloads allow (70B-shaped layer): a decode row whose context fills
    a 2048-page block table (32768 tokens with its new one) and an 8192-token prefill chunk that
    continues 24576 cached tokens, so its last token also sees 32768 keys. The oracle checks every
    decode row and a sample of the chunk (its first and last tokens, the edges of every 128-token
    stretch and 200 seeded tokens); the pool is compared in full."""
    b = wl.make_batch("max", wl.LLAMA70B, [32767, 24576, 15], [1, 8192, 1], seed=31, profile="peaked",
                      chunk_size=8194)
    rng = np.random.default_rng(2)
    chunk = 1 + np.unique(np.concatenate([[0, 8191], np.arange(0, 8192, 128), np.arange(127, 8192, 128),
                                          rng.integers(0, 8192, 200)]))
    sel = np.concatenate([[0], chunk, [8193]]).astype(np.int32)
    want, pool_want = oracle_step(b, sel=sel)
    run = GpuRun(b)
    got = run.step()[sel]
    assert_parity(got, want, "peaked", "maximum sizes")
    assert np.array_equal(run.pool(), pool_want)


def test_a_wait_that_runs_out_is_reported_and_the_next_step_is_clean():
    """Failure path without a fault: with TS_DEBUG_LOSE_APPEND_ARRIVAL the wait in front of the merge of
    a mixed step's decode splits is for one thread block more than stream them, under a limit of
    2 million clock cycles (about a millisecond; never the library's default second). Every block
    then gives that wait up, raises TS_DEV_TIMEOUT and carries on. The step must return, the status
    call must report TS_ERR_DEVICE_TIMEOUT once and then be clean, and a normal context's next
    step on the same device must match the oracle, pool included."""
    from paper_2512_03416_b200 import binding as B
    b = wl.make_batch("tmo", wl.LLAMA8B, [300, 40, 0], [1, 1, 300], seed=41, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64, wait_limit_cycles=2_000_000, debug_flags=B.TS_DEBUG_LOSE_APPEND_ARRIVAL)
    run.lb.step(keep_len=True)
    rc, bits = B.ts_last_device_status(run.dec.ctx, torch.cuda.current_stream().cuda_stream)
    assert rc == B.TS_ERR_DEVICE_TIMEOUT and bits & B.TS_DEV_TIMEOUT
    # all blocks had in fact arrived, so even this step's result is complete
    assert_parity(run.lb.output(), want, "peaked", "step whose merge gave up its wait")
    rc, bits = B.ts_last_device_status(run.dec.ctx, torch.cuda.current_stream().cuda_stream)
    assert rc == B.TS_OK and bits == 0, "the status word was not cleared"
    # the launch's counters are back at zero: the same context runs the step again, still flagged
    run.lb.step(keep_len=True)
    assert run.dec.device_status() == B.TS_DEV_TIMEOUT
    run.dec.close()
    # without a split row nothing waits for the blocks that stream decode rows: the flag changes nothing
    whole = GpuRun(b, chunk_size=0, wait_limit_cycles=2_000_000, debug_flags=B.TS_DEBUG_LOSE_APPEND_ARRIVAL)
    assert_parity(whole.step(), want, "peaked", "flagged step without split rows")
    # and a context without the flag is clean
    ok = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    got = ok.step()
    assert_parity(got, want, "peaked", "step after a timed-out one")
    assert np.array_equal(ok.pool(), pool_want)



@pytest.mark.parametrize("shape", [wl.LLAMA8B, wl.Shape(64, 8, 128), wl.Shape(2, 2, 128)], ids=["32-8", "64-8", "2-2"])
@pytest.mark.parametrize("rows", [
    # (cached tokens, chunk) per row: the chunk starts on and around page and key-tile boundaries, and
    # ends inside a page, at its end, one past a key tile
    [(0, 128), (15, 2), (16, 16), (17, 15)],
    [(127, 129), (128, 127), (129, 40), (1, 255)],
    [(300, 200), (113, 15), (271, 17), (0, 2), (50, 1)],
    [(143, 300), (640, 33), (1000, 1)],
], ids=["starts", "tiles", "mixed", "long"])
def test_chunk_tokens_are_read_from_the_step_tensors(shape, rows):
    """Key tiles of cached tokens, of the chunk's own tokens, and of both, several chunks in one step,
    without decode rows, next to a few, and in a launch of few and of many work units."""
    b = wl.make_batch("own", shape, [c for c, _ in rows], [t for _, t in rows], seed=len(rows) + shape.Hq, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    assert_parity(run.step(keep_len=True), want, "peaked", f"{rows}")
    assert np.array_equal(run.pool(), pool_want)
    assert_parity(run.step(), want, "peaked", f"{rows}, repeated")


def test_another_rows_values_cannot_reach_a_chunk():
    """A key tile of a chunk is copied with whatever tokens follow the chunk in the step's tensors;
    infinities and NaN there must not reach the chunk's output, nor its pages anything but its own tokens."""
    b = wl.make_batch("nan", wl.LLAMA8B, [37, 5, 0], [90, 60, 20], seed=77, profile="peaked")
    want, _ = oracle_step(b)
    b.k_new[90:150] = wl.BF16_NAN
    b.v_new[90:150:2] = 0x7F80
    b.v_new[91:150:2] = wl.BF16_NAN
    _, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    got = run.step()
    clean = np.r_[0:90, 150:170]
    assert_parity(got[clean], want[clean], "peaked", "rows around a row of NaN")
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("shape", [wl.LLAMA8B, wl.Shape(64, 8, 128), wl.Shape(16, 1, 128), wl.Shape(8, 2, 64)], ids=["32-8", "64-8", "16-1", "8-2"])
@pytest.mark.parametrize("split", [64, 4096])
def test_decode_units_of_all_lengths(shape, split):
    """More units than thread blocks, of one page to many: units shorter than a warp's look-ahead follow
    one another, warps without a page of a unit, rows that end on and around page boundaries. The
    largest scores come late in some rows, so that the running reference has to move more than once."""
    ctx = [0, 1, 14, 15, 16, 127, 128, 129, 255, 383, 384, 385, 1000, 2047, 5000] * 3 + [3] * 30
    b = wl.make_batch("units", shape, ctx, [1] * len(ctx), seed=split + shape.Hq, profile="peaked")
    grow = np.linspace(1.0, 6.0, len(b.context_k))[:, None, None]
    b.context_k[:] = wl.f32_to_bf16_bits((wl.bf16_bits_to_f32(b.context_k) * grow).astype(np.float32))
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=split)
    for _ in range(2):                                     # the unit queue is back at zero after a step
        assert_parity(run.step(keep_len=True), want, "peaked", f"split {split}")
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("rows", [[0], [511, 512], [513, 40, 1500], [8191], [1500] * 20, [700, 3000, 150] * 9], ids=lambda r: f"{len(r)}x{r[0]}")
def test_default_splits_of_small_batches(rows):
    """The default split follows the batch: rows around the shortest split, one long row, batches whose
    share per SM lies between the limits; next to a chunk as well."""
    for extra in ([], [(0, 33)]):
        b = wl.make_batch("few", wl.LLAMA8B, rows + [c for c, _ in extra], [1] * len(rows) + [t for _, t in extra], seed=len(rows),
                          profile="peaked")
        want, pool_want = oracle_step(b)
        run = GpuRun(b, chunk_size=0)
        assert_parity(run.step(), want, "peaked", f"{rows} {extra}")
        assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("shape", [wl.LLAMA8B, wl.Shape(16, 1, 128), wl.Shape(8, 2, 64)], ids=["32-8", "16-1", "8-2"])
@pytest.mark.parametrize("chunk", [0, 40], ids=["decode", "mixed"])
def test_a_decode_rows_largest_weight_is_exact(shape, chunk):
    """A row whose softmax is carried by a late key, a little above a key of an earlier page of the same
    warp, everything else far below. The largest weight of a page that brings a new maximum is 1 and thus exact
    in bf16, and earlier sums are rescaled in fp32: what is left is the rounding of the result, 2^-8 of it.
    A weight taken against a reference that lags behind the maximum would be rounded as well: another
    2^-8 of nearly the whole result."""
    ctx = [300, 1100, 131] + [0] * (chunk > 0)
    b = wl.make_batch("late", shape, ctx, [1] * 3 + [chunk] * (chunk > 0), seed=shape.Hq + chunk, profile="peaked")
    G, D = shape.Hq // shape.Hkv, shape.D
    first, late = 5, 130                                   # pages 0 and 8: the same warp of a unit
    starts = np.concatenate([[0], np.cumsum(ctx)])[:3]
    coef = np.full(len(b.context_k), -1000.0)
    for at in starts:
        coef[at + first], coef[at + late] = 1.0, 2.0
    b.context_k[:] = 0
    b.context_k[:, :, 0] = wl.f32_to_bf16_bits(coef.astype(np.float32))[:, None]
    b.k_new[:3] = 0
    b.k_new[:3, :, 0] = wl.f32_to_bf16_bits(np.array([-1000.0], np.float32))[0]
    gap = np.linspace(0.3, 7.6, 3 * shape.Hq).reshape(3, shape.Hq)          # log2(weight of late / of first)
    b.q[:3] = 0
    b.q[:3, :, 0] = wl.f32_to_bf16_bits((gap * math.log(2.0) * math.sqrt(D)).astype(np.float32))
    gap = wl.bf16_bits_to_f32(b.q[:3, :, 0]).astype(np.float64) / (math.log(2.0) * math.sqrt(D))
    v = wl.bf16_bits_to_f32(b.context_v).astype(np.float64)
    run = GpuRun(b, chunk_size=0)
    got = run.step()[:3].astype(np.float64)
    for r, at in enumerate(starts):
        w_first = (1.0 / (1.0 + 2.0 ** gap[r]))[:, None]
        v_first, v_late = (np.repeat(v[at + t], G, axis=0) for t in (first, late))
        want = w_first * v_first + (1.0 - w_first) * v_late
        bound = 2.0 ** -8 * np.abs(want) + 1e-5 * (np.abs(v_first) + np.abs(v_late))
        worst = float((np.abs(got[r] - want) / bound).max())
        assert worst <= 1.0, f"row {r}: error {worst} times its bound"


@pytest.mark.parametrize("chunk", [0, 40], ids=["decode", "mixed"])
def test_a_wait_limit_need_not_cover_a_whole_unit(chunk):
    """The limit of a wait covers the copy of one page. A unit of 6251 pages is streamed by one thread block
    for several times the 300,000 cycles (about 0.15 ms) allowed here, while its scheduler warp, and the
    streaming warps among one another, wait for it: those waits go on as long as pages come in."""
    b = wl.make_batch("limit", wl.Shape(4, 1, 128), [100000] + [0] * (chunk > 0), [1] + [chunk] * (chunk > 0), seed=chunk, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=1 << 20, wait_limit_cycles=300_000)
    assert_parity(run.step(), want, "peaked", "one long unit under a short limit")
    assert np.array_equal(run.pool(), pool_want)
