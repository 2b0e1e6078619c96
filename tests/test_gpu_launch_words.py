"""GPU parity of steps whose row arrays and work list just fit into the launch parameters, or no longer do."""
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


def words(rows, items, combines):
    return -(-(3 * rows + 1) // 8) * 8 + 8 * items + 4 * combines


@pytest.mark.parametrize("chunk", [0, 5], ids=["decode", "mixed"])
@pytest.mark.parametrize("rows", [69, 70, 279, 280, 698, 699])
def test_steps_around_the_sizes_of_the_launch_parameters(rows, chunk):
    """One work item per row, the chunk's row included: 69, 279 and 698 rows are the most that 768, 3072 and 7680 words
    hold. Beyond the last the metadata are uploaded."""
    limit = {69: 768, 70: 768, 279: 3072, 280: 3072, 698: 7680, 699: 7680}[rows]
    decode = rows - (chunk > 0)
    ctx, ql = [(37 * i) % 61 for i in range(decode)] + [9] * (chunk > 0), [1] * decode + [chunk] * (chunk > 0)
    b = wl.make_batch("words", wl.Shape(4, 1, 128), ctx, ql, seed=rows, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    n_items = len(run.dec.plan_step(run.slots, ql, ctx))
    assert n_items == rows and (words(rows, n_items, 0) <= limit) == (rows in (69, 279, 698))
    for _ in range(2):
        assert_parity(run.step(keep_len=True), want, "peaked", f"{rows} rows")
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("heads", [(4, 1, 128), (16, 1, 128), (2, 1, 64)], ids=["4-1", "16-1", "d64"])
def test_the_longest_merge_list_that_gets_a_launch_of_its_own(heads, more):
    """Rows in two splits each on two thirds of the SMs, and one row more, whose splits the decode launch merges. The list is
    part of the launch parameters (4-1: of a step of more than 768 words) or of the uploaded metadata."""
    rows = 2 * torch.cuda.get_device_properties(0).multi_processor_count // 3 // 2 + more
    assert words(rows, 2 * rows, rows) > 768
    b = wl.make_batch("merges", wl.Shape(*heads), [70 + i % 50 for i in range(rows)], [1] * rows, seed=rows, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    run.step(keep_len=True)                                # brings block-table entries along
    before = run.dec.velocity()["kernel_launches"]
    assert_parity(run.step(keep_len=True), want, "peaked", f"{rows} split rows")
    assert run.dec.velocity()["kernel_launches"] - before == (1 if more else 2)
    assert np.array_equal(run.pool(), pool_want)


def test_the_longest_merge_list_of_a_small_step():
    """head_dim 64: a tile and as many rows in two splits as the SMs take next to it, merged by a launch of their own."""
    rows = (torch.cuda.get_device_properties(0).multi_processor_count - 1) // 2
    ctx, ql = [70 + i % 50 for i in range(rows)] + [3], [1] * rows + [5]
    b = wl.make_batch("merges", wl.Shape(2, 1, 64), ctx, ql, seed=rows, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    run.step(keep_len=True)
    before = run.dec.velocity()["kernel_launches"]
    assert_parity(run.step(keep_len=True), want, "peaked", f"{rows} split rows")
    assert run.dec.velocity()["kernel_launches"] - before == 2
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("rows", [192, 193])
@pytest.mark.parametrize("heads", [(4, 1, 128), (16, 1, 128), (2, 1, 64)], ids=["4-1", "16-1", "d64"])
def test_merges_of_many_rows_inside_the_decode_launch(rows, heads):
    """Rows in two splits each, more units than SMs: items and merges as launch parameters (4-1) and uploaded."""
    b = wl.make_batch("merges", wl.Shape(*heads), [70 + i % 50 for i in range(rows)], [1] * rows, seed=rows, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    for _ in range(2):
        assert_parity(run.step(keep_len=True), want, "peaked", f"{rows} split rows")
    assert np.array_equal(run.pool(), pool_want)
