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
    """One work item per row: 69, 279 and 698 decode rows are the most that 768, 3072 and 7680 words hold. Beyond the last
    the metadata are uploaded."""
    limit = {69: 768, 70: 768, 279: 3072, 280: 3072, 698: 7680, 699: 7680}[rows]
    assert (words(rows, rows, 0) <= limit) == (rows in (69, 279, 698))
    ctx = [(37 * i) % 61 for i in range(rows)]
    b = wl.make_batch("words", wl.Shape(4, 1, 128), ctx + [9] * (chunk > 0), [1] * rows + [chunk] * (chunk > 0), seed=rows, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    for _ in range(2):
        assert_parity(run.step(keep_len=True), want, "peaked", f"{rows} rows")
    assert np.array_equal(run.pool(), pool_want)


@pytest.mark.parametrize("rows", [192, 193])
@pytest.mark.parametrize("heads", [(4, 1, 128), (16, 1, 128), (2, 1, 64)], ids=["4-1", "16-1", "d64"])
def test_more_split_rows_than_the_merges_parameters_hold(rows, heads):
    """192 rows in two splits each are the most whose merge list travels with its launch."""
    b = wl.make_batch("merges", wl.Shape(*heads), [70 + i % 50 for i in range(rows)], [1] * rows, seed=rows, profile="peaked")
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0, decode_split_tokens=64)
    for _ in range(2):
        assert_parity(run.step(keep_len=True), want, "peaked", f"{rows} split rows")
    assert np.array_equal(run.pool(), pool_want)
