"""GPU parity of head_dim 64 steps around the size up to which tiles and decode units share a launch."""
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


@pytest.mark.parametrize("shape", [wl.Shape(4, 1, 64), wl.Shape(16, 1, 64), wl.Shape(6, 2, 64)], ids=["4-1", "16-1", "6-2"])
@pytest.mark.parametrize("over", [0, 1])
def test_tiles_and_decode_units_of_head_dim_64_in_one_launch(shape, over):
    """One block per (item, KV head): a chunk of three items and the rows that just fill the SMs, or one row more."""
    chunk = 3 * (64 // (shape.Hq // shape.Hkv)) - 1
    rows = sms() // shape.Hkv - 3 + over
    b = wl.make_batch("small", shape, [(29 * i) % 300 for i in range(rows)] + [21], [1] * rows + [chunk], seed=rows, profile="peaked")
    check(b, 2 if over else 1)


def test_split_rows_of_a_small_step_are_merged():
    b = wl.make_batch("small", wl.Shape(4, 2, 64), [300, 64, 63, 150, 0], [1] * 4 + [70], seed=3, profile="peaked")
    check(b, 2, decode_split_tokens=64)


@pytest.mark.parametrize("last", [8191, 8192])
def test_long_tiles_have_a_launch_of_their_own(last):
    """A tile that sees 8192 keys, and one more."""
    b = wl.make_batch("small", wl.Shape(4, 2, 64), [300, 5, last - 39], [1, 1, 40], seed=last, profile="peaked")
    check(b, 1 if last == 8191 else 2)
