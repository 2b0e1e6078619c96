"""GPU parity of the prefill tiles where the reference maximum of a row moves: P of a block of 128 keys goes to the
tensor cores in two parts, and the move has to be made before the first."""
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


@pytest.mark.parametrize("shape", [wl.LLAMA8B, wl.Shape(6, 2, 128)], ids=["32-8", "6-2"])
@pytest.mark.parametrize("at", [0, 47, 48, 63, 64, 111, 112, 127])
def test_a_new_maximum_anywhere_in_a_block(shape, at):
    """Key `at` of every block is 2^12 times as heavy as that of the block before it, for every second token: its row
    moves its reference in each block, its neighbours' keep theirs. `at` is the first and last key of each part."""
    b = wl.make_batch("move", shape, [700, 131], [40, 2], seed=at + shape.Hq, profile="peaked")
    pos = np.concatenate([np.arange(700), np.arange(131)])
    step = 12.0 * np.sqrt(shape.D) / (8.0 * np.log2(np.e))
    k = wl.bf16_bits_to_f32(b.context_k)
    k[:, :, 0] = np.where(pos % 128 == at, (1 + pos // 128) * step, 0.0)[:, None]
    b.context_k[:] = wl.f32_to_bf16_bits(k.astype(np.float32))
    q = wl.bf16_bits_to_f32(b.q)
    q[:, :, 0] = np.where(np.arange(len(q)) % 2 == 0, 8.0, 0.0)[:, None]
    b.q[:] = wl.f32_to_bf16_bits(q.astype(np.float32))
    want, pool_want = oracle_step(b)
    run = GpuRun(b, chunk_size=0)
    assert_parity(run.step(), want, "needle", f"key {at}")
    assert np.array_equal(run.pool(), pool_want)
