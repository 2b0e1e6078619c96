"""The limit of the kernels' waits covers this launch, not what is left of the launch in front of it: a step whose thread blocks
start early, next to a long launch, does not raise a time-out."""
import numpy as np
import pytest
import torch

from paper_2512_03416_b200 import workloads as wl
from paper_2512_03416_b200.harness import from_dev, to_dev
from paper_2512_03416_b200.layer import DecoderLayer
from tests.helpers import GpuRun
from tests.test_gpu_layer import bits, make_weights

pytestmark = pytest.mark.gpu

LIMIT = 300_000          # clock cycles, about 0.15 ms


@pytest.fixture(autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")


@pytest.fixture(scope="module")
def long_launch():
    """One row of 240,000 keys in one piece: a single thread block, 1.5 ms and more, next to which all other SMs are free."""
    b = wl.make_batch("long", wl.Shape(4, 1, 128), [240_000], [1], seed=1, profile="peaked")
    run = GpuRun(b, chunk_size=0, decode_split_tokens=1 << 20)
    run.step(keep_len=True)
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    run.lb.step(keep_len=True)
    end.record()
    torch.cuda.synchronize()
    assert start.elapsed_time(end) > 4 * LIMIT / 1.9e6, "no longer than the limit of the launches behind it"
    return run


@pytest.mark.parametrize("ctx,ql", [([0], [700]), ([300, 40, 5000, 0], [1, 1, 1, 700])], ids=["chunk", "mixed"])
def test_tiles_behind_a_long_launch(long_launch, ctx, ql):
    run = GpuRun(wl.make_batch("tiles", wl.LLAMA8B, ctx, ql, seed=len(ctx), profile="peaked"), chunk_size=0, wait_limit_cycles=LIMIT)
    want = run.step(keep_len=True)
    for _ in range(3):
        long_launch.lb.step(keep_len=True)
        run.lb.step(keep_len=True)
        assert run.dec.device_status() == 0
        assert np.array_equal(run.lb.output(), want)
    assert long_launch.dec.device_status() == 0


@pytest.mark.parametrize("ctx,ql", [([40, 0, 7], [1, 33, 1]), ([40, 0], [1, 1100])], ids=["few-tokens", "many-tokens"])
def test_projections_behind_a_long_launch(long_launch, ctx, ql):
    """The norm's thread blocks, one per token, all start next to the long launch, so that the projection behind them does too."""
    s, hidden, inter, n = wl.Shape(8, 2, 128), 512, 1024, sum(ql)
    run = GpuRun(wl.make_batch("layer", s, ctx, ql, seed=n, profile="peaked"), chunk_size=n, wait_limit_cycles=LIMIT)
    rng = np.random.default_rng(n)
    dev = {k: to_dev(v) for k, v in make_weights(rng, s, hidden, inter).items()}
    layer = DecoderLayer(run.dec, dev["w_norm1"], dev["w_qkv"], dev["w_o"], dev["w_norm2"], dev["w_gate"], dev["w_up"], dev["w_down"], max_position=4096)
    x_in = to_dev(bits(rng, (n, hidden), 1.0))
    x_out = torch.empty_like(x_in)
    layer.step(run.slots, ql, ctx, x_in, x_out, keep_len=True)
    want = from_dev(x_out)
    for _ in range(3):
        long_launch.lb.step(keep_len=True)
        layer.step(run.slots, ql, ctx, x_in, x_out, keep_len=True)
        assert run.dec.device_status() == 0
        assert np.array_equal(from_dev(x_out), want)
    layer.close()
