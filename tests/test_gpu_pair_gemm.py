"""The projections' CTA-pair kernel at the edges of its token tiles (16 to 256 tokens in steps of 16, as many
tiles as the shape asks for), by itself and in the layer, where its weight rows come in permuted order."""
import pytest

from paper_2512_03416_b200 import workloads as wl
from tests.test_gpu_layer import _need_gpu, test_gemm_matches_the_oracle as gemm_matches, test_layer_step_matches_the_oracle as layer_matches  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 15, 16, 17, 32, 33, 48, 240, 255, 256, 258, 511, 514])
@pytest.mark.parametrize("N,K,residual", [(8, 72, True), (520, 200, False), (1032, 64, True)])
def test_token_tiles(M, N, K, residual):
    gemm_matches((M, N, K, residual), 256)


@pytest.mark.parametrize("ctx,ql", [([3], [1]), ([5, 0], [1, 15]), ([5, 0], [1, 16]), ([0, 9], [40, 1]), ([0], [241]), ([11, 0], [1, 256]),
                                    ([0, 70], [290, 1])], ids=lambda v: "-".join(map(str, v)))
def test_layer_over_token_tiles(ctx, ql):
    layer_matches(wl.Shape(4, 2, 128), 320, 384, ctx, ql)      # the last feature tile of the output projection is ragged
