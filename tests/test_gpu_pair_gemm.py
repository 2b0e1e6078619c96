"""The projections' CTA-pair kernel at the edges of its token tiles (16 to 256 tokens in steps of 16), by itself and
in the layer, where its weight rows come in permuted order: a tile per pair, and so many that every pair takes
three and hands both accumulators over. The layer's narrow and wide tiles, and the one-CTA kernel behind its fused epilogues, are
asserted to be what the plan chooses."""
import math

import numpy as np
import pytest
import torch

import oracle
from oracle import layer as OL
from paper_2512_03416_b200 import binding as B
from paper_2512_03416_b200 import workloads as wl
from paper_2512_03416_b200.harness import LoadedBatch, from_dev, to_dev
from paper_2512_03416_b200.layer import DecoderLayer
from tests.helpers import oracle_pool_with_context
from tests.test_gpu_layer import _need_gpu, bits, make_weights, test_gemm_matches_the_oracle as gemm_matches, test_layer_step_matches_the_oracle as layer_matches  # noqa: F401

pytestmark = pytest.mark.gpu
ROPE, SILU_MUL = 1, 2


@pytest.mark.parametrize("M", [1, 15, 16, 17, 32, 33, 48, 240, 255, 256, 258, 511, 514])
@pytest.mark.parametrize("N,K,residual", [(8, 72, True), (520, 200, False), (1032, 64, True)])
def test_token_tiles(M, N, K, residual):
    gemm_matches((M, N, K, residual), 256)


@pytest.mark.parametrize("M,N,K,residual", [(16, 60008, 72, True), (31, 58000, 200, False), (48, 57352, 136, True), (288, 28808, 64, True),
                                            (512, 28680, 72, False), (2112, 6664, 136, True)], ids=lambda v: str(v))
def test_three_tiles_and_more_per_pair(M, N, K, residual):
    """Tiles of 16, 32, 48, 144, 256 and 240 tokens, more than three per pair of CTAs: each accumulator is filled again
    after its epilogue has let go of it, with one to eight chunks of 32 tokens dealt to two warps."""
    props = torch.cuda.get_device_properties(0)
    assert -(-M // 256) * -(-N // 256) > 3 * (props.multi_processor_count // 2)
    gemm_matches((M, N, K, residual), 256)


@pytest.mark.parametrize("ctx,ql", [([3], [1]), ([5, 0], [1, 15]), ([5, 0], [1, 16]), ([0, 9], [40, 1]), ([0], [241]), ([11, 0], [1, 256]),
                                    ([0, 70], [290, 1])], ids=lambda v: "-".join(map(str, v)))
def test_layer_over_token_tiles(ctx, ql):
    """Steps of few tiles, which the plan keeps narrow (at most 128 tokens)."""
    layer_matches(wl.Shape(4, 2, 128), 320, 384, ctx, ql)      # the last feature tile of the output projection is ragged


def _assert_rows(got, want, rel, what):
    """Every token's row of a bf16 tensor within `rel` in the 2-norm: one value that sits in another feature's or token's
    place moves a row of n values by about sqrt(2 / n), 2 % and more here."""
    g, w = OL.bits_to_f64(got).reshape(len(got), -1), OL.bits_to_f64(want).reshape(len(want), -1)
    assert np.isfinite(g).all(), f"{what}: non-finite"
    err = np.linalg.norm(g - w, axis=1) / np.linalg.norm(w, axis=1)
    assert err.max() <= rel, f"{what}: token {int(err.argmax())} off by {err.max()}"


def _check_layer(s, inter, rows, tokens):
    """One step of `rows` fresh rows of `tokens` tokens each: q, k, v, y, z and the output against the layer's definition."""
    hidden, N = 128, rows * tokens
    rng = np.random.default_rng(N + inter)
    b = wl.make_batch("wide", s, [0] * rows, [tokens] * rows, seed=N, profile="peaked", chunk_size=N)
    wt = make_weights(rng, s, hidden, inter)
    for k in ("w_norm1", "w_norm2"):
        wt[k] = wl.f32_to_bf16_bits((1.0 + wl.bf16_bits_to_f32(wt[k])).astype(np.float32))
    x = bits(rng, (N, hidden), 1.0)
    pool, tm = oracle_pool_with_context(b), b.table_matrix()

    def attention(q, k, v):
        return oracle.mixed_step(pool, s.Hq, s.Hkv, s.D, s.P, 1.0 / math.sqrt(s.D), tm, b.ctx_len, b.q_len, q, k, v)

    want, mid = OL.layer_step(attention, x, wt, OL.positions(b.ctx_len, b.q_len), s.Hq, s.Hkv, s.D, eps=1e-5, theta=500000.0)
    lb = LoadedBatch(b)
    dev = {k: to_dev(v) for k, v in wt.items()}
    layer = DecoderLayer(lb.dec, dev["w_norm1"], dev["w_qkv"], dev["w_o"], dev["w_norm2"], dev["w_gate"], dev["w_up"],
                         dev["w_down"], max_position=64, rms_eps=1e-5, rope_theta=500000.0)
    x_out = torch.full((N, hidden), 0x7FC0, dtype=torch.int16, device="cuda")
    layer.step(lb.slots, b.q_len.tolist(), b.ctx_len.tolist(), to_dev(x), x_out)
    torch.cuda.synchronize()
    assert lb.dec.device_status() == 0
    # the activations are the last part of the layer's workspace, in this order (rows of 256 bytes and more: no gaps)
    ws, at, got = layer.workspace.cpu().numpy().view(np.uint16), layer.workspace.numel() // 2, {}
    qd, kvd = s.Hq * s.D, s.Hkv * s.D
    for name, width in (("z", inter), ("y", hidden), ("a", qd), ("v", kvd), ("k", kvd), ("q", qd)):
        got[name] = ws[at - N * width:at].reshape(N, width)
        at -= N * width
    # q, k, v: a normalised input that rounds the other way (fp32 against 64 bits) is one spacing, at most 2^-7 of
    # that input; the sums follow it by less, and they are then rounded themselves, at most 2^-8 apart.
    for name in "qkv":
        _assert_rows(got[name], mid[name], 2.0 ** -7, name)
    # z and the output: what test_layer_step_matches_the_oracle allows for the chain of tensors in front of them, half of it
    # for z, which is three tensors further to the front
    _assert_rows(got["z"], mid["z"], 1e-2, "z")
    _assert_rows(from_dev(x_out), want, 2e-2, "out")
    layer.close()


# heads of Q and of K/V, intermediate size, rows, tokens per row, tokens of a tile of the QKV and of the gate/up product
WIDE = [(45, 15, 9472, 26, 5, 144, 144), (49, 49, 9600, 25, 10, 256, 256), (45, 15, 9472, 48, 10, 160, 240),
        (33, 11, 4736, 70, 30, 224, 224), (33, 11, 4736, 80, 32, 256, 256), (45, 15, 9472, 64, 33, 240, 240)]


@pytest.mark.parametrize("Hq,Hkv,inter,rows,tokens,nt_qkv,nt_gu", WIDE, ids=lambda v: str(v))
def test_layer_over_wide_token_tiles(Hq, Hkv, inter, rows, tokens, nt_qkv, nt_gu):
    """Tiles of more than 128 tokens through the rotary and the SiLU epilogue, in the steps of more than 2000 tokens more
    than three per pair; odd numbers of heads, where the second CTA of the last pair of heads has none."""
    N, pairs = rows * tokens, torch.cuda.get_device_properties(0).multi_processor_count // 2
    assert (Hq + 2 * Hkv) % 2 == 1
    for n_out, epi, nt in (((Hq + 2 * Hkv) * 128, ROPE, nt_qkv), (2 * inter, SILU_MUL, nt_gu)):
        assert B.ts_gemm_plan(0, N, n_out, 128, epi) == (B.TS_OK, (256, 0, nt))
        assert N < 2000 or -(-N // nt) * -(-n_out // 256) > 3 * pairs
    _check_layer(wl.Shape(Hq, Hkv, 128), inter, rows, tokens)


@pytest.mark.parametrize("rows,tokens", [(1, 2), (5, 7), (16, 8)], ids=lambda v: str(v))
def test_layer_with_fused_epilogues_on_single_ctas(rows, tokens):
    """Few tokens and more feature tiles than there are pairs, but not more than SMs: gemm_kernel's rotary and SiLU epilogues."""
    s, inter = wl.Shape(128, 16, 128), 9728
    for n_out, epi in ((160 * 128, ROPE), (2 * inter, SILU_MUL)):
        assert B.ts_gemm_plan(0, rows * tokens, n_out, 128, epi) == (B.TS_OK, (128, 0, 0))
    _check_layer(s, inter, rows, tokens)


@pytest.mark.parametrize("M", [129, 130, 192, 256])
def test_products_of_few_tiles_split_k(M):
    """A 2048 x 2048 product of a few hundred tokens: four CTAs on a tile's K range (10.6 us) and not pairs (13 us)."""
    assert B.ts_gemm_plan(0, M, 2048, 2048, 0) == (B.TS_OK, (128, 4, 0))
    gemm_matches((M, 2048, 2048, True), 0)


def test_plan_refuses_what_is_no_product():
    for args in ((0, 256, 64, 0), (1, 0, 64, 0), (1, 256, 0, 0), (1, 256, 64, 3), (1, 256, 64, -1)):
        assert B.ts_gemm_plan(0, *args)[0] == B.TS_ERR_INVALID
