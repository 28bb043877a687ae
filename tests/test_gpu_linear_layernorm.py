"""GPU parity (bit-exact) of linear + residual + i-LayerNorm as one operation against the oracle's
linear layer (Q16 output) followed by its i-LayerNorm (Sec. 3.6, Eq. 16).  With the fusion forced, shapes with N a
multiple of 256 run the 128-row cluster kernel and the others the two kernels back to back; by size, few rows run
the small-row cluster kernel."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_same, ctx, dev, host
from paper_2101_01321_b200 import synth

pytestmark = pytest.mark.gpu


def _problem(M, N, K, seed, res_ratio=0.5):
    rng = np.random.default_rng(seed)
    x = rng.integers(-127, 128, (M, K)).astype(np.int8)
    w = rng.integers(-127, 128, (N, K)).astype(np.int8)
    bias = rng.integers(-200000, 200000, N).astype(np.int32)
    res = rng.integers(-127, 128, (M, N)).astype(np.int8)
    S_w = rng.uniform(1e-4, 4e-4, N)
    S_x = 0.03
    amax = 127.0 * 127.0 * np.sqrt(K) * 1.2 * S_x * 2.5e-4       # a few standard deviations of the product
    S_mid = 1.5 * amax / 32767.0
    S_res = res_ratio * amax / 127.0
    gamma = 1.0 + 0.1 * rng.standard_normal(N)
    beta = 0.1 * rng.standard_normal(N)
    S_out = 4.5 / 127.0
    return x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out


def _oracle(x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out):
    mid = oracle.linear(x, S_x, w, S_w, bias, 1, S_mid)
    want, _ = oracle.layernorm(mid, S_mid, res, S_res, gamma, beta, S_out)
    return want


# (rows, channels, reduction): 1..7 CTAs per cluster, ragged row tiles, several tiles per cluster,
# reduction lengths that are not multiples of the 128-byte K block, and shapes the cluster kernel
# does not take (channels not a multiple of 256)
SHAPES = [(1, 256, 64), (127, 256, 128), (300, 512, 144), (129, 768, 768), (1000, 768, 3072), (260, 1024, 1024),
          (515, 1024, 4096), (70, 1280, 256), (40, 1792, 128), (20000, 256, 64), (9000, 768, 256),
          (77, 128, 64), (300, 320, 80), (0, 768, 768)]


@pytest.fixture(autouse=True)
def _restore_fusion_mode():
    yield
    ctx().ibert_set_fusion(0)


@pytest.mark.parametrize("mode", [1, 2, 0])       # cluster kernel forced, two kernels forced, by size
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_linear_layernorm_matches_oracle(M, N, K, mode):
    p = _problem(M, N, K, M + N + K)
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    ctx().ibert_set_fusion(mode)
    out, S_ret = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res,
                                                 gamma, beta, S_out)
    ctx().check()
    assert S_ret == S_out
    if M:
        want = _oracle(*p)
        assert_same(host(out), want, f"linear+LN {M}x{N}x{K} mode {mode}")
        assert np.abs(want).max() > 20


def test_linear_layernorm_constant_rows_and_no_bias():
    """Rows whose pre-LayerNorm values are all equal (variance 0: the standard deviation floor of 1
    applies) and a call without bias."""
    M, N, K = 140, 512, 128
    p = list(_problem(M, N, K, 5))
    p[0][:70] = 0                       # x = 0 -> accumulators = bias
    p[2][:] = 1234                      # the same bias everywhere
    p[3][:70] = 7                       # constant residual
    p[4][:] = 2e-4                      # one weight scale: every channel requantizes alike
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    ctx().ibert_set_fusion(1)
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res,
                                             gamma, beta, S_out)
    ctx().check()
    assert_same(host(out), _oracle(*p), "constant rows")
    p[2] = None
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, None, S_mid, dev(res), S_res,
                                             gamma, beta, S_out)
    ctx().check()
    assert_same(host(out), _oracle(*p), "no bias")


def test_linear_layernorm_equals_the_two_separate_calls():
    M, N, K = 700, 768, 768
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = _problem(M, N, K, 11)
    c = ctx()
    c.ibert_set_fusion(1)
    fused, _ = c.ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res,
                                           gamma, beta, S_out)
    mid, _ = c.ibert_linear_i8(dev(x), S_x, dev(w), S_w, dev(bias), 1, S_mid)
    two, _ = c.ibert_layernorm_i(mid, S_mid, dev(res), S_res, gamma, beta, S_out)
    c.check()
    assert_same(host(fused), host(two), "fused vs separate")


# 768 channels: 192 instead of 256 per CTA while that shortens the rounds of token tiles -- one full round, one tile
# more (256 again), a second round that starts, one that is full, and the third (a short reduction only)
@pytest.mark.parametrize("M,K", [(4224, 128), (4225, 128), (5633, 256), (8448, 144), (12161, 128), (12161, 896)])
def test_linear_layernorm_rounds_of_narrow_tiles(M, K):
    p = _problem(M, 768, K, M + K)
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    ctx().ibert_set_fusion(1)
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res,
                                             gamma, beta, S_out)
    ctx().check()
    assert_same(host(out), _oracle(*p), f"linear+LN {M}x768x{K}")


@pytest.mark.parametrize("B", [32, 64])
def test_encoder_layer_rounds_of_narrow_tiles(B):
    """FFN2 of 192 channels per CTA, its activations in the transposed layout."""
    L, H, F = 128, 768, 256
    x, params = synth.make_model(0, B, layers=1, H=H, heads=12, F=F, L=L)
    layer = ctx().ibert_layer_create(params[0])
    out, _ = ctx().ibert_encoder_layer(layer, dev(x), B, L)
    ctx().check()
    layer.close()
    assert_same(host(out), oracle.encoder_layer(params[0], x, B, L).out, f"encoder layer {B}x{L}")


# sizes at which two kernels need fewer rounds of tiles than the clusters, chosen by size alone; the third
# row has a tile of tokens too many
@pytest.mark.parametrize("M,N,K", [(4225, 1024, 256), (4600, 1024, 1040), (4609, 1024, 256), (18900, 768, 256)])
def test_linear_layernorm_by_rounds_of_tiles(M, N, K):
    p = _problem(M, N, K, M + N + K)
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res,
                                             gamma, beta, S_out)
    ctx().check()
    assert_same(host(out), _oracle(*p), f"linear+LN {M}x{N}x{K}")


# residual scales from 0.34 to about 1000 times the sum's: the multiply-high form exists for none below 1/2 (its offset
# is half a unit of the result), for all tried up to 32 and for fewer and fewer above
@pytest.mark.parametrize("res_ratio", [0.002, 0.011, 0.13, 0.7, 2.9, 5.1, 5.3, 5.5, 5.7, 5.9])
def test_linear_layernorm_residual_forms(res_ratio):
    M, N, K = 5000, 768, 128
    p = _problem(M, N, K, 77, res_ratio)
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    ctx().ibert_set_fusion(1)
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res,
                                             gamma, beta, S_out)
    ctx().check()
    assert_same(host(out), _oracle(*p), f"residual at {S_res / S_mid:.3g} times the scale of the sum")


@pytest.mark.parametrize("M,N,K", [(1, 256, 64), (129, 256, 128), (300, 512, 144), (515, 768, 272), (260, 1024, 128),
                                   (20000, 256, 64), (9000, 768, 256), (7000, 1024, 64)])
def test_linear_layernorm_residual_below_the_sums_scale(M, N, K):
    """No multiply-high form: the epilogue in 16 columns at a time for pairs of tiles (and single ones of 256 channels);
    the last three have several tiles per cluster."""
    p = _problem(M, N, K, M, 0.002)
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    assert S_res < 0.5 * S_mid
    ctx().ibert_set_fusion(1)
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res, gamma, beta, S_out)
    ctx().check()
    assert_same(host(out), _oracle(*p), f"linear+LN {M}x{N}x{K}")


@pytest.mark.parametrize("ratio", [1.0, 37.0, 1500.0])          # |v| up to 127, 4699 and 190500
# K = 64: two kernels by size, the large-tile cluster kernel when forced; K = 256 by size: the one-wave cluster kernel with
# 16 tokens per tile (one per warp) and with 32, 48 and 64
@pytest.mark.parametrize("M,N,mode,K", [(9, 256, 0, 64), (130, 768, 0, 64), (130, 768, 1, 64), (257, 1024, 1, 64),
                                        (300, 256, 1, 64), (16, 768, 0, 256), (321, 768, 0, 256), (600, 768, 0, 256),
                                        (900, 768, 0, 256), (1300, 768, 0, 256), (130, 256, 0, 256), (700, 1024, 0, 256)])
def test_variances_at_perfect_squares(M, N, mode, K, ratio):
    """Zero projection and rows of +-a: the sum of squares is a^2 C, the largest value of one square root below the next;
    one element more or less, and rows of a single value or none, sit on either side of a root's step."""
    rng = np.random.default_rng(N + M)
    x, w = np.zeros((M, K), np.int8), rng.integers(-127, 128, (N, K)).astype(np.int8)
    a = rng.integers(0, 128, (M, 1))
    res = np.where(np.arange(N) % 2 == 0, a, -a)
    res[1::4, 0] = np.maximum(res[1::4, 0] - 1, -127)
    res[2::4, 1] = np.minimum(res[2::4, 1] + 1, 127)
    res[3::4] = 0
    res[3::8, 5] = 1
    res = res.astype(np.int8)
    S_w, S_mid, bias = np.full(N, 2e-4), 1e-3, np.zeros(N, np.int32)
    gamma, beta = 1.0 + 0.1 * rng.standard_normal(N), 0.1 * rng.standard_normal(N)
    ctx().ibert_set_fusion(mode)
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), 0.03, dev(w), S_w, dev(bias), S_mid, dev(res), ratio * S_mid, gamma, beta, 4.5 / 127)
    ctx().check()
    want, _ = oracle.layernorm(oracle.linear(x, 0.03, w, S_w, bias, 1, S_mid), S_mid, res, ratio * S_mid, gamma, beta, 4.5 / 127)
    assert_same(host(out), want, "linear + LayerNorm at perfect squares")


@pytest.mark.parametrize("M,N,K", [(700, 512, 64), (600, 768, 64), (600, 1024, 64)])       # pairs, 192 channels per CTA, single CTAs
def test_linear_layernorm_bias_of_the_kernel_before(M, N, K):
    """A bias written on the stream directly in front of the call, another one every time."""
    p = _problem(M, N, K, 31)
    x, w, bias, res, S_w, S_x, S_mid, S_res, gamma, beta, S_out = p
    c = ctx()
    c.ibert_set_fusion(1)
    xd, wd, rd, bd = dev(x), dev(w), dev(res), dev(bias)
    own = torch.empty_like(bd)
    for i in range(12):
        torch.add(bd, 50000 * i, out=own)
        out, _ = c.ibert_linear_layernorm_i8(xd, S_x, wd, S_w, own, S_mid, rd, S_res, gamma, beta, S_out)
        torch.add(bd, -7, out=own)
        if i % 4 == 3:
            want = _oracle(x, w, (bias + 50000 * i).astype(np.int32), res, S_w, S_x, S_mid, S_res, gamma, beta, S_out)
            assert_same(host(out), want, f"bias {i}")
    c.check()
