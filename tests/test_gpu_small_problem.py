"""GPU parity (bit-exact) of the one-wave kernels for small token counts against the oracle, at the edges of
their tiles (16-token tiles of 128 channels, 256-byte K stages, 8- to 32-column softmax slices) and at the
ends of the range they are chosen for; the first sizes past it run the large-tile kernels."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, ctx, dev, host
from paper_2101_01321_b200 import synth

pytestmark = pytest.mark.gpu


def _linear_problem(M, N, K, seed):
    rng = np.random.default_rng(seed)
    x = rng.integers(-127, 128, (M, K)).astype(np.int8)
    w = rng.integers(-127, 128, (N, K)).astype(np.int8)
    bias = rng.integers(-200000, 200000, N).astype(np.int32)
    S_w = rng.uniform(1e-4, 4e-4, N)
    S_x = 0.03
    return x, w, bias, S_w, S_x, 127.0 * 127.0 * np.sqrt(K) * 1.2 * S_x * 2.5e-4


# one token; a tile and one past it; channel and K tails; the longest ring; the largest one-wave sizes of a wide
# and a narrow layer and the first size past each
@pytest.mark.parametrize("M,N,K", [(1, 128, 256), (16, 144, 272), (17, 2304, 768), (33, 272, 400), (129, 768, 3072),
                                   (50, 4096, 1024), (113, 320, 4096), (576, 3072, 768), (577, 3072, 768), (768, 3072, 768), (769, 3072, 768),
                                   (1024, 2304, 768), (1025, 2304, 768)])
def test_linear_kinds(M, N, K):
    x, w, bias, S_w, S_x, amax = _linear_problem(M, N, K, M + N + K)
    for kind, S_out in ((0, amax / 100.0), (1, amax / 20000.0), (2, 0.0), (3, amax / 20000.0)):
        out, _ = ctx().ibert_linear_i8(dev(x), S_x, dev(w), S_w, dev(bias), kind, S_out)
        assert_same(host(out), oracle.linear(x, S_x, w, S_w, bias, 1 if kind == 3 else kind, S_out), f"kind {kind}")
    S_mid, S_in, S_out = 6.0 / 32767.0, S_x * (6.0 / amax), 6.0 / 127.0
    mid = oracle.linear(x, S_in, w, S_w, bias, 1, S_mid)
    out, _ = ctx().ibert_linear_gelu_i8(dev(x), S_in, dev(w), S_w, dev(bias), S_mid, S_out)
    assert_same(host(out), oracle.gelu(mid, S_mid, S_out)[0], "gelu")
    out, _ = ctx().ibert_linear_hgelu_i8(dev(x), S_in, dev(w), S_w, dev(bias), S_mid, S_out)
    assert_same(host(out), oracle.hgelu(mid, S_mid, S_out)[0], "hgelu")
    ctx().check()


# layers whose QKV or FFN1 GEMM has the widest one-wave tiles (112 and 128 tokens), which only layer-owned weights take
@pytest.mark.parametrize("B,L", [(8, 109), (8, 125), (5, 151), (9, 114)])
def test_encoder_layer_widest_tiles(B, L):
    x, params = synth.make_model(0, B, layers=1, H=768, heads=12, F=3072, L=L)
    layer = ctx().ibert_layer_create(params[0])
    out, _ = ctx().ibert_encoder_layer(layer, dev(x), B, L)
    ctx().check()
    layer.close()
    assert_same(host(out), oracle.encoder_layer(params[0], x, B, L).out, f"encoder layer {B}x{L}")


# 1, 2, 3, 5, 6 and 8 CTAs per cluster (channel counts that are and are not powers of two); 1 to 4 tokens per warp
@pytest.mark.parametrize("M,N,K", [(1, 768, 768), (16, 128, 256), (17, 256, 272), (321, 768, 3072), (400, 384, 512),
                                   (500, 640, 512), (700, 768, 768), (1000, 768, 768), (241, 1024, 4096),
                                   (900, 1024, 1024), (1300, 1024, 1024)])
@pytest.mark.parametrize("constant_rows", [False, True])
def test_linear_layernorm(M, N, K, constant_rows):
    x, w, bias, S_w, S_x, amax = _linear_problem(M, N, K, M + N + K)
    rng = np.random.default_rng(M)
    res = rng.integers(-127, 128, (M, N)).astype(np.int8)
    if constant_rows:                    # variance 0: the standard deviation's floor of 1 applies
        x[: M // 2 + 1], res[: M // 2 + 1], bias[:], S_w[:] = 0, 7, 1234, 2e-4
    S_mid, S_res, S_out = 1.5 * amax / 32767.0, 0.5 * amax / 127.0, 4.5 / 127.0
    gamma, beta = 1.0 + 0.1 * rng.standard_normal(N), 0.1 * rng.standard_normal(N)
    out, _ = ctx().ibert_linear_layernorm_i8(dev(x), S_x, dev(w), S_w, dev(bias), S_mid, dev(res), S_res, gamma, beta, S_out)
    ctx().check()
    mid = oracle.linear(x, S_x, w, S_w, bias, 1, S_mid)
    assert_same(host(out), oracle.layernorm(mid, S_mid, res, S_res, gamma, beta, S_out)[0], "linear + LayerNorm")


# four, two and one copies of the queries; 8, 16 and 32 columns per thread; lengths around multiples of 32; the
# first pair count past the range; score scales with and without a pre-shift, and an exact ln2 / 2^k
@pytest.mark.parametrize("B,L,heads", [(1, 1, 1), (1, 31, 2), (2, 33, 3), (1, 128, 12), (3, 129, 2), (2, 256, 4),
                                       (1, 257, 2), (1, 512, 16), (8, 77, 12), (12, 100, 12), (24, 128, 12), (25, 128, 12)])
@pytest.mark.parametrize("S_qk", [0.02, 0.004, float(np.sqrt(8.0 * np.log(2.0) / 2.0 ** 14))])
def test_attention(B, L, heads, S_qk):
    H = heads * 64
    rng = np.random.default_rng(B * 1000 + L)
    qkv = np.clip(np.rint(rng.standard_normal((B * L, 3 * H)) * 40), -127, 127).astype(np.int8)
    c = ctx()
    out, _ = c.ibert_attention_i8(dev(qkv), B, L, H, heads, S_qk, S_qk, 0.02, 0.006, 255)
    assert_same(host(out), oracle.attention(qkv, B, L, H, heads, S_qk, S_qk, 0.02, 0.006, 255), "attention")
    lens = rng.integers(0, L + 1, B).astype(np.int32)
    lens[0] = L if B > 1 else max(L - 1, 0)
    want = oracle.attention(qkv, B, L, H, heads, S_qk, S_qk, 0.02, 0.006, 127, lens=lens)
    out, _ = c.ibert_attention_masked_i8(dev(qkv), B, L, H, heads, dev(lens), S_qk, S_qk, 0.02, 0.006, 127)
    assert_same(host(out), want, "masked attention")
    rows = np.concatenate([np.arange(b * L, b * L + n) for b, n in enumerate(lens)]).astype(int)
    if rows.size:
        cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        out, _ = c.ibert_attention_packed_i8(dev(np.ascontiguousarray(qkv[rows])), dev(cu), L, H, heads, S_qk, S_qk, 0.02, 0.006, 127)
        assert_same(host(out), want[rows], "packed attention")
    c.check()
