"""GPU parity (bit-exact) of the standalone integer non-linearities against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_same, ctx, dev, host
from paper_2101_01321_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 3, 5, 1000, 4096, 128 * 128 * 7 + 2, (1 << 20) + 3])
@pytest.mark.parametrize("sigma", [1.0, 4.0])
def test_gelu_matches_oracle(n, sigma):
    q, S, S_out = synth.gelu_inputs(max(n, 1), sigma)
    q = q[:n]
    out, S_ret = ctx().ibert_gelu_i(dev(q), S, S_out)
    ctx().check()
    want, _ = oracle.gelu(q, S, S_out)
    assert S_ret == S_out
    assert_same(host(out), want, "gelu")


def test_gelu_full_int32_range_and_odd_scales():
    rng = np.random.default_rng(3)
    q = np.concatenate([rng.integers(-2 ** 31, 2 ** 31, 50000), np.arange(-40000, 40000),
                        [2 ** 31 - 1, -2 ** 31, 0, 32767, -32767, 32768, -32768]]).astype(np.int32)
    for S, S_out in [(1e-3, 4 / 127), (1.2207e-4, 0.031), (1.5e-4, 0.002), (0.05, 1.0), (3e-6, 1e-3), (2.0, 0.5)]:
        out, _ = ctx().ibert_gelu_i(dev(q), S, S_out)
        want, _ = oracle.gelu(q, S, S_out)
        assert_same(host(out), want, f"gelu S={S}")
    ctx().check()


@pytest.mark.parametrize("rows,L", [(5, 1), (9, 7), (33, 64), (17, 65), (96 * 8, 128), (64, 256), (40, 512),
                                    (7, 1000), (12, 1024), (3, 130), (0, 128),
                                    (6, 4), (1, 128), (1027, 100), (2, 124)])   # short rows: four rows per warp
@pytest.mark.parametrize("p_max", [255, 127])
def test_softmax_matches_oracle(rows, L, p_max):
    for sigma in (1.0, 4.0):
        q, S = synth.softmax_inputs(max(rows, 1), L, sigma)
        q = q[:rows]
        out, S_ret = ctx().ibert_softmax_i(dev(q), S, p_max)
        ctx().check()
        assert S_ret == 1.0 / p_max
        if rows:
            want, _ = oracle.softmax(q, S, p_max)
            assert_same(host(out), want, f"softmax L={L}")


@pytest.mark.parametrize("rows,L", [(9, 7), (96 * 8, 128), (40, 512), (12, 1024), (3, 130)])
def test_softmax_with_exp_by_table_equals_the_integer_kernel(rows, L):
    """The table holds the integer function's own values, so the comparison variant agrees bit for bit."""
    for sigma, p_max in ((1.0, 255), (4.0, 127)):
        q, S = synth.softmax_inputs(rows, L, sigma)
        a, _ = ctx().ibert_softmax_lut_i(dev(q), S, p_max)
        ctx().check()
        assert_same(host(a), oracle.softmax(q, S, p_max)[0], f"softmax by table L={L}")
    rng = np.random.default_rng(L)
    q = rng.integers(-2 ** 31, 2 ** 31, (rows, L)).astype(np.int32)
    q[0] = 3
    for S in (1e-3, 2e-5, 1e-8, 0.69):
        a, _ = ctx().ibert_softmax_lut_i(dev(q), S, 255)
        assert_same(host(a), oracle.softmax(q, S, 255)[0], f"softmax by table S={S}")
    ctx().check()


def test_softmax_extreme_inputs_and_scales():
    rng = np.random.default_rng(5)
    L = 96
    q = rng.integers(-2 ** 31, 2 ** 31, (64, L)).astype(np.int32)
    q[0] = 7
    q[1] = np.arange(L) - 2 ** 31
    q[2, :] = -2 ** 31
    q[2, 5] = 2 ** 31 - 1
    q[3] = rng.integers(-50, 50, L)
    q[4:20] = rng.integers(-3000, 3000, (16, L))
    for S in (1e-3, 4.5e-5, 2e-5, 1e-8, 0.3, 0.69, 3.3e-7):
        out, _ = ctx().ibert_softmax_i(dev(q), S, 255)
        want, _ = oracle.softmax(q, S, 255)
        assert_same(host(out), want, f"softmax S={S}")
    ctx().check()


# the coarsest scales (divisors of the exponential 1 to 3, on both sides of 16) and one whose folded multiplier does not
# exist, at row lengths around the 16-byte vectors and lane groups
@pytest.mark.parametrize("q_ln2", [1, 2, 3, 15, 16, 16716])
@pytest.mark.parametrize("L", [1, 3, 31, 33, 64, 101, 128, 130, 509, 512, 1021, 1024])
def test_softmax_scales_at_the_ends(q_ln2, L):
    S = float(np.log(2.0)) / (q_ln2 + 0.5)
    rng = np.random.default_rng(L)
    q = np.rint(rng.standard_normal((67, L)) * rng.choice([0.5, 2.0, 8.0], (67, 1)) / S).astype(np.int32)
    q[0], q[1], q[2] = -2 ** 31, 2 ** 31 - 1, np.arange(L) - 2 ** 31
    for p_max in (255, 127):
        out, _ = ctx().ibert_softmax_i(dev(q), S, p_max)
        assert_same(host(out), oracle.softmax(q, S, p_max)[0], f"softmax q_ln2={q_ln2} L={L}")
    ctx().check()


@pytest.mark.parametrize("rows,C", [(3, 8), (5, 17), (64, 768), (33, 1024), (4, 2047), (2, 1), (9, 260), (0, 768),
                                    (7, 1536)])
@pytest.mark.parametrize("residual", [True, False])
def test_layernorm_matches_oracle(rows, C, residual):
    for sigma in (1.0, 4.0):
        q, S, r, S_r, gamma, beta, S_out = synth.layernorm_inputs(max(rows, 1), C, sigma, with_residual=residual)
        q = q[:rows]
        r = None if r is None else r[:rows]
        gamma = gamma.copy()
        gamma[::5] *= -1.0
        out, S_ret = ctx().ibert_layernorm_i(dev(q), S, None if r is None else dev(r), S_r, gamma, beta, S_out)
        ctx().check()
        assert S_ret == S_out
        if rows:
            want, _ = oracle.layernorm(q, S, r, S_r or 0.0, gamma, beta, S_out)
            assert_same(host(out), want, f"layernorm C={C}")


@pytest.mark.parametrize("rows,C", [(3, 8), (5, 17), (64, 768), (33, 1024), (4, 2047), (2, 1), (9, 260), (0, 768),
                                    (7, 1536), (300, 512), (11, 774)])
@pytest.mark.parametrize("residual", [True, False])
def test_layernorm_on_int16_q16_matches_oracle(rows, C, residual):
    """ibert_layernorm_i16: the same Q16 values in an int16 container (every kernel variant: streamed
    rows, register rows with and without vector loads) against the same oracle."""
    for sigma in (1.0, 4.0):
        q, S, r, S_r, gamma, beta, S_out = synth.layernorm_inputs(max(rows, 1), C, sigma, with_residual=residual)
        q = q[:rows]
        r = None if r is None else r[:rows]
        assert np.abs(q).max(initial=0) <= 32767
        gamma = gamma.copy()
        gamma[::7] *= -1.0
        out, S_ret = ctx().ibert_layernorm_i(dev(q.astype(np.int16)), S, None if r is None else dev(r), S_r, gamma, beta,
                                             S_out)
        ctx().check()
        assert S_ret == S_out
        if rows:
            want, _ = oracle.layernorm(q, S, r, S_r or 0.0, gamma, beta, S_out)
            assert_same(host(out), want, f"layernorm int16 C={C}")


def test_layernorm_degenerate_rows():
    C = 64
    q = np.zeros((6, C), dtype=np.int32)
    q[0] = 1234                      # constant row: sigma clamps to 1
    q[1, 0] = 2 ** 20                # largest allowed magnitude
    q[2] = np.where(np.arange(C) % 2 == 0, 2 ** 20, -2 ** 20)
    q[3, :] = 1
    q[3, 0] = 0
    q[4] = np.arange(C) - 32
    q[5] = -2 ** 20
    gamma = np.linspace(-1.5, 1.5, C)
    beta = np.linspace(-1.0, 1.0, C)
    out, _ = ctx().ibert_layernorm_i(dev(q), 1e-4, None, 0.0, gamma, beta, 0.02)
    want, _ = oracle.layernorm(q, 1e-4, None, 0.0, gamma, beta, 0.02)
    assert_same(host(out), want, "layernorm degenerate")
    ctx().check()


def test_rowops_error_codes_on_device_context():
    from paper_2101_01321_b200.binding import IbertError
    q = torch.zeros((4, 8), dtype=torch.int32, device="cuda")
    with pytest.raises(IbertError) as e:
        ctx().ibert_softmax_i(q, 0.7)                 # q_ln2 would be 0
    assert e.value.code == -3
    with pytest.raises(IbertError) as e:
        ctx().ibert_softmax_i(torch.zeros((1, 1025), dtype=torch.int32, device="cuda"), 1e-3)
    assert e.value.code == -2
    with pytest.raises(IbertError) as e:
        ctx().ibert_gelu_i(q, -1.0, 0.03)
    assert e.value.code == -3
    with pytest.raises(IbertError) as e:
        ctx().ibert_gelu_i(q.view(-1)[1:], 1e-3, 0.03)  # misaligned
    assert e.value.code == -4
    with pytest.raises(IbertError) as e:
        ctx().ibert_layernorm_i(torch.zeros((1, 2048), dtype=torch.int32, device="cuda"), 1e-3, None, 0.0,
                                np.ones(2048), np.zeros(2048), 0.02)
    assert e.value.code == -2
    assert ctx().ibert_last_status() == 0


# From 24, 25 or 32 rows per SM on a warp of the streaming kernel takes two rows together: row counts on both sides of
# the switches (148 SMs: 3552, 3700, 4736) and of full grids of pairs (4736, 7104), odd ones with a last pair of one row.  Shared memory is filled before each call by an int16 call whose every 32-bit word, Q16 values and residuals
# alike, is 2^26 + 2^20 - 1: read as an int32 row it has wrapped sums (sum 2^30 - 2^10, squares below sum^2 / C), whose
# "variance" is as large as 64 bits go -- statistics that a row beside it must not see.
@pytest.mark.parametrize("C", [256, 512, 768, 1008, 1024])
@pytest.mark.parametrize("dtype", [np.int32, np.int16])
def test_layernorm_of_row_pairs(C, dtype):
    c, rng = ctx(), np.random.default_rng(C)
    gamma, beta, S, S_r, S_out = rng.normal(1.0, 0.1, C), rng.normal(0.0, 0.1, C), 1e-3, 2e-5, 4.5 / 127.0
    word = np.array([2 ** 26 + 2 ** 20 - 1], np.int32)
    fill_q, fill_r = dev(np.tile(word.view(np.int16), (7104, 512))), dev(np.tile(word.view(np.int8), (7104, 256)))
    q = rng.integers(-20000, 20001, (7105, C)).astype(np.int32)
    r = rng.integers(-127, 128, (7105, C)).astype(np.int8)
    want = oracle.layernorm(q, S, r, S_r, gamma, beta, S_out)[0]
    qd, rd = dev(q.astype(dtype)), dev(r)
    for rows in (3551, 3552, 3553, 3555, 3699, 3700, 4001, 4721, 4735, 4736, 4737, 7103, 7104, 7105):
        c.ibert_layernorm_i(fill_q, S, fill_r, S_r, np.ones(1024), np.zeros(1024), S_out)
        c.check()                                             # (the filling blocks have left their SMs)
        out, _ = c.ibert_layernorm_i(qd[:rows], S, rd[:rows], S_r, gamma, beta, S_out)
        assert_same(host(out), want[:rows], f"layernorm {rows}x{C}")
    c.check()


@pytest.mark.parametrize("C", [512, 752, 1024])
def test_layernorm_of_row_pairs_at_perfect_squares(C):
    """Rows of +-a up to the largest input: the variance is a perfect square, one element more or less puts it on either
    side of a root's step; means of both signs, on and off a whole number."""
    rng = np.random.default_rng(C)
    rows = 4800
    a = np.where(np.arange(rows) % 5 == 0, 1 << 20, np.rint(2.0 ** rng.uniform(0, 19.9, rows))).astype(np.int64)[:, None]
    q = np.where(np.arange(C) % 2 == 0, a, -a)
    q[1::4, 0] -= 1
    q[2::4, 1] += 1
    shift = rng.integers(-(1 << 18), 1 << 18, (rows, 1))
    q[3::7] = (q[3::7] >> 1) + shift[3::7]
    q[5::11, 3] = 0
    q = np.clip(q, -(1 << 20), 1 << 20).astype(np.int32)
    r = np.zeros((rows, C), np.int8)
    gamma, beta = 1.0 + 0.1 * rng.standard_normal(C), 0.1 * rng.standard_normal(C)
    out, _ = ctx().ibert_layernorm_i(dev(q), 1e-4, dev(r), 0.02, gamma, beta, 0.04)
    ctx().check()
    assert_same(host(out), oracle.layernorm(q, 1e-4, r, 0.02, gamma, beta, 0.04)[0], "layernorm at perfect squares")


def test_layernorm_constants_follow_every_element_of_their_arrays():
    """The constants of a call are found again by a sample of what they derive from: arrays that differ in one element
    outside it, or in their order, are others; so they are after more scales than are kept."""
    rng = np.random.default_rng(5)
    rows, C = 6, 256
    q = rng.integers(-30000, 30001, (rows, C)).astype(np.int32)
    r = rng.integers(-127, 128, (rows, C)).astype(np.int8)
    gamma, beta = 1.0 + 0.1 * rng.standard_normal(C), 0.1 * rng.standard_normal(C)
    others = []
    for i in (1, 3, 129, 255):
        g = gamma.copy()
        g[i] = 2.0
        others.append((g, beta))
        b = beta.copy()
        b[i] = 0.7
        others.append((gamma, b))
    pairs = [(gamma, beta), *others, (beta, gamma), (gamma, beta)]
    want = [oracle.layernorm(q, 1e-4, r, 0.02, g, b, 0.04)[0] for g, b in pairs]
    for _ in range(2):
        for (g, b), w in zip(pairs, want):
            assert_same(host(ctx().ibert_layernorm_i(dev(q), 1e-4, dev(r), 0.02, g, b, 0.04)[0]), w, "layernorm constants")
    qd, rd = dev(q), dev(r)
    for i in range(1100):
        for _ in range(2):                                     # the second call keeps them
            ctx().ibert_layernorm_i(qd, 1e-4, rd, 0.02, gamma, beta, 0.04 + 1e-5 * (i + 1))
    for (g, b), w in zip(pairs, want):
        assert_same(host(ctx().ibert_layernorm_i(qd, 1e-4, rd, 0.02, g, b, 0.04)[0]), w, "layernorm constants")
    ctx().check()
