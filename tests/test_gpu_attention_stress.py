"""The persistent attention kernel over many (batch, head) pairs, launched again and again: its operand barriers
turn over thousands of times per launch, so a warp that can miss a phase shows as an expired wait."""
import pytest
import torch

import oracle
from gpu_util import assert_same, ctx, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,heads", [(20000, 128, 12), (3000, 256, 4)])
def test_many_pairs_many_launches(B, L, heads):
    H = heads * 64
    gen = torch.Generator(device="cuda").manual_seed(3)
    qkv = torch.randint(-60, 61, (B * L, 3 * H), generator=gen, device="cuda", dtype=torch.int8)
    c = ctx()
    outs = []
    for _ in range(12):
        out, _ = c.ibert_attention_i8(qkv, B, L, H, heads, 0.02, 0.02, 0.02, 0.006)
        c.check()
        outs.append(out)
        if len(outs) > 1:
            assert torch.equal(outs[0], outs.pop())
    for b in (0, B // 2, B - 1):
        want = oracle.attention(host(qkv[b * L:(b + 1) * L]), 1, L, H, heads, 0.02, 0.02, 0.02, 0.006, 255)
        assert_same(host(outs[0][b * L:(b + 1) * L]), want, f"sequence {b}")
