"""How the kernels leave, read from their source: the ways out after a wait has run out are not provoked on a GPU."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2101_01321_b200" / "csrc"


def _kernels():
    """(name, body without comments) of every __global__ function."""
    for path in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        for m in re.finditer(r"__global__\s+void\b[^{;]*?(\w+_kernel)\s*\([^{;]*\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield m.group(1), text[m.end():i - 1]


KERNELS = dict(_kernels())


def test_kernels_are_found():
    assert {"gemm_ln_small_kernel", "gemm_small_kernel", "attention_small_kernel", "gemm_ln_kernel", "gemm_splitk_kernel",
            "gemm_i8_kernel", "layernorm_pipe_kernel"} <= set(KERNELS)


def _lambdas(body):
    """{name: text} of the lambdas of a kernel, and the body without them."""
    found, rest = {}, body
    while m := re.search(r"auto\s+(\w+)\s*=\s*\[[&=]?\]\s*(?:\([^)]*\))?\s*\{", rest):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(rest[i], 0)
            i += 1
        found[m.group(1)], rest = rest[m.end():i - 1], rest[:m.start()] + rest[i:]
    return found, rest


@pytest.mark.parametrize("name", sorted(n for n, b in KERNELS.items() if "map_to_cta" in b))
def test_no_cta_leaves_while_a_peer_may_write_to_it(name):
    """A kernel that reaches into a peer's shared memory leaves early only behind a barrier of its cluster, and at its
    end behind one or behind the wait that counts what every peer sends."""
    body = KERNELS[name]
    lambdas, main = _lambdas(body)
    barriers = ["cluster_sync"] + [n for n, text in lambdas.items() if "cluster_sync()" in text]
    for m in re.finditer(r"\breturn\s*;", main):
        before = main[:m.start()].rstrip()
        assert re.search(rf"\b({'|'.join(barriers)})\(\)\s*;$", before), f"{name}: a return without a cluster barrier"
    last = max(m.end() for m in re.finditer(r"map_to_cta|ld_cluster|st_async|mbar_arrive_remote|bulk_copy_to_cta", body))
    assert re.search(r"cluster_sync\(\)|mbar_wait_cluster\(", body[last:]), f"{name}: nothing holds a CTA at its end"


def _end_of_block(text, i):
    """Position behind the block whose opening brace lies before `i`."""
    depth = 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return i


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_no_warp_vote_that_an_elected_lane_may_miss(name):
    """What one elected lane found out (`ok` of a wait that ran out) is voted on by its whole warp before any branch on
    it holds a vote or barrier: a lane that skips the branch would leave the others waiting there for good."""
    body = KERNELS[name]
    for m in re.finditer(r"if \([^;{}]*elect_one\(\)\)\s*\{", body):
        end = _end_of_block(body, m.end())
        if not re.search(r"\bok\s*=", body[m.end():end]):
            continue
        vote = re.search(r"__all_sync\(|__syncthreads_and\(|__any_sync\(", body[end:])
        if not vote:
            continue
        for cond in re.finditer(r"if \(([^;{}]*)\)\s*(\{)?", body[end:end + vote.start()]):
            if not re.search(r"\bok\b", cond.group(1)):
                continue
            at = end + cond.end()
            stop = _end_of_block(body, at) if cond.group(2) else body.index(";", at)
            assert stop < end + vote.start(), f"{name}: a vote inside `if ({cond.group(1)})`"


def test_a_callers_bias_is_read_behind_the_dependency_wait():
    """The fused GEMM + LayerNorm kernel starts before its predecessor has finished: constants of the context may be read at
    once, a bias that comes with the call only where the predecessor's results are visible (layers: w_static)."""
    lambdas, rest = _lambdas(KERNELS["gemm_ln_kernel"])
    assert "args.bias" in lambdas["load_bias"] and "args.bias" not in rest
    assert not any("args.bias" in text for name, text in lambdas.items() if name != "load_bias")
    calls = [m.start() for m in re.finditer(r"load_bias\(", rest)]
    assert len(calls) == 2
    early, late = calls
    assert rest[:early].rstrip().endswith("if (args.w_static)")
    epilogue = rest[:late]
    assert epilogue.count("ptx::grid_dep_wait();") == 3          # every thread (constants in front), producer, epilogue
    assert re.search(r"if constexpr \(!kLateConstants\) ptx::grid_dep_wait\(\);", epilogue)
    assert re.search(r"if constexpr \(kLateConstants\) \{\s*load_constants\([^)]*\);\s*ptx::grid_dep_wait\(\);\s*\}\s*if \(kLateConstants "
                     r"\|\| !args\.w_static\) \{\s*$", epilogue)
