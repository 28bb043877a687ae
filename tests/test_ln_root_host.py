"""The square root of the LayerNorm statistics (`ln_root`) on the CPU: its text is taken from the kernels' header and
compiled for the host with the undefined-behaviour checks on.  Against its definition at both ends of every root's
interval, and on sums that belong to no row at all: the row-pair LayerNorm evaluates it for the missing row of an odd row
count too, on whatever lies in shared memory, and discards the value."""
import re
import subprocess
from pathlib import Path

import pytest

HEADER = Path(__file__).resolve().parent.parent / "paper_2101_01321_b200" / "csrc" / "device_utils.cuh"

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#define __device__
#define __forceinline__ inline
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline uint32_t shr_clamped(uint32_t v, uint32_t n) { return n > 31u ? 0u : v >> n; }
"""

MAIN = r"""
static uint32_t root_k(uint32_t C) { return (uint32_t)std::fmin(4294967295.0, std::floor(4294967296.0 / std::sqrt((double)C))); }
template <int STEPS>
static void at_steps(uint32_t C, uint32_t from, uint32_t to, uint32_t step) {
  for (uint32_t s = from; s < to; s += step) {
    const uint64_t lo = (uint64_t)s * s * C, hi = (uint64_t)(s + 1) * (s + 1) * C - 1;
    if (ln_root<STEPS>(lo, C, root_k(C)) != s || ln_root<STEPS>(hi, C, root_k(C)) != s) {
      std::printf("C %u, s %u, %d steps\n", C, s, STEPS);
      std::exit(1);
    }
  }
}
int main(int argc, char** argv) {
  if (argc > 1) {                      // any 64 bits
    uint64_t x = 1, keep = 0;
    for (int i = 0; i < 2000000; ++i) {
      x = x * 6364136223846793005ull + 1442695040888963407ull;
      keep ^= ln_root<3>(x, 768, root_k(768)) ^ ln_root<3>(x >> (i & 63), 272, root_k(272));
    }
    for (int b = 0; b < 64; ++b) keep ^= ln_root<3>(uint64_t(1) << b, 1024, root_k(1024)) ^ ln_root<3>(~uint64_t(0) >> b, 1024, root_k(1024));
    std::printf("%llu\n", (unsigned long long)keep);
    return 0;
  }
  for (uint32_t C : {2u, 16u, 128u, 192u, 256u, 272u, 384u, 512u, 640u, 752u, 768u, 896u, 1008u, 1024u}) {
    at_steps<2>(C, 0, 1u << 18, 1);
    at_steps<3>(C, 0, 1u << 16, 1);
    at_steps<3>(C, 1u << 16, 1u << 22, 61);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    text = HEADER.read_text()
    root = re.search(r"template <int STEPS = 2>\n__device__.*?\n}\n", text, re.S).group(0)
    assert "ln_root" in root
    d = tmp_path_factory.mktemp("ln_root")
    (d / "root.cpp").write_text(SHIM + root + MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-o", str(d / "root"),
                    str(d / "root.cpp")], check=True, capture_output=True, text=True)
    return str(d / "root")


def test_root_at_both_ends_of_its_interval(program):
    r = subprocess.run([program], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_root_of_any_bits_is_defined(program):
    r = subprocess.run([program, "any"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
