// INT8 GEMMs for small token counts: the linear layers of an encoder layer (INT8 x INT8 -> INT32, dyadic
// requantization, i-GELU) and the projections with residual + i-LayerNorm, as ONE wave of CTAs each.
//
// With one sentence or a few, a launch is bound by latency, not by a rate: what counts is the chain
// "previous kernel done -> operands here -> MMA -> epilogue -> stored".  Two things shorten it:
//   * channels on the TMEM lanes (A = 128 weight rows) and FEW tokens per tile (B = 16..128 token rows): the
//     tile count fills the SMs, and of a CTA's operands only the small token part depends on the previous
//     kernel.  The weight rows -- all of them when K <= 1024 -- are requested before the dependency wait and
//     arrive while the previous kernel still runs (layer-owned weights only: `w_static`).
//   * the LayerNorm form keeps a token tile inside one cluster (H / 128 CTAs, each 128 channels of all tokens):
//     two numbers per token and CTA cross distributed shared memory, and the separate LayerNorm launch goes.
// The epilogue loops are short (8 columns per step): at these sizes a warp runs its code once or twice, and
// fetching instructions costs as much as executing them.
#include <cuda.h>

#include <algorithm>
#include <cmath>

#include "device_utils.cuh"
#include "sm100_ptx.cuh"

namespace ibert {
namespace {

constexpr int kCh = 128;           // output channels per CTA = TMEM lanes
constexpr int kSpan = 128;         // K bytes of one swizzle span
constexpr int kBK = 2 * kSpan;     // K bytes per operand stage: one wait and one commit per eight MMAs
constexpr int kUmmaK = 32;
constexpr int kWSpan = kCh * kSpan, kWBytes = kCh * kBK;
constexpr int kMaxStages = 8;
constexpr int kIssuers = 2;        // MMA-issuing warps
constexpr int kMaxTok = 128;       // tokens per tile (plain form)
constexpr int kMaxTokLateW = 96;   // the same when the weights are no layer's own
constexpr int kMaxTokLn = 64;      // tokens per tile (LayerNorm form)
constexpr int kMaxCluster = 8;     // CTAs per token tile (LayerNorm form): H <= 1024
constexpr int kMaxSmallThreads = 512;
// behind the operand ring: full[8], empty[8], acc, TMEM base; LayerNorm: partial sums [kMaxCluster][tokens]
constexpr int kBarBytes = 256;
constexpr int kPartBar = kBarBytes - 8;   // LayerNorm: barrier of the partial sums
constexpr int kSmemLimit = 227 * 1024;

struct SmallArgs {
  int T, N, K;
  int nt;            // tokens per tile: a multiple of 16
  int stages;        // operand stages in shared memory
  int w_static;      // the weights and constants are no product of earlier work on the stream
  uint32_t tmem_cols;
  const int32_t* b;
  const int32_t* c;
  const int32_t* bias;
  GeluConsts gelu;
  void* out;
  int32_t* status;
  // LayerNorm form
  const int8_t* res;
  const int32_t* b_i;
  const int64_t* B_i;
  LnConsts ln;
};

struct Tile {
  uint8_t* smem;
  uint32_t tmem_base;
  int split;           // accumulators to add up (at columns 0, nt)
  bool ok;
};

// eight accumulator columns of a warp's lanes
__device__ __forceinline__ void load_acc8(const Tile& t, uint32_t addr, int nt, uint32_t (&v)[8]) {
  ptx::tmem_ld8(addr, v);
  if (t.split == 2) {
    uint32_t u[8];
    ptx::tmem_ld8(addr + (uint32_t)nt, u);
    ptx::tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] += u[i];
  } else {
    ptx::tmem_wait_ld();
  }
}

// The part both forms share: barriers and TMEM, the operand ring, the MMAs.  On return every thread has seen
// the accumulators complete (or ok = false after a bounded wait ran out).
// `constants` loads what only depends on layer-owned data, `inputs` what the previous kernel may have written.
template <bool CLUSTER, typename Constants, typename Inputs>
__device__ __forceinline__ Tile run_main_loop(const CUtensorMap& map_w, const CUtensorMap& map_x, const SmallArgs& a,
                                              int c0, int t0, Constants&& constants, Inputs&& inputs) {
  extern __shared__ uint8_t smem_raw[];
  Tile r;
  r.smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  r.ok = true;
  const uint32_t base = ptx::smem_addr(r.smem);
  const uint32_t stage_bytes = (uint32_t)(kWBytes + a.nt * kBK);
  const uint32_t bar_full = base + a.stages * stage_bytes, bar_empty = bar_full + 8 * kMaxStages;
  const uint32_t bar_acc = bar_empty + 8 * kMaxStages;
  const uint32_t s_tmem = bar_acc + 8;
  const int warp = threadIdx.x >> 5;
  const int k_blocks = (a.K + kBK - 1) / kBK;
  const int first = min(a.stages, k_blocks);
  r.split = min(kIssuers, k_blocks);

  // the weight / token half of K block `kb` (two swizzle spans each; past K: zero fill)
  auto load_w = [&](int stage, int kb) {
    const uint32_t dst = base + stage * stage_bytes, bar = bar_full + 8 * stage;
    ptx::tma_load_2d(dst, &map_w, bar, kb * kBK, c0);
    ptx::tma_load_2d(dst + kWSpan, &map_w, bar, kb * kBK + kSpan, c0);
  };
  auto load_x = [&](int stage, int kb) {
    const uint32_t dst = base + stage * stage_bytes + kWBytes, bar = bar_full + 8 * stage;
    ptx::tma_load_2d(dst, &map_x, bar, kb * kBK, t0);
    ptx::tma_load_2d(dst + a.nt * kSpan, &map_x, bar, kb * kBK + kSpan, t0);
  };

  if (warp == 0) {
    if (ptx::elect_one()) {
      for (int s = 0; s < a.stages; ++s) {
        ptx::mbar_init(bar_full + 8 * s, 1);
        ptx::mbar_init(bar_empty + 8 * s, 1);
      }
      ptx::mbar_init(bar_acc, (uint32_t)r.split);
      if constexpr (CLUSTER) ptx::mbar_init(bar_full + kPartBar, 1);
      ptx::fence_mbar_init();
      // (the records of every CTA of the cluster, 16 bytes per token)
      if constexpr (CLUSTER) ptx::mbar_arrive_expect_tx(bar_full + kPartBar, (uint32_t)(a.N / kCh * a.nt * 16));
      for (int s = 0; s < first; ++s) {
        ptx::mbar_arrive_expect_tx(bar_full + 8 * s, stage_bytes);
        if (a.w_static) load_w(s, s);
      }
      ptx::tma_prefetch_desc(&map_x);
    }
  } else if (warp == 1) {
    ptx::tmem_alloc(s_tmem, a.tmem_cols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  if constexpr (CLUSTER) ptx::cluster_sync();        // (every CTA runs: its shared memory may be written from now on)
  else __syncthreads();
  ptx::tc_fence_after_sync();
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r.tmem_base) : "r"(s_tmem));
  ptx::grid_dep_launch();
  if (a.w_static) constants();
  ptx::grid_dep_wait();

  if (warp == 0) {
    if (ptx::elect_one()) {
      for (int s = 0; s < first; ++s) {
        if (!a.w_static) load_w(s, s);
        load_x(s, s);
      }
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = first; kb < k_blocks; ++kb) {
        if (!ptx::mbar_wait_parked(bar_empty + 8 * stage, phase)) { r.ok = false; break; }
        ptx::mbar_arrive_expect_tx(bar_full + 8 * stage, stage_bytes);
        load_w(stage, kb);
        load_x(stage, kb);
        if (++stage == a.stages) { stage = 0; phase ^= 1; }
      }
    }
    __syncwarp();
  } else if (warp <= kIssuers) {
    // issuer i takes every kIssuers-th K block into its own accumulator (columns i nt ..): with few tokens an MMA
    // is short and the issuing lane, not the tensor pipe, sets the pace (K = 3072, 16 tokens: 2.95 -> 2.35 us)
    const int issuer = warp - 1;
    if (issuer < k_blocks && ptx::elect_one()) {
      const uint32_t idesc = ptx::make_idesc_i8(kCh, a.nt, true, true);
      const uint32_t x_span = (uint32_t)(a.nt * kSpan) >> 4;      // (descriptor addresses count 16 bytes)
      const uint32_t d_tmem = r.tmem_base + (uint32_t)(issuer * a.nt);
      int stage = issuer;
      uint32_t phase = 0;
#pragma unroll 1
      for (int kb = issuer; kb < k_blocks; kb += kIssuers) {
        if (stage >= a.stages) { stage -= a.stages; phase ^= 1; }
        if (!ptx::mbar_wait_parked(bar_full + 8 * stage, phase)) { r.ok = false; break; }
        ptx::tc_fence_after_sync();
        const uint32_t sw = base + stage * stage_bytes;
        const uint64_t dw = ptx::make_kmajor_desc(sw, 1024, ptx::kSwizzle128);
        const uint64_t dx = ptx::make_kmajor_desc(sw + kWBytes, 1024, ptx::kSwizzle128);
#pragma unroll
        for (int k = 0; k < kBK / kUmmaK; ++k) {                  // +32 bytes inside a span, then the next span
          const uint32_t in = 2 * (k & 3);
          ptx::mma_i8_ss(d_tmem, dw + in + (k >> 2) * (kWSpan >> 4), dx + in + (k >> 2) * x_span, idesc, (kb >= kIssuers || k != 0) ? 1u : 0u);
        }
        if (kb + a.stages < k_blocks) ptx::mma_commit(bar_empty + 8 * stage);   // only stages that are filled again
        stage += kIssuers;
      }
      ptx::mma_commit(bar_acc);
    }
    __syncwarp();
  }
  if (!a.w_static) constants();
  inputs();
  if (!ptx::mbar_wait(bar_acc, 0)) r.ok = false;
  r.ok = __all_sync(0xffffffffu, r.ok);
  ptx::tc_fence_after_sync();
  return r;
}

// per-channel constants of the thread's channel
struct ChannelConsts {
  int32_t b = 0, c = 0, bias = 0;
  int64_t add = 0;
};
template <int KIND>
__device__ __forceinline__ ChannelConsts load_channel(const SmallArgs& a, int n) {
  ChannelConsts k;
  if (n < a.N) {
    k.bias = a.bias ? __ldg(a.bias + n) : 0;
    if constexpr (KIND != EPI_RAW) {
      k.b = __ldg(a.b + n);
      k.c = __ldg(a.c + n);
      k.add = (int64_t)k.bias * k.b + rounding_half(k.c);
    }
  }
  return k;
}

// i-GELU behind multipliers of 1/2 and more (the wide upper-word form), a kind of its own inside this file
constexpr int kEpiGeluWideForm = 16;

// ------------------------------------------------------------------------------------------ plain form
// Tile = 128 channels x nt tokens; 128 * parts threads, thread = channel x every parts-th chunk of 8 tokens.
template <int KIND, bool FAST>
__global__ void __launch_bounds__(kMaxSmallThreads, 1)
gemm_small_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x,
                  const SmallArgs a) {
  constexpr int kElem = (KIND == EPI_RAW || KIND == EPI_Q16) ? 4 : (KIND == EPI_Q16H ? 2 : 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quad = warp & 3, part = warp >> 2, parts = (int)blockDim.x >> 7;
  const int c_tiles = (a.N + kCh - 1) / kCh;
  const int c0 = ((int)blockIdx.x % c_tiles) * kCh, t0 = ((int)blockIdx.x / c_tiles) * a.nt;
  const int row = quad * 32 + lane;
  ChannelConsts k;
  const Tile tile = run_main_loop<false>(map_w, map_x, a, c0, t0, [&] { k = load_channel<KIND>(a, c0 + row); }, [] {});

  // results -> shared memory (the operand ring is free), token-major: a warp's 32 lanes write 32 neighbours
  const int live = min(a.nt, a.T - t0);
  if (tile.ok) {
    const GeluConsts gk = a.gelu;
    const int64_t gelu_half = rounding_half(gk.c);
    const int32_t gelu_rnd = (1 << gk.s_f) - 1;
    const uint32_t t_lane = tile.tmem_base + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
    for (int col = part * 8; col < live; col += parts * 8) {
      uint32_t v[8];
      load_acc8(tile, t_lane + col, a.nt, v);
      const uint32_t dst = ptx::smem_addr(tile.smem) + (uint32_t)((col * kCh + row) * kElem);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        int32_t o;
        if constexpr (KIND == kEpiGeluWideForm)
          o = clamp_sym(igelu_magnitude_upper(requant_upper_wide((int32_t)v[i] + k.bias, k.b, k.c), gk, gelu_rnd), 127);
        else
          o = epilogue_value<KIND, FAST>((int32_t)v[i], k.bias, k.b, k.c, k.add, gk, gelu_half, gelu_rnd);
        if constexpr (kElem == 4) asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + i * kCh * 4), "r"(o) : "memory");
        else if constexpr (kElem == 2) asm volatile("st.shared.u16 [%0], %1;" ::"r"(dst + i * kCh * 2), "h"((uint16_t)o) : "memory");
        else asm volatile("st.shared.u8 [%0], %1;" ::"r"(dst + i * kCh), "r"(o) : "memory");
      }
    }
  }
  if (!tile.ok) atomicCAS(a.status, 0, IBERT_ERR_TIMEOUT);
  ptx::tc_fence_before_sync();
  const bool ok = __syncthreads_and(tile.ok);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tile.tmem_base, a.tmem_cols);
  }
  if (!ok) return;
  // shared memory -> global: 16 bytes per thread, whole 128-byte rows per eight lanes
  constexpr int kChunks = 8 * kElem;                        // 16-byte chunks of a tile row
  const int n_bytes = min(kCh, a.N - c0) * kElem;
  uint8_t* out = static_cast<uint8_t*>(a.out) + ((int64_t)t0 * a.N + c0) * kElem;
  const int64_t pitch = (int64_t)a.N * kElem;
  for (int i = threadIdx.x; i < live * kChunks; i += blockDim.x) {
    const int t = i / kChunks, ch = (i % kChunks) * 16;
    if (ch < n_bytes)
      *reinterpret_cast<uint4*>(out + t * pitch + ch) = *reinterpret_cast<const uint4*>(tile.smem + t * (kCh * kElem) + ch);
  }
}

// ------------------------------------------------------------------------------------------ LayerNorm form
// A cluster of H / 128 CTAs owns nt tokens.  After the MMAs the Q16 values go to shared memory token-major, so
// that from there on a warp owns TPW tokens and a lane four adjacent channels of each: residual in and result
// out as whole words, row sums by warp reductions, per-channel LayerNorm constants in registers.
template <int TPW, bool FAST>
__global__ void __launch_bounds__(kMaxSmallThreads, 1)
gemm_ln_small_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x,
                     const SmallArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quad = warp & 3, part = warp >> 2, parts = (int)blockDim.x >> 7;
  const int cl = a.N / kCh;
  const int rank = (int)ptx::cluster_ctarank();
  const int c0 = rank * kCh, t0 = ((int)blockIdx.x / cl) * a.nt;
  const int row = quad * 32 + lane;
  const int ch = c0 + lane * 4;                              // this lane's channels from pass 2 on
  const LnConsts ln = a.ln;
  ChannelConsts k;
  int4 bv;
  longlong2 B01, B23;
  uint32_t rw[TPW];
  const Tile tile = run_main_loop<true>(map_w, map_x, a, c0, t0, [&] {
    k = load_channel<EPI_Q16>(a, c0 + row);
    bv = __ldg(reinterpret_cast<const int4*>(a.b_i + ch));
    B01 = __ldg(reinterpret_cast<const longlong2*>(a.B_i + ch));
    B23 = __ldg(reinterpret_cast<const longlong2*>(a.B_i + ch + 2));
  }, [&] {
#pragma unroll
    for (int j = 0; j < TPW; ++j)                            // (tokens past the end: any row, never stored)
      rw[j] = *reinterpret_cast<const uint32_t*>(a.res + (int64_t)min(t0 + warp * TPW + j, a.T - 1) * a.N + ch);
  });
  bool ok = tile.ok;
  const uint32_t s_part = ptx::smem_addr(tile.smem) + a.stages * (kWBytes + a.nt * kBK) + kBarBytes;
  const uint32_t bar_part = s_part - kBarBytes + kPartBar;

  // pass 1: requantized values, token-major in shared memory (int32; the operand ring is free)
  int32_t* s_v = reinterpret_cast<int32_t*>(tile.smem);
  if (ok) {
    const uint32_t t_lane = tile.tmem_base + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
    for (int col = part * 8; col < a.nt; col += parts * 8) {
      uint32_t v[8];
      load_acc8(tile, t_lane + col, a.nt, v);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        s_v[(col + i) * kCh + row] = FAST ? clamp_sym(requant_upper((int32_t)v[i] + k.bias, k.b), 32767)
                                          : requant_add((int32_t)v[i], k.b, k.add, k.c, 32767);
      }
    }
  }
  if (!ok) atomicCAS(a.status, 0, IBERT_ERR_TIMEOUT);
  ptx::tc_fence_before_sync();
  ok = __syncthreads_and(ok);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tile.tmem_base, a.tmem_cols);
  }

  // pass 2: residual added; this CTA's share of the row sums goes to every CTA of the cluster, each 16-byte
  // record credited to the receiver's barrier (one way through the cluster network, no barrier round trip)
  int32_t v[TPW][4];
#pragma unroll
  for (int j = 0; j < TPW; ++j) {
    const int t = warp * TPW + j;
    const int4 q = *reinterpret_cast<const int4*>(s_v + t * kCh + lane * 4);
    v[j][0] = q.x; v[j][1] = q.y; v[j][2] = q.z; v[j][3] = q.w;
    int32_t s1 = 0;
    uint64_t s2 = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[j][i] += (sext_byte(rw[j], i) * ln.res_nb + ln.res_nhalf) >> ln.res_nc;
      s1 += v[j][i];
      s2 += (uint64_t)((int64_t)v[j][i] * (int64_t)v[j][i]);
    }
    // |v| < 2^18: a lane's squares stay below 2^38 and reduce as two halves of 25 and 13 bits
    s1 = __reduce_add_sync(0xffffffffu, s1);
    const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)s2 & 0x1ffffffu);
    const uint32_t hi = __reduce_add_sync(0xffffffffu, (uint32_t)(s2 >> 25));
    if (lane < cl)
      ptx::st_async_v4(ptx::map_to_cta(s_part + (uint32_t)((rank * a.nt + t) * 16), (uint32_t)lane), (uint32_t)s1, lo, hi, 0u,
                       ptx::map_to_cta(bar_part, (uint32_t)lane));
  }
  if (!ptx::mbar_wait_cluster(bar_part, 0)) ok = false;
  ok = __all_sync(0xffffffffu, ok);
  // After an expired wait nothing is stored, and nobody leaves while a peer may still send records here: the barrier of
  // the cluster waits for the threads that have not exited, and a peer that has all its records has sent its own.
  auto give_up = [&] {
    atomicCAS(a.status, 0, IBERT_ERR_TIMEOUT);
    ptx::cluster_sync();
#pragma unroll 1
    for (int i = 0; i < 10000 && !ptx::mbar_test_cluster(bar_part, 0); ++i);   // records still on their way
  };
  if (TPW == 1 && !ok) {
    give_up();
    return;
  }

  // pass 3: mean and I-Sqrt of the variance (sum (v - mu)^2 = sum v^2 - 2 mu sum v + C mu^2 in integers).  One token
  // per warp: every lane the same, no exchange.  More
  // tokens: a thread per token, because the warp form repeats some 200 instructions for every token and CTA
  // (95 instructions per element at 48 tokens); encoder layer Large B = 7, L = 128 43.0 -> 40.4 us, Base B = 8,
  // L = 77 30.1 -> 29.7.
  const int C = a.N;
  auto mean_of = [&](int32_t sum) { return ln_mean(sum, C, ln); };
  LnNorm one{};
  if constexpr (TPW == 1) {
    uint32_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
    if (lane < cl)
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(p0), "=r"(p1), "=r"(p2), "=r"(p3)
                   : "r"(s_part + (uint32_t)((lane * a.nt + warp) * 16)));
    const int32_t sum = __reduce_add_sync(0xffffffffu, (int32_t)p0);
    // (at most eight records with low words below 2^30: their 16-bit halves reduce as 32-bit sums)
    const uint64_t sumsq = (uint64_t)__reduce_add_sync(0xffffffffu, p1 & 0xffffu) +
                           ((uint64_t)__reduce_add_sync(0xffffffffu, p1 >> 16) << 16) +
                           ((uint64_t)__reduce_add_sync(0xffffffffu, p2) << 25);
    const int32_t mu = mean_of(sum);
    one = ln_norm(mu, ln_root(sumsq + (uint64_t)((int64_t)mu * (int64_t)(C * mu - 2 * sum)), (uint32_t)C, ln.root_k));
  } else {
    if ((int)threadIdx.x < a.nt) {
      int32_t sum = 0;
      uint64_t sumsq = 0;
#pragma unroll 2
      for (int r = 0; r < cl; ++r) {
        uint32_t p0, p1, p2, p3;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(p0), "=r"(p1), "=r"(p2), "=r"(p3)
                     : "r"(s_part + (uint32_t)((r * a.nt + (int)threadIdx.x) * 16)));
        sum += (int32_t)p0;
        sumsq += (uint64_t)p1 + ((uint64_t)p2 << 25);
      }
      const int32_t mu = mean_of(sum);
      const LnNorm pr = ln_norm(mu, ln_root(sumsq + (uint64_t)((int64_t)mu * (int64_t)(C * mu - 2 * sum)), (uint32_t)C, ln.root_k));
      // (the token's own records are consumed: the first one's place takes the result)
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(s_part + threadIdx.x * 16), "r"(pr.scale), "r"(pr.shift), "r"(pr.rho), "r"(0) : "memory");
    }
    if (!__syncthreads_and(ok)) {                            // (several tokens per warp: the warps of a CTA meet here)
      give_up();
      return;
    }
  }
  // pass 4: normalize, affine + requantize, store
  const int32_t bb[4] = {bv.x, bv.y, bv.z, bv.w};
  const int64_t BB[4] = {B01.x, B01.y, B23.x, B23.y};
#pragma unroll
  for (int j = 0; j < TPW; ++j) {
    const int t = warp * TPW + j;
    LnNorm pr = one;
    int32_t unused;
    if constexpr (TPW > 1)
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(pr.scale), "=r"(pr.shift), "=r"(pr.rho), "=r"(unused) : "r"(s_part + (uint32_t)(t * 16)));
    int32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[i] = max(requant_upper_add(ln_normalize(v[j][i], pr) << ln.out_sh, bb[i], BB[i]), -127);
    }
    if (t0 + t < a.T)
      *reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(a.out) + (int64_t)(t0 + t) * a.N + ch) = pack4_sat_s8(o[0], o[1], o[2], o[3]);
  }
}

int operand_maps(CUtensorMap* mw, CUtensorMap* mx, const int8_t* w, const int8_t* x, int64_t M, int N, int K, int nt) {
  const uint64_t wdims[2] = {(uint64_t)K, (uint64_t)N}, xdims[2] = {(uint64_t)K, (uint64_t)M}, str[1] = {(uint64_t)K};
  const uint32_t wbox[2] = {kSpan, kCh}, xbox[2] = {kSpan, (uint32_t)nt};
  if (int rc = encode_tensor_map(mw, w, 2, wdims, str, wbox, 128)) return rc;
  return encode_tensor_map(mx, x, 2, xdims, str, xbox, 128);
}

uint32_t tmem_columns(int n) {
  uint32_t c = 32;
  while ((int)c < n) c <<= 1;
  return c;
}

// Tokens per tile that give one wave of CTAs, or 0 when the problem is larger than that.  Weights that may not be read
// ahead of the dependency wait leave the two-stage ring of 112 and 128 tokens without its head start, and the large
// tiles are faster there (single linear layers, us, this kernel / large tiles: 765 x 2304 x 768, 96 tokens, 4.5 / 4.6;
// 1021 x 2304 x 768, 128 tokens, 5.0 / 4.3; 1725 x 1024 x 4096, 96 tokens, 8.6 / 10.3; 2301 x 1024 x 4096, 128 tokens,
// 12.0 / 8.7).  Inside a layer it is the other way round: Base 4 x 256 34.7 / 42.0 us, 7 x 128 31.2 / 32.9.
int small_tile_tokens(const ibert_ctx* ctx, int64_t M, int N, bool w_static) {
  const int c_tiles = (N + kCh - 1) / kCh, t_max = ctx->num_sms / c_tiles;
  if (t_max < 1 || M > (int64_t)t_max * (w_static ? kMaxTok : kMaxTokLateW)) return 0;
  const int per = (int)((M + t_max - 1) / t_max);
  return std::max((per + 15) & ~15, 16);
}

template <int KIND, bool FAST>
int launch_small_kind(ibert_ctx* ctx, int grid, int threads, int smem, const CUtensorMap& mw, const CUtensorMap& mx,
                      const SmallArgs& a) {
  static bool attr_dev[kMaxDevices] = {false};
  bool& attr = attr_dev[ctx->device % kMaxDevices];
  if (!attr) {
    if (cudaFuncSetAttribute(gemm_small_kernel<KIND, FAST>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess)
      return IBERT_ERR_CUDA;
    attr = true;
  }
  return launch_pdl(gemm_small_kernel<KIND, FAST>, dim3(grid), dim3(threads), (size_t)smem, ctx->stream, 1, mw, mx, a);
}

// Clusters of `cl` CTAs that are resident at once, one CTA per SM.  A cluster lies inside one GPC, so this is
// less than num_sms / cl (148 SMs: 15 clusters of eight, not 18); asked of the driver once per device.
int small_clusters(const ibert_ctx* ctx, int cl) {
  static int known[kMaxDevices][kMaxCluster + 1] = {};
  int& n = known[ctx->device % kMaxDevices][cl];
  if (n == 0) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(kMaxSmallThreads);
    cfg.dynamicSmemBytes = kSmemLimit;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int got = 0;
    if (cudaFuncSetAttribute(gemm_ln_small_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&got, gemm_ln_small_kernel<1, true>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      got = ctx->num_sms / 10 / cl * 8;
    }
    n = std::max(got, 1);
  }
  return n;
}

int small_ln_tile_tokens(const ibert_ctx* ctx, int64_t M, int cl) {
  const int t_max = small_clusters(ctx, cl);
  if (M > (int64_t)t_max * kMaxTokLn) return 0;
  const int per = (int)((M + t_max - 1) / t_max);
  return std::max((per + 15) & ~15, 16);
}

template <int TPW, bool FAST>
int launch_ln_small_tpw(ibert_ctx* ctx, int grid, int smem, int cl, const CUtensorMap& mw, const CUtensorMap& mx,
                        const SmallArgs& a) {
  static bool attr_dev[kMaxDevices] = {false};
  bool& attr = attr_dev[ctx->device % kMaxDevices];
  if (!attr) {
    if (cudaFuncSetAttribute(gemm_ln_small_kernel<TPW, FAST>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess)
      return IBERT_ERR_CUDA;
    attr = true;
  }
  return launch_pdl(gemm_ln_small_kernel<TPW, FAST>, dim3(grid), dim3(kMaxSmallThreads), (size_t)smem, ctx->stream, cl, mw, mx, a);
}

SmallArgs small_args(ibert_ctx* ctx, int64_t M, int N, int K, int nt, int extra_smem, const GemmEpilogue& epi, void* out) {
  SmallArgs a{};
  a.T = (int)M; a.N = N; a.K = K; a.nt = nt;
  const int stage = kWBytes + nt * kBK, k_blocks = (K + kBK - 1) / kBK;
  a.stages = std::min({k_blocks, kMaxStages, (kSmemLimit - kBarBytes - 1024 - extra_smem) / stage});
  // a stage that is filled again must stay with one issuer: the other could reach it before its first filling and
  // take the barrier's initial phase for the second one
  if (a.stages < k_blocks) a.stages -= a.stages % kIssuers;
  a.w_static = epi.w_static ? 1 : 0;
  a.tmem_cols = tmem_columns(kIssuers * nt);
  a.b = epi.d_b; a.c = epi.d_c; a.bias = epi.d_bias; a.gelu = epi.gelu; a.out = out; a.status = ctx->d_status;
  return a;
}

}  // namespace

bool gemm_small_takes(const ibert_ctx* ctx, int64_t M, int N, int K, bool w_static) {
  return M > 0 && K >= 256 && K % 16 == 0 && small_tile_tokens(ctx, M, N, w_static) > 0;
}

int launch_gemm_small_i8(ibert_ctx* ctx, const int8_t* x, const int8_t* w, int64_t M, int N, int K,
                         const GemmEpilogue& epi, void* out) {
  if (!gemm_small_takes(ctx, M, N, K, epi.w_static)) return IBERT_ERR_ARG;
  const SmallArgs a = small_args(ctx, M, N, K, small_tile_tokens(ctx, M, N, epi.w_static), 0, epi, out);
  CUtensorMap mw, mx;
  if (int rc = operand_maps(&mw, &mx, w, x, M, N, K, a.nt)) return rc;
  const int grid = ((N + kCh - 1) / kCh) * (int)((M + a.nt - 1) / a.nt);
  const int threads = 128 * std::min(a.nt / 8, 4);
  const int smem = a.stages * (kWBytes + a.nt * kBK) + kBarBytes + 1024;
  const bool fast = epi.fast != 0 && ((epi.kind != EPI_GELU && epi.kind != EPI_HGELU) || epi.gelu.fast != 0);
  if (epi.fast == 2) {
    if (epi.kind != EPI_GELU || !fast) return IBERT_ERR_ARG;      // tables in a form nothing else reads
    return launch_small_kind<kEpiGeluWideForm, true>(ctx, grid, threads, smem, mw, mx, a);
  }
#define IBERT_SMALL(KIND)                                                              \
  return fast ? launch_small_kind<KIND, true>(ctx, grid, threads, smem, mw, mx, a)     \
              : launch_small_kind<KIND, false>(ctx, grid, threads, smem, mw, mx, a)
  switch (epi.kind) {
    case EPI_INT8: IBERT_SMALL(EPI_INT8);
    case EPI_Q16: IBERT_SMALL(EPI_Q16);
    case EPI_Q16H: IBERT_SMALL(EPI_Q16H);
    case EPI_GELU: IBERT_SMALL(EPI_GELU);
    case EPI_HGELU: IBERT_SMALL(EPI_HGELU);
    default: return launch_small_kind<EPI_RAW, false>(ctx, grid, threads, smem, mw, mx, a);
  }
#undef IBERT_SMALL
}

bool gemm_ln_small_supported(const ibert_ctx* ctx, int64_t M, int H, int K, const GemmEpilogue& epi, const LnConsts& ln) {
  if (M <= 0 || H % kCh != 0 || H / kCh > kMaxCluster || K < 256 || K % 16 != 0) return false;
  if (epi.kind != EPI_Q16 || !ln.has_res || !ln.res_fast || !ln.res_narrow || !ln.out_fast || ln.C != H) return false;
  if (127.0 * std::ldexp((double)ln.b_r, ln.res_sh - 32) >= 200000.0) return false;      // |v| < 2^18, as the sums assume
  return small_ln_tile_tokens(ctx, M, H / kCh) > 0;
}

int launch_gemm_ln_small_i8(ibert_ctx* ctx, const int8_t* x, const int8_t* w, int64_t M, int H, int K,
                            const GemmEpilogue& epi, const int8_t* res, const LnConsts& ln, const int32_t* d_b_i,
                            const int64_t* d_B_i, int8_t* out) {
  if (!gemm_ln_small_supported(ctx, M, H, K, epi, ln)) return IBERT_ERR_ARG;
  const int cl = H / kCh, nt = small_ln_tile_tokens(ctx, M, cl), part_bytes = kMaxCluster * nt * 16;
  SmallArgs a = small_args(ctx, M, H, K, nt, part_bytes, epi, out);
  a.res = res; a.b_i = d_b_i; a.B_i = d_B_i; a.ln = ln;
  CUtensorMap mw, mx;
  if (int rc = operand_maps(&mw, &mx, w, x, M, H, K, nt)) return rc;
  const int grid = cl * (int)((M + nt - 1) / nt);
  const int smem = a.stages * (kWBytes + nt * kBK) + kBarBytes + part_bytes + 1024;
  // 16 warps of 1, 2, 3 or 4 tokens
#define IBERT_LNS(TPW)                                                                \
  return epi.fast ? launch_ln_small_tpw<TPW, true>(ctx, grid, smem, cl, mw, mx, a)    \
                  : launch_ln_small_tpw<TPW, false>(ctx, grid, smem, cl, mw, mx, a)
  if (nt == 16) IBERT_LNS(1);
  if (nt == 32) IBERT_LNS(2);
  if (nt == 48) IBERT_LNS(3);
  IBERT_LNS(4);
#undef IBERT_LNS
}

}  // namespace ibert
