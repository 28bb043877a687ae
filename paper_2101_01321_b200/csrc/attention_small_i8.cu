// Fused integer-only attention for few (batch, head) pairs -- S = Q K^T, i-softmax (Algorithm 3), P V,
// requantization, as in attention_i8.cu, for launches that do not fill the SMs with one CTA per pair.
//
// At one sentence there are 12 or 16 pairs for 148 SMs and the softmax of a 128-query tile is the longest part
// of the launch.  A CTA therefore takes 128 / REP queries of a pair (REP = 1, 2, 4) and the operand tile of the
// score MMA holds them REP times: rows c 128/REP .. of the tile are copy c.  Every copy's lanes of tensor memory
// then hold the same scores, and the 4 REP column groups (copy, warp quarter) each take their own CPT <= 32
// columns: 512 threads share 128 / REP rows.  A thread's scores stay in registers from the maximum to the
// probabilities (no tensor-memory write-back), row maximum and row sum meet in shared memory.  The wasted
// MMA rows cost nothing here: the MMA takes 128 rows whatever they hold.  Measured inside an encoder layer (12
// pairs of 128 x 128): MMA to probabilities 3.3 -> 0.9 us, launch 6.9 -> 3.9 us.
#include <cuda.h>

#include <algorithm>

#include "device_utils.cuh"
#include "sm100_ptx.cuh"

namespace ibert {
namespace {

constexpr int kSmallThreads = 512;

struct SmallAttnArgs {
  int B, L, H, heads;
  int n_slabs;           // 128-key tiles: ceil(L / 128)
  int rep, q_tiles;      // copies of the queries in the operand tile; tiles of 128 / rep queries per sequence
  uint32_t tmem_cols;
  AttnConsts k;
  const int32_t* lens;   // padded: [B] valid keys or nullptr; packed: [B + 1] first rows
  int8_t* out;
  int32_t* status;
};

// PACKED: the tensor maps see one "batch" of all rows, sequence b = rows lens[b] .. lens[b + 1] - 1
template <bool PACKED, int CPT>
__global__ void __launch_bounds__(kSmallThreads, 2)
attention_small_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kv,
                       const SmallAttnArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int kSlab = 128 * kHeadDim;                        // 8 KB: 128 rows of 64 bytes, 64-byte swizzle
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + kSlab;                                    // [n_slabs]
  uint8_t* sV = sK + a.n_slabs * kSlab;                        // [n_slabs]
  uint8_t* sP = sV + a.n_slabs * kSlab;                        // [n_slabs][128 rows][128 B], 128-byte swizzle
  int32_t* s_max = reinterpret_cast<int32_t*>(sP + a.n_slabs * 128 * 128);   // [128]
  uint32_t* s_sum = reinterpret_cast<uint32_t*>(s_max + 128);                // [128]
  const uint32_t bar_qk = ptx::smem_addr(s_sum + 128), bar_v = bar_qk + 8, bar_mma = bar_qk + 16, s_tmem = bar_qk + 24;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quad = warp & 3, quads = 4 / a.rep;                // lane quadrants per copy
  const int row = (quad % quads) * 32 + lane;                  // query inside the tile
  const int c0 = ((quad / quads) * 4 + (warp >> 2)) * CPT;     // this thread's first column
  const int rows = 128 / a.rep;
  const int qt = (int)blockIdx.x % a.q_tiles, pair = (int)blockIdx.x / a.q_tiles;
  const int head = pair % a.heads, batch = pair / a.heads;

  if (warp == 0) {
    if (ptx::elect_one()) {
      ptx::mbar_init(bar_qk, 1);
      ptx::mbar_init(bar_v, 1);
      ptx::mbar_init(bar_mma, 1);
      ptx::fence_mbar_init();
      ptx::tma_prefetch_desc(&map_q);
      ptx::tma_prefetch_desc(&map_kv);
    }
  } else if (warp == 1) {
    ptx::tmem_alloc(s_tmem, a.tmem_cols);
    ptx::tmem_relinquish();
  }
  if (tid < 128) {
    s_max[tid] = INT32_MIN;
    s_sum[tid] = 0;
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  uint32_t tmem_base;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(s_tmem));
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();              // the kernel that wrote qkv has completed

  // valid keys n (key-padding mask: keys >= n take no part in maximum and sum and get probability 0)
  const int row0 = PACKED ? __ldg(a.lens + batch) : 0;
  const int len = PACKED ? __ldg(a.lens + batch + 1) - row0 : (a.lens ? __ldg(a.lens + batch) : a.L);
  if (PACKED && len > a.L && tid == 0) atomicCAS(a.status, 0, IBERT_ERR_VALUE_RANGE);   // longer than the stated maximum
  const int n = min(max(len, 0), a.L);
  const int Lp = max((n + 31) & ~31, 32);                      // MMA granularity of both products
  const int q_end = PACKED ? n : a.L;                          // query rows that exist
  const bool live = qt * rows < q_end;                         // (packed: a tile past its sequence's end does nothing)
  bool ok = true;

  if (live && warp == 0) {
    if (ptx::elect_one()) {
      const int z = PACKED ? 0 : batch, slabs = (Lp + 127) >> 7;
      ptx::mbar_arrive_expect_tx(bar_qk, (uint32_t)((1 + slabs) * kSlab));
      for (int c = 0; c < a.rep; ++c)
        ptx::tma_load_3d(ptx::smem_addr(sQ) + c * rows * kHeadDim, &map_q, bar_qk, head * kHeadDim, row0 + qt * rows, z);
      for (int s = 0; s < slabs; ++s)
        ptx::tma_load_3d(ptx::smem_addr(sK) + s * kSlab, &map_kv, bar_qk, a.H + head * kHeadDim, row0 + s * 128, z);
      ptx::mbar_arrive_expect_tx(bar_v, (uint32_t)(slabs * kSlab));
      for (int s = 0; s < slabs; ++s)
        ptx::tma_load_3d(ptx::smem_addr(sV) + s * kSlab, &map_kv, bar_v, 2 * a.H + head * kHeadDim, row0 + s * 128, z);
      // S = Q K^T: K = 64 bytes = two MMA K-steps; N in chunks of at most 256 columns
      ok = ptx::mbar_wait(bar_qk, 0);
      if (ok) {
        ptx::tc_fence_after_sync();
        const uint64_t dq = ptx::make_kmajor_desc(ptx::smem_addr(sQ), 512, ptx::kSwizzle64);
#pragma unroll 1
        for (int n0 = 0; n0 < Lp; n0 += 256) {
          const uint32_t idesc = ptx::make_idesc_i8(128, min(256, Lp - n0), true, true);
          const uint64_t dk = ptx::make_kmajor_desc(ptx::smem_addr(sK) + n0 * kHeadDim, 512, ptx::kSwizzle64);
          ptx::mma_i8_ss(tmem_base + n0, dq, dk, idesc, 0u);
          ptx::mma_i8_ss(tmem_base + n0, dq + 2, dk + 2, idesc, 1u);
        }
        ptx::mma_commit(bar_mma);
      }
    }
    __syncwarp();
  }
  const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
  if (live) ok = ptx::mbar_wait(bar_mma, 0) && ok;
  ok = __all_sync(0xffffffffu, ok);
  const bool active = live && ok && c0 < Lp;

  // ---- i-softmax: maximum, i-exp and sum, probabilities; the thread's CPT scores stay in v
  uint32_t v[CPT];
  if (active) {
    ptx::tc_fence_after_sync();
    ptx::tmem_ld(t_lane + c0, v);
    ptx::tmem_wait_ld();
    if (c0 + CPT > n) {
#pragma unroll
      for (int i = 0; i < CPT; ++i)
        if (c0 + i >= n) v[i] = (uint32_t)INT32_MIN;
    }
    int32_t mx = (int32_t)v[0];
#pragma unroll
    for (int i = 1; i < CPT; ++i) mx = max(mx, (int32_t)v[i]);
    atomicMax(s_max + row, mx);
  }
  __syncthreads();
  const ExpConsts& ek = a.k.e;
  if (active) {
    const uint32_t mx = (uint32_t)s_max[row];
    if (iexp_takes_folded(ek)) {
      const int64_t mk = iexp_folded_addend(ek);
      const int32_t neg_m = -(int32_t)ek.fold_m, wk = iexp_folded_offset(ek, (int32_t)mx);
#pragma unroll
      for (int i = 0; i < CPT; ++i)
        v[i] = iexp_folded((int32_t)(v[i] + (uint32_t)wk) >> ek.s_in, mk, neg_m, ek.q_ln2, ek.q_c);
    } else {
#pragma unroll
      for (int i = 0; i < CPT; ++i) v[i] = iexp_dist_wide(mx - v[i], ek);
    }
    if (c0 + CPT > n) {
#pragma unroll
      for (int i = 0; i < CPT; ++i)
        if (c0 + i >= n) v[i] = 0u;
    }
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < CPT; ++i) sum += v[i];
    atomicAdd(s_sum + row, sum);
  }
  __syncthreads();
  if (active) {
    const RowDivisor rd = make_row_divisor(max(s_sum[row], 1u), ek.p_max);   // sum = 0 only without valid keys
#pragma unroll
    for (int h = 0; h < CPT / 8; ++h) {
      uint32_t w[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int j = h * 8 + i * 4;
        w[i] = ((softmax_quotient(v[j + 3], rd) * 256u + softmax_quotient(v[j + 2], rd)) * 256u + softmax_quotient(v[j + 1], rd)) * 256u +
               softmax_quotient(v[j], rd);
      }
      *reinterpret_cast<uint2*>(sP + sw128_offset((uint32_t)row, (uint32_t)(c0 + h * 8), 128)) = make_uint2(w[0], w[1]);
    }
    ptx::fence_proxy_async_smem();
  }
  ptx::tc_fence_before_sync();
  ok = __syncthreads_and(ok);               // P complete; every score is in registers

  // ---- ctx = P V: K = Lp in steps of 32, accumulator in columns 0..63
  if (live && ok && warp == 0) {
    if (ptx::elect_one()) {
      ok = ptx::mbar_wait(bar_v, 0);
      if (ok) {
        ptx::tc_fence_after_sync();
        // B = V as loaded ([key][head dim], head dim contiguous): the MN-major operand form (bit 16)
        const uint32_t idesc = ptx::make_idesc_i8(128, kHeadDim, false, true) | (1u << 16);       // u8 x s8
#pragma unroll 1
        for (int kk = 0; kk < Lp / 32; ++kk) {
          const uint64_t dp = ptx::make_kmajor_desc(ptx::smem_addr(sP) + (kk >> 2) * 128 * 128, 1024, ptx::kSwizzle128) + 2 * (kk & 3);
          const uint32_t va = ptx::smem_addr(sV) + kk * 32 * kHeadDim;
          const uint64_t dv = (uint64_t)((va & 0x3FFFFu) >> 4) | ((uint64_t)(512 >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) |
                              ((uint64_t)1 << 46) | ((uint64_t)ptx::kSwizzle64 << 61);
          ptx::mma_i8_ss(tmem_base, dp, dv, idesc, kk != 0 ? 1u : 0u);
        }
        ptx::mma_commit(bar_mma);
      }
    }
    ok = __all_sync(0xffffffffu, ok);       // (the warp goes on together: one lane alone waited for V)
  }
  // ---- epilogue: copy 0's lanes, 16 of the 64 context values per thread
  const int q_row = qt * rows + row;
  if (live && ok && quad < quads) {
    ok = __all_sync(0xffffffffu, ptx::mbar_wait(bar_mma, 1) && ok);
    if (ok) {
      ptx::tc_fence_after_sync();
      const int d0 = (warp >> 2) * 16;
      const int64_t half = rounding_half(a.k.c);
      uint32_t o[16], w[4];
      ptx::tmem_ld16(t_lane + d0, o);
      ptx::tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; ++i)
        o[i] = (uint32_t)(a.k.fast ? max(requant_upper((int32_t)o[i], a.k.b2), -127)
                                   : requant_add((int32_t)o[i], a.k.b, half, a.k.c, 127));
#pragma unroll
      for (int i = 0; i < 4; ++i)
        w[i] = pack4_sat_s8((int32_t)o[4 * i], (int32_t)o[4 * i + 1], (int32_t)o[4 * i + 2], (int32_t)o[4 * i + 3]);
      if (q_row < q_end) {
        const int64_t r = PACKED ? (int64_t)row0 + q_row : (int64_t)batch * a.L + q_row;
        *reinterpret_cast<uint4*>(a.out + r * a.H + head * kHeadDim + d0) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
  if (!ok) atomicCAS(a.status, 0, IBERT_ERR_TIMEOUT);
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, a.tmem_cols);
  }
}

struct SmallShape { int rep, q_tiles, cpt; };

// Copies: the most (4, 2, 1) that keep the grid within two CTAs per SM, but enough that a thread's columns fit
// its registers (32: Lp <= 128 rep).  rep = 0: too many pairs for this kernel.
SmallShape small_shape(const ibert_ctx* ctx, int B, int L, int heads) {
  const int Lp = (L + 31) & ~31;
  for (int rep = 4; rep >= 1 && Lp <= 128 * rep; rep >>= 1) {
    const int q_tiles = (L + 128 / rep - 1) / (128 / rep);
    if ((int64_t)B * heads * q_tiles > 2 * (int64_t)ctx->num_sms) continue;
    const int per = (Lp + 4 * rep - 1) / (4 * rep);
    return {rep, q_tiles, per <= 8 ? 8 : (per <= 16 ? 16 : 32)};
  }
  return {0, 0, 0};
}

template <bool PACKED, int CPT>
int launch_small_inst(ibert_ctx* ctx, int grid, int smem, const CUtensorMap& mq, const CUtensorMap& mkv, const SmallAttnArgs& a) {
  static bool attr_dev[kMaxDevices] = {false};
  bool& attr = attr_dev[ctx->device % kMaxDevices];
  if (!attr) {
    if (cudaFuncSetAttribute(attention_small_kernel<PACKED, CPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) != cudaSuccess)
      return IBERT_ERR_CUDA;
    attr = true;
  }
  return launch_pdl(attention_small_kernel<PACKED, CPT>, dim3(grid), dim3(kSmallThreads), (size_t)smem, ctx->stream, 1, mq, mkv, a);
}

}  // namespace

bool attention_small_takes(const ibert_ctx* ctx, int B, int L, int heads, const AttnConsts& k) {
  return k.e.wide_post >= 0 && small_shape(ctx, B, L, heads).rep != 0;
}

int launch_attention_small(ibert_ctx* ctx, const int8_t* qkv, int B, int L, int H, int heads, const AttnConsts& k,
                           const int32_t* lens, int8_t* out, const int32_t* cu_seqlens, int64_t total_rows) {
  const SmallShape sh = small_shape(ctx, B, L, heads);
  if (sh.rep == 0 || k.e.wide_post < 0) return IBERT_ERR_ARG;
  SmallAttnArgs a{};
  a.B = B; a.L = L; a.H = H; a.heads = heads;
  a.n_slabs = (L + 127) / 128; a.rep = sh.rep; a.q_tiles = sh.q_tiles;
  a.tmem_cols = 64;
  while ((int)a.tmem_cols < ((L + 31) & ~31)) a.tmem_cols <<= 1;
  a.k = k; a.lens = cu_seqlens ? cu_seqlens : lens; a.out = out; a.status = ctx->d_status;
  const uint64_t n_rows = cu_seqlens ? (uint64_t)total_rows : (uint64_t)L;
  const uint64_t dims[3] = {(uint64_t)3 * H, n_rows, cu_seqlens ? (uint64_t)1 : (uint64_t)B};
  const uint64_t str[2] = {(uint64_t)3 * H, (uint64_t)3 * H * n_rows};
  const uint32_t box_q[3] = {kHeadDim, (uint32_t)(128 / sh.rep), 1}, box_kv[3] = {kHeadDim, 128, 1};
  CUtensorMap mq, mkv;
  if (int rc = encode_tensor_map(&mq, qkv, 3, dims, str, box_q, 64)) return rc;
  if (int rc = encode_tensor_map(&mkv, qkv, 3, dims, str, box_kv, 64)) return rc;
  const int grid = B * heads * sh.q_tiles;
  const int smem = (1 + 2 * a.n_slabs) * 128 * kHeadDim + a.n_slabs * 128 * 128 + 2 * 128 * 4 + 64 + 1024;
#define IBERT_AS(CPT) \
  return cu_seqlens ? launch_small_inst<true, CPT>(ctx, grid, smem, mq, mkv, a) : launch_small_inst<false, CPT>(ctx, grid, smem, mq, mkv, a)
  if (sh.cpt == 8) IBERT_AS(8);
  if (sh.cpt == 16) IBERT_AS(16);
  IBERT_AS(32);
#undef IBERT_AS
}

}  // namespace ibert
