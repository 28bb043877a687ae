// Standalone integer non-linearities: i-GELU (Algorithm 2), i-softmax (Algorithm 3) and
// residual + i-LayerNorm (Sec. 3.6, Algorithm 4).  All three are HBM-streaming kernels:
// 128-bit coalesced loads of the int32 inputs, all arithmetic in registers, packed int8
// stores.  Rows are owned by one warp and reduced with warp shuffles.
#include <algorithm>
#include <type_traits>

#include "device_utils.cuh"
#include "sm100_ptx.cuh"

namespace ibert {

namespace {

constexpr int kThreads = 256;

// ----------------------------------------------------------------------------- i-GELU
// Each thread converts 4 int4 vectors (16 values); vector j of a thread sits 32 vectors
// after vector j-1 so that every load and store instruction of a warp is contiguous.
// FORM: the upper-word form of i-GELU without / with the pre-shift of the erf argument and without / with a lower clamp
// (GeluConsts::low_free), that of h-GELU, and both functions with the 64-bit product for the other constant sets.  Bound
// by the ALU pipe with shift and clamp (12 of 20 instructions per element), close to HBM without: 2^24 elements
// 16.7 -> 14.5 us.  One form per instance: chosen per element at run time h-GELU takes 15.5 us instead of 13.1.
// The next kernel may start once a block has stored its last values, not before: its blocks would take the places
// of this one's second and third wave.  us, trigger first / last: 2^17 elements 1.69 / 1.64, 2^20 2.60 / 2.13, 2^21
// 3.57 / 2.93, 5 10^6 5.11 / 5.25, 2^24 13.65 / 13.61.
enum { kGeluPlain, kGeluShift, kGeluClamp, kGeluShiftClamp, kGeluExact, kHgelu, kHgeluExact };
template <int FORM>
__global__ void __launch_bounds__(kThreads) gelu_kernel(const int32_t* __restrict__ q, int64_t n,
                                                        GeluConsts k, int8_t* __restrict__ out) {
  ptx::grid_dep_wait();
  const int64_t half = rounding_half(k.c);
  const int64_t n_vec = n >> 2;
  const int32_t rnd_f = (1 << k.s_f) - 1;
  const int lane = threadIdx.x & 31;
  const int64_t warp_global = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int64_t warp_count = ((int64_t)gridDim.x * kThreads) >> 5;
  const int4* q4 = reinterpret_cast<const int4*>(q);
  uint32_t* o4 = reinterpret_cast<uint32_t*>(out);
  auto gelu = [&](int32_t x) {
    if constexpr (FORM == kHgelu) return max(ihgelu_upper(x, k), -127);
    else if constexpr (FORM == kHgeluExact) return ihgelu_to_int8(clamp_sym(x, 32767), k, half);
    else if constexpr (FORM == kGeluExact) return igelu_q16_to_int8(clamp_sym(x, 32767), k, half);
    else {
      const int32_t r = igelu_magnitude_upper<FORM == kGeluShift || FORM == kGeluShiftClamp>(x, k, rnd_f);
      return FORM == kGeluClamp || FORM == kGeluShiftClamp ? max(r, -127) : r;
    }
  };
  for (int64_t base = warp_global * 128; base < n_vec; base += warp_count * 128) {
    int4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t idx = base + j * 32 + lane;
      v[j] = idx < n_vec ? __ldcs(q4 + idx) : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t idx = base + j * 32 + lane;
      if (idx < n_vec) __stcs(o4 + idx, pack4_sat_s8(gelu(v[j].x), gelu(v[j].y), gelu(v[j].z), gelu(v[j].w)));
    }
  }
  ptx::grid_dep_launch();
  // ragged tail (n not a multiple of 4)
  const int64_t tid = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t tail = n_vec << 2;
  if (tid < n - tail) out[tail + tid] = (int8_t)min(gelu(q[tail + tid]), 127);
}

// ----------------------------------------------------------------------------- table look-up GELU
// The alternative the paper argues against: a 65535-entry table of the int8 result for every Q16
// input, built by running the i-GELU kernel once over the ramp -32767 .. 32767 (so its bits are the
// integer function's), then one load per element.
__global__ void __launch_bounds__(kThreads) ramp_q16_kernel(int32_t* __restrict__ q) {
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i < 65535) q[i] = i - 32767;
}

__global__ void __launch_bounds__(kThreads) gelu_lut_kernel(const int32_t* __restrict__ q, int64_t n,
                                                            const int8_t* __restrict__ table,
                                                            int8_t* __restrict__ out) {
  const int64_t n_vec = n >> 2;
  const int4* q4 = reinterpret_cast<const int4*>(q);
  uint32_t* o4 = reinterpret_cast<uint32_t*>(out);
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t idx = (int64_t)blockIdx.x * kThreads + threadIdx.x; idx < n_vec; idx += stride) {
    const int4 v = __ldcs(q4 + idx);
    const uint32_t a = (uint8_t)__ldg(table + clamp_sym(v.x, 32767) + 32767);
    const uint32_t b = (uint8_t)__ldg(table + clamp_sym(v.y, 32767) + 32767);
    const uint32_t c = (uint8_t)__ldg(table + clamp_sym(v.z, 32767) + 32767);
    const uint32_t d = (uint8_t)__ldg(table + clamp_sym(v.w, 32767) + 32767);
    __stcs(o4 + idx, a | (b << 8) | (c << 16) | (d << 24));
  }
  const int64_t tid = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t tail = n_vec << 2;
  if (tid < n - tail) out[tail + tid] = __ldg(table + clamp_sym(q[tail + tid], 32767) + 32767);
}

// ----------------------------------------------------------------------------- i-softmax
// table[i] = i-exp of the pre-shifted distance i, for i = 0 .. d_max
__global__ void __launch_bounds__(kThreads) exp_table_kernel(ExpConsts k, uint32_t* __restrict__ table) {
  const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
  if (i > k.d_max) return;
  const uint32_t d = i << k.s_in;
  const int mode = exp_div_mode(k);
  table[i] = mode == 0 ? iexp_dist<0>(d, k) : (mode == 1 ? iexp_dist<1>(d, k) : iexp_dist<2>(d, k));
}

// ----------------------------------------------------------------------------- i-LayerNorm
// Four consecutive Q16 values of a row, from an int32 or an int16 container (16 / 8 bytes)
template <typename QT>
__device__ __forceinline__ void load_q4(const QT* p, int32_t (&v)[4], bool streaming) {
  if constexpr (sizeof(QT) == 4) {
    const int4 t = streaming ? __ldcs(reinterpret_cast<const int4*>(p)) : *reinterpret_cast<const int4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
    const uint2 t = streaming ? __ldcs(reinterpret_cast<const uint2*>(p)) : *reinterpret_cast<const uint2*>(p);
    // sign-extending halves of a word: one byte permute each
    v[0] = sext_half(t.x, 0); v[1] = sext_half(t.x, 1);
    v[2] = sext_half(t.y, 0); v[3] = sext_half(t.y, 1);
  }
}

// One warp per row, the whole row in registers (VPL int4 vectors per lane).
// FAST: residual rescale and output requantization are in upper-word form (one multiply-add each).
// Resident CTAs per SM the register budget is tuned for: the kernel is latency-bound on the row
// loads, so short rows trade registers for more warps in flight.
constexpr int ln_min_blocks(int vpl) { return vpl <= 4 ? 4 : (vpl <= 6 ? 3 : (vpl <= 8 ? 2 : 1)); }

template <int VPL, bool VEC, bool FAST, typename QT>
__global__ void __launch_bounds__(kThreads, ln_min_blocks(VPL)) layernorm_kernel(const QT* __restrict__ q,
                                                             const int8_t* __restrict__ r, int64_t rows,
                                                             LnConsts k, const int32_t* __restrict__ b_i,
                                                             const int64_t* __restrict__ B_i,
                                                             int8_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int C = k.C;
  const int64_t warp_global = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int64_t warp_count = ((int64_t)gridDim.x * kThreads) >> 5;
  const int64_t half_r = rounding_half(k.c_r);
  for (int64_t row = warp_global; row < rows; row += warp_count) {
    const QT* qr = q + row * C;
    const int8_t* rr = r + row * C;
    int8_t* orow = out + row * C;
    int32_t v[VPL][4];
    int32_t sum = 0;
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int col = 4 * (j * 32 + lane);
      if (VEC) {
        if (col < C) {
          load_q4(qr + col, v[j], true);
          if (k.has_res) {
            const uint32_t rw = __ldcs(reinterpret_cast<const uint32_t*>(rr + col));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int32_t rv = (int32_t)(int8_t)(rw >> (8 * i));
              if (FAST) v[j][i] += requant_upper(rv << k.res_sh, k.b_r);
              else v[j][i] += (int32_t)(((int64_t)rv * k.b_r + half_r) >> k.c_r);
            }
          }
        } else {
          v[j][0] = v[j][1] = v[j][2] = v[j][3] = 0;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          int32_t t = 0;
          if (col + i < C) {
            t = (int32_t)qr[col + i];
            if (k.has_res) t += (int32_t)(((int64_t)rr[col + i] * k.b_r + half_r) >> k.c_r);
          }
          v[j][i] = t;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) sum += v[j][i];
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    // mu = floor(sum / C)
    int32_t mu = sum / C;
    if (sum - mu * C < 0) mu -= 1;
    uint64_t ss = 0;
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int col = 4 * (j * 32 + lane);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int32_t y = (col + i < C) ? v[j][i] - mu : 0;
        v[j][i] = y;
        ss += (uint64_t)((int64_t)y * (int64_t)y);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    uint32_t sigma = warp_isqrt_of_quotient(ss, (uint32_t)C, lane);   // I-Sqrt(floor(ss / C))
    sigma = sigma < 1u ? 1u : sigma;
    const int64_t rho64 = (int64_t)(0x80000000u / sigma);            // floor(2^31 / sigma)
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int col = 4 * (j * 32 + lane);
      int32_t o[4] = {0, 0, 0, 0};
      if (FAST) {
        if (col < C) {
          const int4 bb = __ldg(reinterpret_cast<const int4*>(b_i + col));
          const longlong2 B01 = __ldg(reinterpret_cast<const longlong2*>(B_i + col));
          const longlong2 B23 = __ldg(reinterpret_cast<const longlong2*>(B_i + col + 2));
          const int32_t bv[4] = {bb.x, bb.y, bb.z, bb.w};
          const int64_t Bv[4] = {B01.x, B01.y, B23.x, B23.y};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            // normalized value floor(y * rho / 2^15), then pre-shifted by out_sh (|.| < 2^31)
            const int32_t nrm = (int32_t)(((int64_t)v[j][i] * rho64) >> 15) << k.out_sh;
            o[i] = max(requant_upper_add(nrm, bv[i], Bv[i]), -127);
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (col + i < C) {
            const int32_t nrm = (int32_t)(((int64_t)v[j][i] * rho64) >> 15);
            int64_t t;
            if (k.out_fast) {   // the addend table is pre-shifted: undo it on this path
              t = ((int64_t)nrm * ((int64_t)__ldg(b_i + col + i) << k.out_sh) + __ldg(B_i + col + i)) >> 32;
            } else {
              t = ((int64_t)nrm * (int64_t)__ldg(b_i + col + i) + __ldg(B_i + col + i)) >> k.c;
            }
            t = t > 127 ? 127 : t;
            t = t < -127 ? -127 : t;
            o[i] = (int32_t)t;
          }
        }
      }
      if (VEC) {
        if (col < C) __stcs(reinterpret_cast<uint32_t*>(orow + col), pack4_sat_s8(o[0], o[1], o[2], o[3]));
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (col + i < C) orow[col + i] = (int8_t)o[i];
      }
    }
  }
}

// Same row computation, fed by bulk async copies: every warp streams its rows (Q16 rows and int8 residual rows)
// through a private ring of DEPTH shared-memory slots of R rows, so the loads of the next rows are in flight while
// the current ones are reduced.  Requires C % 16 == 0 (16-byte aligned rows), upper-word constants, and a residual.
// R = 2: a warp finishes two adjacent rows together -- half-warps share what is scalar per row (mean, square root,
// divisions: some 150 instructions), both rows use a constant once it is loaded, and the second row hides the
// latency of the first one's reductions.  One row per warp was bound by instruction issue (31 per element):
// [16384, 768] 19.5 -> 17.5 us with int32, 19.1 -> 16.5 with int16 input, [32768, 1024] 44.1 -> 37.0, [16384, 256] 12.7 -> 8.1.
// FULL: C == 128 VPL, no lane ever runs past the row.
template <int VPL, int R, int DEPTH, typename QT, bool FULL>
__global__ void __launch_bounds__(kThreads, VPL * R > 12 ? 2 : 3)
layernorm_pipe_kernel(const QT* __restrict__ q, const int8_t* __restrict__ r, int64_t rows, LnConsts k,
                      const int32_t* __restrict__ b_i, const int64_t* __restrict__ B_i, int8_t* __restrict__ out,
                      int32_t* status) {
  extern __shared__ __align__(128) uint8_t ln_smem[];
  // (row groups of a warp; 32 bits where 64 would spill: int32 pairs of 257 to 768 channels, 16384 x 768 from HBM 18.7 ->
  // 18.2 us, 32768 x 640 26.8 -> 26.1, 8192 x 768 10.8 -> 11.0; int16 pairs lose 2 % with it, 1024 channels keep their time)
  using Index = std::conditional_t<R == 2 && (VPL == 4 || VPL == 6) && sizeof(QT) == 4, uint32_t, int64_t>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int C = k.C;
  const uint32_t q_bytes = (uint32_t)C * (uint32_t)sizeof(QT), r_bytes = (uint32_t)C;
  const uint32_t slot_bytes = R * (q_bytes + r_bytes);           // multiple of 16: R Q16 rows, then R residual rows
  uint8_t* ring = ln_smem + (size_t)warp * DEPTH * slot_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ln_smem + (size_t)(kThreads / 32) * DEPTH * slot_bytes) + warp * DEPTH;
  // the per-channel tables, copied once per CTA: every row reads all of them
  int64_t* s_B = reinterpret_cast<int64_t*>(ln_smem + (size_t)(kThreads / 32) * DEPTH * slot_bytes + (kThreads / 32) * DEPTH * 8);
  int32_t* s_b = reinterpret_cast<int32_t*>(s_B + C);
  const Index groups = (Index)((rows + R - 1) / R);
  const Index warp_global = (Index)(((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5);
  const Index warp_count = (Index)(((int64_t)gridDim.x * kThreads) >> 5);

  for (int i = threadIdx.x; i < C; i += kThreads) {        // constants, not outputs of the previous kernel
    s_b[i] = __ldg(b_i + i);
    s_B[i] = __ldg(B_i + i);
  }
  __syncthreads();

  ptx::grid_dep_launch();
  ptx::grid_dep_wait();              // the kernel that produced q (and r) has completed
  auto issue = [&](Index group, int slot) {
    const uint32_t bar = ptx::smem_addr(bars + slot);
    const uint32_t dst = ptx::smem_addr(ring + (size_t)slot * slot_bytes);
    const int64_t row = (int64_t)group * R;
    const uint32_t n = (uint32_t)min((int64_t)R, rows - row);
    ptx::mbar_arrive_expect_tx(bar, n * (q_bytes + r_bytes));
    ptx::bulk_load_1d(dst, q + row * C, n * q_bytes, bar);
    ptx::bulk_load_1d(dst + R * q_bytes, r + row * C, n * r_bytes, bar);
  };
  if (lane == 0) {
    for (int s = 0; s < DEPTH; ++s) ptx::mbar_init(ptx::smem_addr(bars + s), 1);
    ptx::fence_mbar_init();
    for (int s = 0; s < DEPTH; ++s) {
      const Index group = warp_global + (Index)s * warp_count;
      if (group < groups) issue(group, s);
    }
  }
  __syncwarp();

  int slot = 0;
  uint32_t phase = 0;
  for (Index group = warp_global; group < groups; group += warp_count) {
    const bool ok = __all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_addr(bars + slot), phase));
    if (!ok) {
      if (lane == 0) atomicCAS(status, 0, IBERT_ERR_TIMEOUT);
      // the copies already issued into the other slots must land (or run out of time as well)
      // before this CTA's shared memory is given up
      for (int j = 1; j < DEPTH; ++j) {
        int s2 = slot + j;
        uint32_t ph2 = phase;
        if (s2 >= DEPTH) { s2 -= DEPTH; ph2 ^= 1; }
        if (group + (Index)j * warp_count < groups) ptx::mbar_wait(ptx::smem_addr(bars + s2), ph2);
      }
      break;
    }
    const uint8_t* sq = ring + (size_t)slot * slot_bytes;
    // (an odd row count: the last group has one row, and in place of the other lies whatever was there.  Its
    // statistics are discarded, so the sums are unsigned and both square roots take any bits; all that it shares with
    // the first row is the number of rounds of the root search, of which more than a row needs change nothing)
    int32_t v[R][VPL][4];
    uint32_t rw[R][VPL];
#pragma unroll
    for (int h = 0; h < R; ++h)
#pragma unroll
      for (int j = 0; j < VPL; ++j) {
        const int col = 4 * (j * 32 + lane);
        if (FULL || col < C) {
          load_q4(reinterpret_cast<const QT*>(sq + h * q_bytes) + col, v[h][j], false);
          rw[h][j] = *reinterpret_cast<const uint32_t*>(sq + R * q_bytes + h * r_bytes + col);
        } else {
          v[h][j][0] = v[h][j][1] = v[h][j][2] = v[h][j][3] = 0;
          rw[h][j] = 0;
        }
      }
    __syncwarp();                                    // every lane has its copy: the slot can be refilled
    if (lane == 0) {
      const Index next = group + (Index)DEPTH * warp_count;
      if (next < groups) issue(next, slot);
    }
    if (++slot == DEPTH) { slot = 0; phase ^= 1; }

    // one pass over a row: sum v and sum v^2 (columns past C hold zeros); the centred sum of squares
    // follows exactly in integers: sum (v - mu)^2 = sum v^2 - 2 mu sum v + C mu^2
    int32_t sum = 0;
    uint64_t s2 = 0;
#pragma unroll
    for (int h = 0; h < R; ++h) {
      uint32_t t = 0;
      uint64_t t2 = 0;
#pragma unroll
      for (int j = 0; j < VPL; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int32_t res = (sext_byte(rw[h][j], i) * k.res_nb + k.res_nhalf) >> k.res_nc;   // rescaled (narrow form)
          v[h][j][i] = (int32_t)((uint32_t)v[h][j][i] + (uint32_t)res);
          t += (uint32_t)v[h][j][i];
          t2 += (uint64_t)((int64_t)v[h][j][i] * (int64_t)v[h][j][i]);
        }
      t = __reduce_add_sync(0xffffffffu, t);
      // a lane's share is below 2^50 (|v| <= 2^21, at most 64 values): two 25-bit halves reduce as 32-bit sums
      t2 = (uint64_t)__reduce_add_sync(0xffffffffu, (uint32_t)t2 & 0x1ffffffu) +
           ((uint64_t)__reduce_add_sync(0xffffffffu, (uint32_t)(t2 >> 25)) << 25);
      if (h == 0 || lane >= 16) { sum = (int32_t)t; s2 = t2; }            // (two rows: the upper half-warp takes the second)
    }
    // mu = floor(sum / C) and I-Sqrt(floor(ss / C)).  Row pairs of more than 256 channels: a product with the reciprocal,
    // off by one at most, and Newton's iteration in every lane, instead of a division and six rounds of votes (16384 x 768
    // 14.9 -> 14.3 us with int32, 14.7 -> 14.2 with int16 input, inputs from HBM 18.7 -> 18.2 and 16.6 -> 16.2; 32768 x 512 20.7
    // -> 20.1; at 256 channels 20000 rows behind each other 9.0 -> 10.3, so those and single rows keep the search)
    LnNorm own;
    if constexpr (R == 2 && VPL > 2) {
      int32_t mu = __mulhi(sum, (int32_t)k.mean_m) >> k.mean_sh;
      const int32_t rest = (int32_t)((uint32_t)sum - (uint32_t)mu * (uint32_t)C);
      mu += rest >= C ? 1 : (rest < 0 ? -1 : 0);
      own = ln_norm(mu, ln_root<3>(s2 + (uint64_t)((int64_t)mu * ((int64_t)C * mu - 2 * (int64_t)sum)), (uint32_t)C, k.root_k));
    } else {
      int32_t mu = sum / C;
      if (sum - mu * C < 0) mu -= 1;
      const uint64_t ss = s2 + (uint64_t)((int64_t)mu * ((int64_t)C * mu - 2 * (int64_t)sum));
      own = ln_norm(mu, warp_isqrt_of_quotient<32 / R>(ss, (uint32_t)C, lane));
    }
    LnNorm norm[R];
#pragma unroll
    for (int h = 0; h < R; ++h)
      norm[h] = R == 1 ? own : LnNorm{__shfl_sync(0xffffffffu, own.scale, 16 * h), __shfl_sync(0xffffffffu, own.shift, 16 * h),
                                      __shfl_sync(0xffffffffu, own.rho, 16 * h)};
    int8_t* orow = out + (int64_t)group * R * C;
    const bool second = R == 1 || (int64_t)group * R + 1 < rows;
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int col = 4 * (j * 32 + lane);
      if (FULL || col < C) {
        const int4 bb = *reinterpret_cast<const int4*>(s_b + col);
        const longlong2 B01 = *reinterpret_cast<const longlong2*>(s_B + col);
        const longlong2 B23 = *reinterpret_cast<const longlong2*>(s_B + col + 2);
        const int32_t bv[4] = {bb.x, bb.y, bb.z, bb.w};
        const int64_t Bv[4] = {B01.x, B01.y, B23.x, B23.y};
#pragma unroll
        for (int h = 0; h < R; ++h) {
          int32_t o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            o[i] = max(requant_upper_add(ln_normalize(v[h][j][i], norm[h]) << k.out_sh, bv[i], Bv[i]), -127);
          if (h == 0 || second) __stcs(reinterpret_cast<uint32_t*>(orow + (size_t)h * C + col), pack4_sat_s8(o[0], o[1], o[2], o[3]));
        }
      }
    }
  }
}

// ----------------------------------------------------------------------------- embedding gather
// One warp per token: 16 bytes of the word row and of the position row per lane and step.
// Packed batches (cu != nullptr: [B + 1] first rows of the sequences): the position of token t is
// its distance from the first row of its sequence, found by bisection; a position beyond the
// position table (a sequence longer than the stated maximum) records IBERT_ERR_VALUE_RANGE.
__global__ void __launch_bounds__(kThreads) embed_gather_kernel(const int32_t* __restrict__ ids, int64_t T, int L,
                                                                const int8_t* __restrict__ word, int64_t V,
                                                                const int8_t* __restrict__ pos, int H,
                                                                int32_t* __restrict__ q, int8_t* __restrict__ r,
                                                                int32_t* status, const int32_t* __restrict__ cu, int B) {
  const int lane = threadIdx.x & 31;
  const int64_t warp_global = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int64_t warp_count = ((int64_t)gridDim.x * kThreads) >> 5;
  for (int64_t t = warp_global; t < T; t += warp_count) {
    int64_t id = __ldg(ids + t);
    if (id < 0 || id >= V) {
      if (lane == 0) atomicCAS(status, 0, IBERT_ERR_VALUE_RANGE);
      id = 0;
    }
    int64_t p = t % L;
    if (cu) {
      int lo = 0, hi = B;                    // the last sequence whose first row is <= t
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((int64_t)__ldg(cu + mid) <= t) lo = mid; else hi = mid;
      }
      p = t - (int64_t)__ldg(cu + lo);
      if (p >= L) {
        if (lane == 0) atomicCAS(status, 0, IBERT_ERR_VALUE_RANGE);
        p = L - 1;
      }
    }
    const int8_t* wrow = word + id * H;
    const int8_t* prow = pos + p * H;
    for (int c = lane * 16; c < H; c += 512) {
      const uint4 wv = __ldg(reinterpret_cast<const uint4*>(wrow + c));
      const uint4 pv = __ldg(reinterpret_cast<const uint4*>(prow + c));
      const uint32_t ww[4] = {wv.x, wv.y, wv.z, wv.w};
      int32_t o[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) o[i] = (int32_t)(int8_t)(ww[i >> 2] >> (8 * (i & 3)));
      int4* qd = reinterpret_cast<int4*>(q + t * H + c);
#pragma unroll
      for (int i = 0; i < 4; ++i) qd[i] = make_int4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
      *reinterpret_cast<uint4*>(r + t * H + c) = pv;
    }
  }
}

// ----------------------------------------------------------------------------- wait self-test
// Two warps wait on an mbarrier nobody arrives on, with a short limit: one by the polling form of the
// bounded wait (mbar_wait_ns), one by the parked form the GEMM feeder threads use (mbar_wait_parked_ns).
// When BOTH limits have run out the kernel records IBERT_ERR_TIMEOUT like every kernel of the library
// does, and returns normally.
__global__ void __launch_bounds__(64) wait_timeout_kernel(uint64_t limit_ns, int32_t* status) {
  __shared__ uint64_t bar;
  __shared__ int expired;
  if (threadIdx.x == 0) {
    ptx::mbar_init(ptx::smem_addr(&bar), 1);
    ptx::fence_mbar_init();
    expired = 0;
  }
  __syncthreads();
  const bool ok = (threadIdx.x < 32) ? __all_sync(0xffffffffu, ptx::mbar_wait_ns(ptx::smem_addr(&bar), 0, limit_ns))
                                     : __all_sync(0xffffffffu, ptx::mbar_wait_parked_ns(ptx::smem_addr(&bar), 0, limit_ns));
  if (!ok && (threadIdx.x & 31) == 0) atomicAdd(&expired, 1);
  __syncthreads();
  if (threadIdx.x == 0 && expired == 2) atomicCAS(status, 0, IBERT_ERR_TIMEOUT);
}

// Row cu[b] of x (the first token of sequence b of a packed batch) -> row b of out; one warp per row.
__global__ void __launch_bounds__(kThreads) gather_first_rows_kernel(const int8_t* __restrict__ x, const int32_t* __restrict__ cu,
                                                                     int B, int H, int8_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int b = (int)(((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5);
  if (b >= B) return;
  const int8_t* src = x + (int64_t)__ldg(cu + b) * H;
  for (int c = lane * 16; c < H; c += 512)
    *reinterpret_cast<uint4*>(out + (int64_t)b * H + c) = __ldg(reinterpret_cast<const uint4*>(src + c));
}

// i-softmax with LPR lanes per row (32 / LPR rows per warp side by side) and VPL 16-byte vectors per lane.  Bound by
// instruction issue with one row per warp: maximum, sum and the division by the sum cost a lane the same for
// four values as for 16 (34 instructions per element).  Few lanes per row and many values per lane keep that
// share small, and i-exp takes quotient and shift from one multiply-high: [196608, 128] 37.5 -> 22.6 us (0.85 of the
// measured copy bandwidth), [262144, 512] 151 -> 108, [100000, 101] 25.4 -> 18.8, [200000, 33] 47.7 -> 15.1.
// Rows of any length: the vectors are the 16-byte aligned ones that cover the row, elements of the neighbouring rows
// in the first and the last are masked.
// FULL: 4 LPR VPL elements per row exactly, nothing to mask.  EXP: the exponential's form.
enum { kExpFold = 0, kExpFoldShift = 1, kExpTable = 2 };
template <int LPR, int VPL, bool FULL, int EXP>
__global__ void __launch_bounds__(kThreads, VPL > 4 ? 3 : 4) softmax_group_kernel(const int32_t* __restrict__ q, int64_t rows, int L,
                                                                     RowExpConsts k, uint8_t* __restrict__ out,
                                                                     const uint32_t* __restrict__ table) {
  constexpr int kRows = 32 / LPR;
  const int lane = threadIdx.x & 31, li = lane % LPR;
  const int64_t warp_global = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int64_t warp_count = ((int64_t)gridDim.x * kThreads) >> 5;
  ptx::grid_dep_launch();
  ptx::grid_dep_wait();
  const int64_t total = rows * L;
  const int4* q4 = reinterpret_cast<const int4*>(q);
  const int32_t wk = k.q_b - k.s_out * (int32_t)k.q_ln2 + k.row_add;
  for (int64_t row0 = warp_global * kRows; row0 < rows; row0 += warp_count * kRows) {
    const int64_t row = row0 + lane / LPR;
    const bool live = row < rows;
    const int64_t vec0 = (row * L) >> 2;                      // first vector of the row
    const int off = FULL ? 0 : (int)((row * L) & 3);          // elements of the row before in it
    uint32_t v[VPL][4];
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int vi = li + LPR * j;
      int4 t = make_int4(INT32_MIN, INT32_MIN, INT32_MIN, INT32_MIN);
      if (live && (FULL || 4 * vi < off + L)) {
        if (FULL || 4 * (vec0 + vi) + 3 < total) t = __ldcs(q4 + vec0 + vi);
        else {                                                // the tensor's last, partial vector
          const int32_t* e = q + 4 * (vec0 + vi);
          const int left = (int)(total - 4 * (vec0 + vi));
          t.x = e[0];
          if (left > 1) t.y = e[1];
          if (left > 2) t.z = e[2];
        }
      }
      v[j][0] = t.x; v[j][1] = t.y; v[j][2] = t.z; v[j][3] = t.w;
      if constexpr (!FULL) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if ((uint32_t)(4 * vi + i - off) >= (uint32_t)L) v[j][i] = (uint32_t)INT32_MIN;
      }
    }
    int32_t mx = INT32_MIN;
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      mx = __vimax3_s32(mx, (int32_t)v[j][0], (int32_t)v[j][1]);
      mx = __vimax3_s32(mx, (int32_t)v[j][2], (int32_t)v[j][3]);
    }
    if constexpr (LPR == 32) mx = __reduce_max_sync(0xffffffffu, mx);
    else {
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t d = (uint32_t)mx - v[j][i];
        if constexpr (EXP == kExpTable) v[j][i] = __ldg(table + min(d >> k.s_in, k.d_max));
        else {
          // d' = min(d >> s_in, 31 q_ln2); n = floor(d' / q_ln2) + s_out; e = ((q_b - r)^2 + q_c) >> n
          if constexpr (EXP == kExpFoldShift) d >>= k.s_in;
          d = min(d, k.d_max) + (uint32_t)k.row_add;
          const uint32_t n = __umulhi(d, k.row_m) + (uint32_t)k.s_out;
          const int32_t t = (int32_t)(n * k.q_ln2) + (wk - (int32_t)d);
          v[j][i] = shr_clamped((uint32_t)(t * t + k.q_c), n);
        }
      }
      sum = sum + v[j][0] + v[j][1];
      sum = sum + v[j][2] + v[j][3];
    }
    if constexpr (!FULL) {
      // masked elements sit at INT32_MIN: their exponential is 0 unless the whole row is within 31 ln2 of it
      const bool low = ((uint32_t)(mx - INT32_MIN) >> k.s_in) < k.d_max;
      if (__any_sync(0xffffffffu, low)) {
        sum = 0;
#pragma unroll
        for (int j = 0; j < VPL; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if ((uint32_t)(4 * (li + LPR * j) + i - off) >= (uint32_t)L) v[j][i] = 0u;
            sum += v[j][i];
          }
      }
    }
    if constexpr (LPR == 32) sum = __reduce_add_sync(0xffffffffu, sum);
    else {
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    const RowDivisor rd = make_row_divisor(max(sum, 1u), k.p_max);
    const bool nopre = __all_sync(0xffffffffu, rd.pre == 0);
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      uint32_t p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = softmax_quotient_nopre(nopre ? v[j][i] : v[j][i] << rd.pre, rd);
      const uint32_t w = __byte_perm(__byte_perm(p[0], p[1], 0x0040), __byte_perm(p[2], p[3], 0x0040), 0x5410);
      const int vi = li + LPR * j, c = 4 * vi - off;          // the word's first column
      if (live && (FULL || (c >= 0 && c + 3 < L))) __stcs(reinterpret_cast<uint32_t*>(out) + vec0 + vi, w);
      else if (!FULL && live) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (c + i >= 0 && c + i < L) out[4 * (vec0 + vi) + i] = (uint8_t)p[i];
      }
    }
  }
}

int grid_for(ibert_ctx* ctx, int64_t work_warps, int max_ctas_per_sm) {
  const int64_t ctas = (work_warps + (kThreads / 32) - 1) / (kThreads / 32);
  const int64_t cap = (int64_t)ctx->num_sms * max_ctas_per_sm;
  return (int)(ctas < 1 ? 1 : (ctas > cap ? cap : ctas));
}

// grid of at most one wave of resident CTAs of `kernel` (its registers decide how many an SM holds: a larger
// grid of grid-stride CTAs runs as a full wave plus a partial one)
template <typename Kernel>
int wave_grid(ibert_ctx* ctx, Kernel kernel, int64_t work_warps) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, 0) != cudaSuccess || per_sm < 1) per_sm = 1;
  return grid_for(ctx, work_warps, std::min(per_sm, 8));
}

int check_launch() { return cudaGetLastError() == cudaSuccess ? IBERT_OK : IBERT_ERR_CUDA; }

}  // namespace

int launch_wait_timeout(ibert_ctx* ctx, uint64_t limit_ns) {
  wait_timeout_kernel<<<1, 64, 0, ctx->stream>>>(limit_ns, ctx->d_status);
  return check_launch();
}

int launch_embed_gather(ibert_ctx* ctx, const int32_t* ids, int64_t T, int L, const int8_t* word, int64_t V,
                        const int8_t* pos, int H, int32_t* q, int8_t* r, const int32_t* cu_seqlens, int B) {
  if (T == 0) return IBERT_OK;
  embed_gather_kernel<<<grid_for(ctx, T, 8), kThreads, 0, ctx->stream>>>(ids, T, L, word, V, pos, H, q, r,
                                                                          ctx->d_status, cu_seqlens, B);
  return check_launch();
}

int launch_gather_first_rows(ibert_ctx* ctx, const int8_t* x, const int32_t* cu_seqlens, int B, int H, int8_t* out) {
  if (B == 0) return IBERT_OK;
  gather_first_rows_kernel<<<(B + kThreads / 32 - 1) / (kThreads / 32), kThreads, 0, ctx->stream>>>(x, cu_seqlens, B, H, out);
  return check_launch();
}

int launch_gelu_table(ibert_ctx* ctx, const GeluConsts& k, int32_t* ramp_scratch, int8_t* table) {
  ramp_q16_kernel<<<(65535 + kThreads - 1) / kThreads, kThreads, 0, ctx->stream>>>(ramp_scratch);
  if (int rc = check_launch()) return rc;
  return launch_gelu(ctx, ramp_scratch, 65535, k, table);
}

int launch_gelu_lut(ibert_ctx* ctx, const int32_t* q, int64_t n, const int8_t* table, int8_t* out) {
  if (n == 0) return IBERT_OK;
  const int64_t warps = ((n >> 2) + 31) / 32 / 8 + 1;          // ~8 vectors per thread
  gelu_lut_kernel<<<wave_grid(ctx, gelu_lut_kernel, warps), kThreads, 0, ctx->stream>>>(q, n, table, out);
  return check_launch();
}

int launch_gelu(ibert_ctx* ctx, const int32_t* q, int64_t n, const GeluConsts& k, int8_t* out) {
  if (n == 0) return IBERT_OK;
  const int64_t warps = ((n >> 2) + 127) / 128 + 1;
#define IBERT_GELU(F) \
  return launch_pdl(gelu_kernel<F>, dim3(wave_grid(ctx, gelu_kernel<F>, warps)), dim3(kThreads), 0, ctx->stream, 1, q, n, k, out)
  if (k.hard && k.fast) IBERT_GELU(kHgelu);
  if (k.hard) IBERT_GELU(kHgeluExact);
  if (!k.fast) IBERT_GELU(kGeluExact);
  if (k.low_free && k.s_in == 0) IBERT_GELU(kGeluPlain);
  if (k.low_free) IBERT_GELU(kGeluShift);
  if (k.s_in == 0) IBERT_GELU(kGeluClamp);
  IBERT_GELU(kGeluShiftClamp);
#undef IBERT_GELU
}

int launch_exp_table(ibert_ctx* ctx, const ExpConsts& k, uint32_t* table) {
  exp_table_kernel<<<(int)((k.d_max + kThreads) / kThreads), kThreads, 0, ctx->stream>>>(k, table);
  return check_launch();
}

int launch_softmax(ibert_ctx* ctx, const int32_t* q, int64_t rows, int L, const RowExpConsts& k, uint8_t* out,
                   const uint32_t* exp_table) {
  if (rows == 0) return IBERT_OK;
  const bool vec = (L % 4) == 0;
  // lanes per row: the fewest (4 to 32) that hold the row in at most four vectors each; L > 509: 32 of eight
  const int vecs = (L + (vec ? 0 : 3) + 3) / 4;
  int lpr = 4;
  while (lpr < 32 && vecs > 4 * lpr) lpr *= 2;
  const int vpl = std::max((vecs + lpr - 1) / lpr, 2);
  const bool full = vec && L == 4 * lpr * vpl;
  const int form = exp_table ? kExpTable : (k.s_in == 0 ? kExpFold : kExpFoldShift);
  const int64_t warps = (rows + 32 / lpr - 1) / (32 / lpr);
#define IBERT_SG3(LPR, VPL, FULL, EXP)                                                                       \
  return launch_pdl(softmax_group_kernel<LPR, VPL, FULL, EXP>,                                               \
                    dim3(wave_grid(ctx, softmax_group_kernel<LPR, VPL, FULL, EXP>, warps)), dim3(kThreads), 0, \
                    ctx->stream, 1, q, rows, L, k, out, exp_table)
#define IBERT_SG2(LPR, VPL, FULL)                                             \
  do {                                                                        \
    if (form == kExpFold) IBERT_SG3(LPR, VPL, FULL, kExpFold);                \
    else if (form == kExpFoldShift) IBERT_SG3(LPR, VPL, FULL, kExpFoldShift); \
    else IBERT_SG3(LPR, VPL, FULL, kExpTable);                                \
  } while (0)
#define IBERT_SG(LPR)                            \
  do {                                           \
    if (vpl == 2) IBERT_SG2(LPR, 2, false);      \
    else if (vpl == 3) IBERT_SG2(LPR, 3, false); \
    else if (full) IBERT_SG2(LPR, 4, true);      \
    else IBERT_SG2(LPR, 4, false);               \
  } while (0)
  if (vpl > 8) IBERT_SG2(32, 9, false);            // (1022 and 1023 elements off a 16-byte boundary)
  else if (vpl > 4) IBERT_SG2(32, 8, false);
  else if (lpr == 4) IBERT_SG(4);
  else if (lpr == 8) IBERT_SG(8);
  else if (lpr == 16) IBERT_SG(16);
  else IBERT_SG(32);
  return IBERT_ERR_ARG;
#undef IBERT_SG
#undef IBERT_SG2
#undef IBERT_SG3
}

template <typename QT>
static int launch_layernorm_t(ibert_ctx* ctx, const QT* q, const int8_t* r, int64_t rows, const LnConsts& k,
                              const int32_t* d_b, const int64_t* d_B, int8_t* out) {
  if (rows == 0) return IBERT_OK;
  const bool vec = (k.C % 4) == 0;
  const int vpl = (k.C + 127) / 128;
  const bool fast = vec && k.out_fast && (!k.has_res || k.res_fast);
  if (fast && k.has_res && k.res_narrow && k.C % 16 == 0 && k.C <= 1024) {
    // streaming variant: per-warp ring of row slots filled by bulk async copies.  Two rows per warp once the warps of the
    // resident wave have work that way; below, one row per warp keeps more warps busy.  From 257 to 768 channels the
    // two cross later, int16 rows just past one full wave of single rows, int32 rows a third further (us with one row /
    // with two, behind an unrelated kernel and, in brackets, call behind call; 1.6 us of the former are that kernel):
    //   C = 256 int32   3553 rows 5.1 / 5.0 (3.1 / 3.6)   3800 5.4 / 5.0 (3.9 / 3.7)   4735 5.6 / 5.1
    //   C = 768 int16   3553 rows 6.5 / 6.9 (4.5 / 6.4)   3800 7.4 / 7.0 (5.4 / 6.4)   4735 7.5 / 7.1
    //   C = 768 int32   3553 rows 6.7 / 7.4 (4.7 / 6.7)   4000 7.4 / 7.4 (5.5 / 6.8)   4737 7.6 / 7.7 (7.0 / 6.8)   7000 9.8 / 9.1
    //   C = 1024 int32  3553 rows 7.8 / 8.3 (6.7 / 6.5)   3800 8.7 / 8.3 (6.9 / 6.5)   7000 11.6 / 10.5 (9.6 / 10.8)
    // (one-row slots are double-buffered, two-row slots single: the registers are the second buffer)
    const size_t smem = (size_t)(kThreads / 32) * 2 * (size_t)k.C * (sizeof(QT) + 1) + (kThreads / 32) * 2 * 8 +
                        (size_t)k.C * 12;                  // rows in flight, barriers, the two tables
    const int line = k.C <= 256 || k.C > 768 ? 24 : sizeof(QT) == 4 ? 32 : 25;       // rows per SM
    const bool two = rows >= (int64_t)ctx->num_sms * line;
    // one wave of resident CTAs: by registers three per SM (two for two rows of more than 768 channels), fewer when
    // the row slots take more shared memory (C = 1024 with int32 input: two)
    const int by_regs = two && k.C > 768 ? 2 : 3;
    const int per_sm = (int)std::min<size_t>(by_regs, (size_t)(227 * 1024) / (smem + 1024));
    const int64_t groups = two ? (rows + 1) / 2 : rows;
    const int pgrid = (int)std::min<int64_t>((groups + 7) / 8, (int64_t)ctx->num_sms * std::max(per_sm, 1));
#define IBERT_LNP3(V, R, F)                                                                                 \
  do {                                                                                                      \
    static bool attr_dev[kMaxDevices] = {false};                                                            \
    bool& attr = attr_dev[ctx->device % kMaxDevices];                                                       \
    if (!attr) {                                                                                            \
      if (cudaFuncSetAttribute(layernorm_pipe_kernel<V, R, 3 - R, QT, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                               100 * 1024) != cudaSuccess) return IBERT_ERR_CUDA;                           \
      attr = true;                                                                                          \
    }                                                                                                       \
    return launch_pdl(layernorm_pipe_kernel<V, R, 3 - R, QT, F>, dim3(pgrid), dim3(kThreads), smem, ctx->stream, 1, q, r, \
                      rows, k, d_b, d_B, out, ctx->d_status);                                               \
  } while (0)
#define IBERT_LNP(V)                          \
  do {                                        \
    const bool full = k.C == 128 * V;         \
    if (two && full) IBERT_LNP3(V, 2, true);  \
    if (two) IBERT_LNP3(V, 2, false);         \
    if (full) IBERT_LNP3(V, 1, true);         \
    IBERT_LNP3(V, 1, false);                  \
  } while (0)
    if (k.C <= 256) IBERT_LNP(2);
    if (k.C <= 512) IBERT_LNP(4);
    if (k.C <= 768) IBERT_LNP(6);
    IBERT_LNP(8);
#undef IBERT_LNP
#undef IBERT_LNP3
  }
#define IBERT_LN(V)                                                                                              \
  do {                                                                                                           \
    if (fast) layernorm_kernel<V, true, true, QT><<<wave_grid(ctx, layernorm_kernel<V, true, true, QT>, rows), kThreads, 0, ctx->stream>>>(q, r, rows, k, d_b, d_B, out);  \
    else if (vec) layernorm_kernel<V, true, false, QT><<<wave_grid(ctx, layernorm_kernel<V, true, false, QT>, rows), kThreads, 0, ctx->stream>>>(q, r, rows, k, d_b, d_B, out); \
    else layernorm_kernel<V, false, false, QT><<<wave_grid(ctx, layernorm_kernel<V, false, false, QT>, rows), kThreads, 0, ctx->stream>>>(q, r, rows, k, d_b, d_B, out);     \
  } while (0)
  if (vpl <= 2) IBERT_LN(2);
  else if (vpl <= 4) IBERT_LN(4);
  else if (vpl <= 6) IBERT_LN(6);
  else if (vpl <= 8) IBERT_LN(8);
  else IBERT_LN(16);
#undef IBERT_LN
  return check_launch();
}

int launch_layernorm(ibert_ctx* ctx, const int32_t* q, const int8_t* r, int64_t rows, const LnConsts& k,
                     const int32_t* d_b, const int64_t* d_B, int8_t* out) {
  return launch_layernorm_t<int32_t>(ctx, q, r, rows, k, d_b, d_B, out);
}

int launch_layernorm_i16(ibert_ctx* ctx, const int16_t* q, const int8_t* r, int64_t rows, const LnConsts& k,
                         const int32_t* d_b, const int64_t* d_B, int8_t* out) {
  return launch_layernorm_t<int16_t>(ctx, q, r, rows, k, d_b, d_B, out);
}

}  // namespace ibert
