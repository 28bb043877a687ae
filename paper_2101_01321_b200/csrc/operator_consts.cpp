// The constants of operator calls (scales and per-channel arrays come with every call) and how long the context keeps
// them.  No CUDA call of its own: device tables come from cached_upload.
#include <algorithm>
#include <cstring>

#include "ibert_internal.h"

namespace ibert {

// Hash of a constant table, eight bytes at a step in four chains (byte by byte FNV-1a took 35 us for the two
// tables of a 3072-channel layer).  It only finds a candidate: the bytes decide.
uint64_t table_hash(const void* data, size_t bytes, uint64_t seed) {
  const unsigned char* p = static_cast<const unsigned char*>(data);
  constexpr uint64_t kPrime = 0x9e3779b97f4a7c15ull;
  uint64_t h[4] = {seed ^ 1469598103934665603ull, seed + kPrime, seed ^ (kPrime << 7), seed + bytes};
  size_t i = 0;
  for (; i + 32 <= bytes; i += 32)
    for (int j = 0; j < 4; ++j) {
      uint64_t w;
      std::memcpy(&w, p + i + 8 * j, 8);
      h[j] = (h[j] ^ w) * kPrime;
      h[j] ^= h[j] >> 29;
    }
  for (; i < bytes; ++i) h[i & 3] = (h[i & 3] ^ p[i]) * kPrime;
  uint64_t r = h[0];
  for (int j = 1; j < 4; ++j) r = ((r ^ (r >> 31)) + h[j]) * kPrime;
  return r ^ (r >> 32);
}

namespace {

// Constants of an operator call by the bytes they follow from: `scalars`, then the arrays.  Deriving them takes 3 to
// 10 us a call for 768 to 3072 channels and finding their tables again by content as long as comparing the arrays
// here (0.1 to 0.4 us), so a caller with its own graph pays for them twice per layer and not once per call: the first
// call leaves its key only.  Constants that never return (scales taken from every batch) then cost no copy of their
// arrays and push nothing out.  `derive` fills the entry; nothing is kept when it fails.
struct Bytes {
  const void* p;
  size_t n;
};
template <typename Derive>
int operator_consts(ibert_ctx* ctx, uint64_t tag, const double (&scalars)[5], const Bytes (&arrays)[2],
                    OperatorConsts* once, OperatorConsts** out, Derive&& derive) {
  // a sample finds the candidate: the scalars, 32 words of each array
  uint64_t key = table_hash(scalars, sizeof(scalars), tag);
  for (const Bytes& a : arrays)
    for (size_t i = 0, step = std::max<size_t>(a.n / 32, 8); i + 8 <= a.n; i += step) {
      uint64_t w;
      std::memcpy(&w, static_cast<const unsigned char*>(a.p) + i, 8);
      key = (key ^ w) * 0x9e3779b97f4a7c15ull;
      key ^= key >> 31;
    }
  const uint64_t sample = key;
  const size_t total = sizeof(scalars) + arrays[0].n + arrays[1].n;
  for (auto it = ctx->consts.find(key); it != ctx->consts.end(); it = ctx->consts.find(++key)) {
    const std::vector<unsigned char>& from = it->second.from;
    if (from.size() == total && std::memcmp(from.data(), scalars, sizeof(scalars)) == 0 &&
        std::memcmp(from.data() + sizeof(scalars), arrays[0].p, arrays[0].n) == 0 &&
        (arrays[1].n == 0 || std::memcmp(from.data() + sizeof(scalars) + arrays[0].n, arrays[1].p, arrays[1].n) == 0)) {
      it->second.used = true;
      *out = &it->second;
      return IBERT_OK;
    }
  }
  OperatorConsts c;
  if (int rc = derive(&c)) return rc;
  if (ctx->consts_seen.size() >= 4096) ctx->consts_seen.clear();
  if (ctx->consts_seen.insert(sample).second) {
    *once = std::move(c);
    *out = once;
    return IBERT_OK;
  }
  ctx->consts_seen.erase(sample);
  c.from.resize(total);
  std::memcpy(c.from.data(), scalars, sizeof(scalars));
  std::memcpy(c.from.data() + sizeof(scalars), arrays[0].p, arrays[0].n);
  if (arrays[1].n) std::memcpy(c.from.data() + sizeof(scalars) + arrays[0].n, arrays[1].p, arrays[1].n);
  *out = &(ctx->consts[key] = std::move(c));
  ctx->consts_bytes += total;
  return IBERT_OK;
}

}  // namespace

// Above 1024 entries or 16 MB, those that no call has found again since the last time go; all of them if that is not enough.
void trim_consts(ibert_ctx* ctx) {
  const auto above = [&] { return ctx->consts.size() > 1024 || ctx->consts_bytes > (size_t(16) << 20); };
  if (!above()) return;
  for (auto it = ctx->consts.begin(); it != ctx->consts.end();) {
    if (it->second.used) {
      it->second.used = false;
      ++it;
    } else {
      ctx->consts_bytes -= it->second.from.size();
      it = ctx->consts.erase(it);
    }
  }
  if (above()) drop_consts(ctx);
}
void drop_consts(ibert_ctx* ctx) {
  ctx->consts.clear();
  ctx->consts_bytes = 0;
}

int linear_consts(ibert_ctx* ctx, double S_x, const double* S_w, int N, double S_out, bool upper_ok, GemmEpilogue* epi) {
  OperatorConsts* k = nullptr;
  const double scalars[5] = {S_x, S_out, (double)N, upper_ok ? 1.0 : 0.0, 1.0};
  const Bytes arrays[2] = {{S_w, sizeof(double) * (size_t)N}, {nullptr, 0}};
  int rc = operator_consts(ctx, 1, scalars, arrays, &ctx->consts_once[0], &k, [&](OperatorConsts* o) -> int {
    std::vector<int32_t> b, c, upper;
    bool fits = false;
    if (int r = make_linear_tables(S_x, S_w, N, nullptr, S_out, &b, &c, &upper, &fits)) return r;
    o->fast = upper_ok && fits;
    if (o->fast) b.swap(upper);
    if (int r = cached_upload(ctx, b.data(), b.size() * sizeof(int32_t), 21, &o->d_b)) return r;
    o->d_c = o->d_b;                                    // (the upper-word form has no separate shifts)
    return o->fast ? IBERT_OK : cached_upload(ctx, c.data(), c.size() * sizeof(int32_t), 22, &o->d_c);
  });
  if (rc) return rc;
  epi->fast = k->fast ? 1 : 0;
  epi->d_b = static_cast<const int32_t*>(k->d_b);
  epi->d_c = static_cast<const int32_t*>(k->d_c);
  return IBERT_OK;
}

int derive_ln(double S_r, double S, const double* gamma, const double* beta, int C, double S_out, LnConsts* k,
              std::vector<int32_t>* b_i, std::vector<int64_t>* B_i) {
  k->C = C;
  k->has_res = S_r != 0.0;
  if (k->has_res)
    if (int rc = make_ln_residual(S_r, S, k)) return rc;
  return make_ln_tables(gamma, beta, C, S_out, k, b_i, B_i);
}
int ln_consts(ibert_ctx* ctx, double S_r, double S, const double* gamma, const double* beta, int C, double S_out,
              OperatorConsts** out) {
  const double scalars[5] = {S_r, S, S_out, (double)C, 2.0};
  const Bytes arrays[2] = {{gamma, sizeof(double) * (size_t)C}, {beta, sizeof(double) * (size_t)C}};
  return operator_consts(ctx, 2, scalars, arrays, &ctx->consts_once[1], out, [&](OperatorConsts* o) -> int {
    std::vector<int32_t> b_i;
    std::vector<int64_t> B_i;
    if (int r = derive_ln(S_r, S, gamma, beta, C, S_out, &o->ln, &b_i, &B_i)) return r;
    if (int r = cached_upload(ctx, b_i.data(), b_i.size() * sizeof(int32_t), 11, &o->d_b)) return r;
    return cached_upload(ctx, B_i.data(), B_i.size() * sizeof(int64_t), 12, &o->d_c);
  });
}
void ln_consts_high(OperatorConsts* k) {
  if (!k->high_known && k->ln.has_res) make_ln_residual_high(&k->ln);
  k->high_known = true;
}

}  // namespace ibert
