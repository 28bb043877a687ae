// Host program around the constants of operator calls: linked with operator_consts.cpp and host_consts.cpp, it
// stands in for the device side (cached_upload keeps host copies) and runs one check, named by its argument.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>

#include "ibert_internal.h"

using namespace ibert;

static int uploads = 0;
static std::vector<std::unique_ptr<std::vector<unsigned char>>> device;

int ibert::cached_upload(ibert_ctx*, const void* host, size_t bytes, uint64_t, void** dev) {
  ++uploads;
  const unsigned char* p = static_cast<const unsigned char*>(host);
  device.push_back(std::make_unique<std::vector<unsigned char>>(p, p + bytes));
  *dev = device.back()->data();
  return IBERT_OK;
}

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

constexpr int C = 768;
static std::vector<double> gamma_(C), beta_(C);

static OperatorConsts* ln(ibert_ctx& ctx, double S_r, double S_out) {
  OperatorConsts* k = nullptr;
  return ln_consts(&ctx, S_r, 1e-4, gamma_.data(), beta_.data(), C, S_out, &k) == IBERT_OK ? k : nullptr;
}

// the one-multiply form of the residual is searched only for the kernel that reads it
static int residual_search() {
  ibert_ctx ctx;
  LnConsts want{};
  CHECK(make_ln_residual(0.02, 1e-4, &want) == IBERT_OK);
  make_ln_residual_high(&want);
  CHECK(want.res_high == 1);
  for (int call = 0; call < 3; ++call) {
    OperatorConsts* k = ln(ctx, 0.02, 0.04);
    CHECK(k && k->ln.has_res && k->ln.res_narrow);
    CHECK(k->ln.res_high == 0 && k->ln.res_hm == 0);
  }
  OperatorConsts* k = ln(ctx, 0.02, 0.04);
  ln_consts_high(k);
  CHECK(k->ln.res_high == 1 && k->ln.res_hm == want.res_hm && k->ln.res_hk == want.res_hk);
  OperatorConsts* none = ln(ctx, 0.0, 0.04);
  ln_consts_high(none);
  CHECK(none->ln.res_high == 0 && !none->ln.has_res);
  return 0;
}

// constants that never return leave nothing behind and push nothing out
static int one_off() {
  ibert_ctx ctx;
  for (int call = 0; call < 2; ++call) CHECK(ln(ctx, 0.02, 0.04));
  CHECK(ctx.consts.size() == 1);
  for (int i = 0; i < 10000; ++i) {
    trim_consts(&ctx);
    CHECK(ln(ctx, 0.02 * (1.0 + 1e-6 * (i + 1)), 0.04));
    device.clear();
  }
  CHECK(ctx.consts.size() == 1 && ctx.consts_seen.size() <= 4096);
  const int before = uploads;
  CHECK(ln(ctx, 0.02, 0.04));
  CHECK(uploads == before);
  return 0;
}

// what is in use stays when others pass through in numbers, and the copies of the arrays are bounded
static int in_use() {
  ibert_ctx ctx;
  std::vector<double> S_w(100000, 1e-3);
  GemmEpilogue e{};
  for (int call = 0; call < 2; ++call) CHECK(ln(ctx, 0.02, 0.04));
  for (int i = 0; i < 3000; ++i) {
    for (int call = 0; call < 2; ++call) {
      trim_consts(&ctx);
      const int before = uploads;
      CHECK(ln(ctx, 0.02, 0.04));
      CHECK(uploads == before);
      trim_consts(&ctx);
      if (i % 10 == 0) CHECK(linear_consts(&ctx, 0.03, S_w.data(), (int)S_w.size(), 0.05 * (1.0 + 1e-5 * i), true, &e) == IBERT_OK);
      else CHECK(ln(ctx, 0.02, 0.05 * (1.0 + 1e-5 * i)));
      device.clear();
    }
    CHECK(ctx.consts.size() <= 1025);
    size_t bytes = 0;
    for (auto& kv : ctx.consts) bytes += kv.second.from.size();
    CHECK(bytes == ctx.consts_bytes && bytes <= (size_t(16) << 20) + 8 * S_w.size() + 64);
  }
  return 0;
}

// one array element outside the sample, and the form of the rest of the epilogue, make other constants
static int linear_keys() {
  ibert_ctx ctx;
  std::vector<double> S_w(3072, 1e-3), other = S_w;
  other[1] = 1.5e-3;
  for (int call = 0; call < 4; ++call) {
    for (int form = 0; form < 4; ++form) {
      const std::vector<double>& s = form & 1 ? other : S_w;
      GemmEpilogue e{};
      CHECK(linear_consts(&ctx, 0.03, s.data(), 3072, 0.05, (form & 2) != 0, &e) == IBERT_OK);
      CHECK(e.fast == (form >> 1));
      int32_t b = 0, c = 0;
      for (int i : {0, 1, 2, 3071}) {
        CHECK(dyadic((0.03 * s[i]) / 0.05, &b, &c) == IBERT_OK);
        if (form & 2) CHECK(e.d_b[i] == (int32_t)((int64_t)b << (32 - c)));
        else CHECK(e.d_b[i] == b && e.d_c[i] == c);
      }
    }
  }
  CHECK(ctx.consts.size() == 4);
  return 0;
}

int main(int argc, char** argv) {
  for (int i = 0; i < C; ++i) { gamma_[i] = 1.0 + 0.1 * std::sin(i); beta_[i] = 0.1 * std::cos(3 * i); }
  if (argc < 2) return 2;
  if (!std::strcmp(argv[1], "residual_search")) return residual_search();
  if (!std::strcmp(argv[1], "one_off")) return one_off();
  if (!std::strcmp(argv[1], "in_use")) return in_use();
  if (!std::strcmp(argv[1], "linear_keys")) return linear_keys();
  return 2;
}
