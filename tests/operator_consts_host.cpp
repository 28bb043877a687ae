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

int main(int argc, char** argv) {
  for (int i = 0; i < C; ++i) { gamma_[i] = 1.0 + 0.1 * std::sin(i); beta_[i] = 0.1 * std::cos(3 * i); }
  if (argc < 2) return 2;
  if (!std::strcmp(argv[1], "residual_search")) return residual_search();
  return 2;
}
