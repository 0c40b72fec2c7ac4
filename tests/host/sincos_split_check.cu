// Host-side check of the acceptance's sine and cosine (mcp_device.cuh,
// split_terms and the combination with the table) against extended precision.
// Bounds, from the operations: sin r misses r^5/120 (2.4e-19) and rounds r^3/6
// four times in FP32 (2^-22 of 2.0e-11) and once in FP64 (2^-53 of 2^-11): 5e-18.
// cos r - 1 misses r^6/720 (2e-23) and rounds r^2's remainder (2^-24 of 2^-46)
// and r^4/24 (2^-22 of 2.4e-15), and the sum once in FP64 (2^-53 of 2^-23): 6e-21.
// With the table's rounding (2^-54), the inner sum's (2^-53: it may pass 1) and
// the outer's (2^-54) the result is within 2^-52 and 6e-18.
#include <cmath>
#include <cstdio>
#include "../../paper_2604_13323_gb300/csrc/mcp_device.cuh"
using namespace mcp;
int main() {
  static_assert(sizeof(long double) > sizeof(double), "no extended precision here");
  static double2 tab[2 * SPLIT_TAB_HALF + 1];
  for (int m = -SPLIT_TAB_HALF; m <= SPLIT_TAB_HALF; ++m) {
    const long double h = static_cast<long double>(m) / 1024.0L;
    tab[m + SPLIT_TAB_HALF] = make_double2(static_cast<double>(sinl(h)), static_cast<double>(cosl(h)));
  }
  long double e_sr = 0, e_cm = 0, e_s = 0, e_c = 0;
  const auto check = [&](float x) {
    const float mf = rintf(x * SPLIT_TAB_PER_RAD);
    const float r = fmaf(-mf, 1.f / SPLIT_TAB_PER_RAD, x);
    double sr, cm;
    split_terms(r, sr, cm);
    const long double half = sinl(0.5L * r);
    e_sr = std::max(e_sr, std::fabs(sr - sinl(static_cast<long double>(r))));
    e_cm = std::max(e_cm, std::fabs(cm + 2.0L * half * half));  // cos r - 1 without cancellation
    const double2 t = tab[static_cast<int>(mf) + SPLIT_TAB_HALF];
    const double s = std::fma(t.x, cm, std::fma(t.y, sr, t.x)), c = std::fma(t.y, cm, std::fma(-t.x, sr, t.y));
    e_s = std::max(e_s, std::fabs(s - sinl(static_cast<long double>(x))));
    e_c = std::max(e_c, std::fabs(c - cosl(static_cast<long double>(x))));
  };
  unsigned long long v = 0x2545F4914F6CDD1Dull;
  for (int i = 0; i < 2000000; ++i) {
    v ^= v << 13;
    v ^= v >> 7;
    v ^= v << 17;
    check(static_cast<float>((static_cast<double>(v >> 11) / 9007199254740992.0 - 0.5) * 8.0));
  }
  for (int m = -4095; m < 4096; ++m) {  // the largest remainders, exact table angles and their neighbours
    const float h = static_cast<float>(m) / 1024.f;
    for (float x : {h, h + 1.f / 2048.f, std::nextafterf(h, 9.f), std::nextafterf(h + 1.f / 2048.f, 9.f)}) check(x);
  }
  for (float x : {0.f, 1e-30f, -1e-20f, 1e-8f, 4.f, -4.f}) check(x);
  printf("sin r %.3Lg, cos r - 1 %.3Lg, sin x %.3Lg, cos x %.3Lg\n", e_sr, e_cm, e_s, e_c);
  const long double top = 0x1p-52L + 6e-18L;
  return e_sr <= 5e-18L && e_cm <= 6e-21L && e_s <= top && e_c <= top ? 0 : 1;
}
