// Host check of fx_to_double_scaled and fx_quarter (csrc/hw_fixed.h) against __int128 and IEEE arithmetic. Prints the
// largest error of the scaled conversion in units in the last place (as the bound's excess over 1/2), the number of
// wrong special values, and the number of wrong quarters.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "hw_fixed.h"

using namespace hw;

int main(int argc, char** argv) {
  const int n = atoi(argv[1]);
  std::mt19937_64 g(atoi(argv[2]));
  double worst = 0;
  long wrong = 0, quarters = 0;
  for (int k = 0; k < n; ++k) {
    // magnitudes of every length, the ends of the range, round-to-even neighbourhoods
    int64_t x = (int64_t)(g() >> (1 + g() % 63));
    if (k % 8 == 0) x = (int64_t)((1ull << (g() % 63)) - (g() & 1));
    if (k % 16 == 1) x = INT64_MAX - (int64_t)(g() % 3);
    if (g() & 1) x = -x;
    uint64_t b = ((g() % 80 + 984) << 52) | (g() >> 12);
    if (k % 4 == 0) b &= ~0xfffffffffffffull;
    if (k % 4 == 1) b |= 0xfffffffffffffull;
    double c;
    memcpy(&c, &b, 8);
    bool bad = false;
    const FxScale s = fx_scale(c, bad);
    const int u = (int)(g() % 1800) - 900;
    const double r = fx_to_double_scaled(x, u, s);
    if (bad || (x == 0 && r != 0.0) || std::signbit(r) != (x < 0)) { ++wrong; continue; }
    if (x == 0) continue;
    // exact product x m with m the constant's 53-bit integer, against the result's mantissa at the same scale
    const uint64_t mc = (b & 0xfffffffffffffull) | (1ull << 52), ax = x < 0 ? 0ull - (uint64_t)x : (uint64_t)x;
    const unsigned __int128 p = (unsigned __int128)ax * mc;  // value = p 2^(u + ec - 1075)
    int er;
    const double fr = frexp(fabs(r), &er);  // fr in [1/2, 1): integer fr 2^53 at 2^(er - 53)
    const uint64_t mr = (uint64_t)ldexp(fr, 53);
    const int sh = (er - 53) - (u + (int)(b >> 52) - 1075);  // mr 2^sh against p
    long double err;
    if (sh >= 0) {
      const unsigned __int128 q = (unsigned __int128)mr << sh, d = p > q ? p - q : q - p;
      err = (long double)d / ldexpl(1.0L, sh);
    } else {
      err = fabsl((long double)p * ldexpl(1.0L, -sh) - (long double)mr);
    }
    if ((double)err > worst) worst = (double)err;
  }
  for (int k = 0; k < n; ++k) {
    uint64_t b = g();
    if (k % 2 == 0) b = (b & 0x800fffffffffffffull) | ((g() % 5) << 52);  // subnormal and the smallest normal
    if (k % 64 == 1) b = (b & (1ull << 63)) | (k % 128 == 1 ? 0 : 0x7ffull << 52);
    if (k % 64 == 3) b = (b & (1ull << 63)) | (g() % 9);
    double x;
    memcpy(&x, &b, 8);
    const double q = fx_quarter(x), want = x * 0.25;
    if (!(q == want || (std::isnan(q) && std::isnan(want))) || std::signbit(q) != std::signbit(want)) ++quarters;
  }
  bool none = false, low = false, high = false, neg = false;
  fx_scale(1.0, none);
  fx_scale(1e-30, low);
  fx_scale(1e30, high);
  fx_scale(-1.0, neg);
  wrong += none + !low + !high + !neg;
  printf("%.6f %ld %ld\n", worst, wrong, quarters);
}
