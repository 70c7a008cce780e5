// Host check of fx_scale's range (csrc/hw_fixed.h): for the factors of spacings from 1e-17 to 1e27 and every unit and integer
// the sweeps may form, the scaled conversion stays in the normal range and within one unit in the last place of the product
// in long double. Prints the number of refused factors, of wrong values, and of factors beyond the range that are accepted.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "hw_fixed.h"

using namespace hw;

int main(int argc, char** argv) {
  std::mt19937_64 g(atoi(argv[1]));
  long refused = 0, wrong = 0, accepted = 0;
  for (int k = 0; k < 200000; ++k) {
    const double dx = k == 0 ? 1e-17 : k == 1 ? 1e27 : pow(10.0, -17.0 + 44.0 * (double)(g() >> 11) / 9007199254740992.0);
    const double c = k % 2 ? 1.0 / (24.0 * dx) : 9.812 / (2.0 * dx);
    bool bad = false;
    const FxScale s = fx_scale(c, bad);
    refused += bad;
    int64_t x = k % 5 == 0 ? INT64_MAX : (int64_t)(g() >> (1 + g() % 63)) | 1;
    if (g() & 1) x = -x;
    const int u = k % 7 == 0 ? 900 : k % 7 == 1 ? -900 : (int)(g() % 1801) - 900;
    const double r = fx_to_double_scaled(x, u, s);
    const long double want = ldexpl((long double)x * (long double)c, u);
    if (!std::isnormal(r) || !(fabsl(((long double)r - want) / want) <= 0x1p-52L)) ++wrong;
  }
  const double out[] = {0x1p60, 0x1p-97, 0.0, INFINITY, NAN, -1.0};
  for (double c : out) {
    bool bad = false;
    fx_scale(c, bad);
    accepted += !bad;
  }
  printf("%ld %ld %ld\n", refused, wrong, accepted);
}
