// Limbs with a low limb of both signs (values of lines that are not folded): h 2^28 + l is the value's
// fixed-point form, |l| <= 2^27, at every shift; after a renormalisation and after a rounding shift too.
// Exit code: the check that failed.
#include <cmath>
#include <random>

#include "fxp.h"

using namespace se;

int main() {
  std::mt19937_64 rng(5);
  const int half = 1 << 27;
  for (int q = 0; q < 200000; ++q) {
    double v = std::ldexp(2.0 * ((rng() >> 11) * 0x1p-53) - 1.0, 0);
    if (q % 7 == 0) v = std::ldexp(q % 14 ? -1.0 : 1.0, -(int)(rng() % 60));
    const int E = 1023 + (int)(rng() % 8);
    int h, l, h0, l0;
    fx_split<58>(v, E, h, l);
    fx_split<58, false>(v, E, h0, l0);
    if (l < -half || l > half) return 1;
    if (((long long)h << 28) + l != ((long long)h0 << 28) + l0) return 2;
    fx_split<57, true>(v, E, h, l);
    fx_split<57, false>(v, E, h0, l0);
    if (l < -half || l > half || ((long long)h << 28) + l != ((long long)h0 << 28) + l0) return 3;
  }
  for (int q = 0; q < 200000; ++q) {
    long long R = (long long)(rng() >> 1);
    if (q % 5 == 0) R = (1ll << 62) | (q % 10 ? 0x3fffffffffffffffll : 0);
    R >>= rng() % 62;
    if (rng() & 1) R = -R;
    const int n = fx_norm(fx_high(R));
    const long long x = (long long)((unsigned long long)R << n);
    int h, l;
    fx_renorm<58>(R, n, h, l);
    if (l < -half || l > half || ((long long)h << 28) + l != x >> 5) return 4;
    fx_renorm<57>(R, n, h, l);
    if (l < -half || l > half || ((long long)h << 28) + l != x >> 6) return 5;
    const int s = 4 + (int)(rng() % 80);
    fx_shift_limbs(x, s, h, l);
    const long double want = std::floor(std::ldexp((long double)x, -(s + 1)) + 0.5L);
    if (l < -half || l > half || (long double)(((long long)h << 28) + l) != want) return 6;
  }
  return 0;
}
