// Lines whose values are zeros of either sign, or are shifted out by their scale, through fx_split and
// fx_contract: both limbs and every result exactly 0.  Exit code: the check that failed.
#include <cmath>
#include <random>

#include "fxp.h"

using namespace se;

static std::mt19937_64 rng(11);

template <int NR, int NC, int SYM>
static bool zeros_stay() {
  for (int rep = 0; rep < 500; ++rep) {
    double M[NR * NC];
    for (int r = 0; r < NR; ++r)
      for (int c = 0; c < NC; ++c) {
        const double a = 2.0 * ((rng() >> 11) * 0x1p-53) - 1.0;
        M[r * NC + c] = a;
        M[(NR - 1 - r) * NC + (NC - 1 - c)] = SYM * a;
      }
    const auto t = fx_fold_tables<NR, NC>(M, SYM, 60);
    int h[NC], l[NC];
    const int E = rep % 2 ? FX_EMIN : 900;
    for (int c = 0; c < NC; ++c) {
      // a zero, a subnormal, or a value more than 2^57 below the scale, of a random sign
      double v = rep % 3 == 0 ? 0.0 : (rep % 3 == 1 ? 4e-310 : std::ldexp(1.9, E - 1023 - 58));
      if (rng() & 1) v = -v;
      fx_split(v, E, h[c], l[c]);
      if (h[c] != 0 || l[c] != 0) return false;
    }
    bool ok = true;
    fx_contract<NR, NC, SYM>(t, h, l, [&](int, long long R) { ok = ok && R == 0; });
    if (!ok) return false;
  }
  return true;
}

int main() {
  // limbs of a value and of its opposite are opposite
  for (int q = 0; q < 20000; ++q) {
    const double v = std::ldexp(2.0 * ((rng() >> 11) * 0x1p-53) - 1.0, (int)(rng() % 60));
    int h, l, hm, lm;
    fx_split(v, 1023 + 61, h, l);
    fx_split(-v, 1023 + 61, hm, lm);
    if (h != -hm || l != -lm) return 1;
  }
  if (!zeros_stay<8, 8, -1>() || !zeros_stay<9, 9, -1>() || !zeros_stay<2, 2, -1>()) return 2;
  if (!zeros_stay<8, 6, 1>() || !zeros_stay<5, 3, 1>() || !zeros_stay<3, 8, 1>() || !zeros_stay<4, 2, 1>()) return 3;
  return 0;
}
