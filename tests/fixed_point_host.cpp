// Line contractions of fxp.h on the host against long double, and the plain FP64 dot product's error
// on the same lines.  Prints one line per (N, spread): spread is the binary range of the line's
// magnitudes.  Columns: the fixed-point error over (2^-55 max|v| rowsum + 2^-53 |exact|), its bound;
// the 2-norm error of the fixed-point and of the FP64 results over all lines.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "fxp.h"

using namespace se;

static std::mt19937_64 rng(7);
static double uniform() { return 2.0 * ((rng() >> 11) * 0x1p-53) - 1.0; }

template <int N, int SYM>
static void lines(int spread, int shift) {
  double worst = 0.0;
  long double e_fx = 0, e_64 = 0, nrm = 0;
  for (int rep = 0; rep < 400; ++rep) {
    double M[N * N], v[N];
    for (int r = 0; r < N; ++r)
      for (int c = 0; c < N; ++c) {
        const double a = uniform() * std::exp2(4.0 * uniform());
        M[r * N + c] = a;
        M[(N - 1 - r) * N + (N - 1 - c)] = SYM * a;
      }
    if (SYM < 0 && N % 2) M[(N / 2) * N + N / 2] = 0.0;
    double vmax = 0.0, rows = 0.0;
    for (int c = 0; c < N; ++c) {
      v[c] = std::ldexp(uniform(), shift - (int)(rng() % (spread + 1)));
      vmax = std::fmax(vmax, std::fabs(v[c]));
    }
    const auto t = fx_fold_tables<N, N>(M, SYM, 60);
    unsigned mag = 0;
    for (int c = 0; c < N; ++c) mag = fx_mag(v[c]) > mag ? fx_mag(v[c]) : mag;
    if (fx_bad(mag)) std::exit(3);
    const int E = fx_exponent(mag);
    int h[N], l[N];
    for (int c = 0; c < N; ++c) fx_split(v[c], E, h[c], l[c]);
    double out[N];
    fx_contract<N, N, SYM>(t, h, l, [&](int k, long long R) {
      if (R > (1ll << 62) || R < -(1ll << 62)) std::exit(4);
      out[k] = fx_double(R, E - t.k);
    });
    for (int r = 0; r < N; ++r) {
      double s = 0.0;
      for (int c = 0; c < N; ++c) s += std::fabs(M[r * N + c]);
      rows = std::fmax(rows, s);
    }
    for (int r = 0; r < N; ++r) {
      long double ex = 0;
      double d = 0.0;
      for (int c = 0; c < N; ++c) {
        ex += (long double)M[r * N + c] * v[c];
        d = std::fma(M[r * N + c], v[c], d);
      }
      const long double bound = 0x1p-55L * vmax * rows + 0x1p-53L * std::fabs(ex);
      if (bound > 0) worst = std::fmax(worst, (double)(std::fabs((long double)out[r] - ex) / bound));
      const long double sc = std::ldexp(1.0L, -shift);
      e_fx += ((long double)out[r] - ex) * sc * ((long double)out[r] - ex) * sc;
      e_64 += ((long double)d - ex) * sc * ((long double)d - ex) * sc;
      nrm += ex * sc * ex * sc;
    }
  }
  std::printf("%d %d %d %d %.4f %.4e %.4e\n", N, SYM, spread, shift, worst, (double)std::sqrt(e_fx / nrm),
              (double)std::sqrt(e_64 / nrm));
}

template <int N>
static void all() {
  for (int spread : {0, 6, 40, 400})
    for (int shift : {0, -900, 900}) {
      if (shift == -900 && spread == 400) continue;
      lines<N, -1>(spread, shift);
      lines<N, 1>(spread, shift);
    }
}

int main() {
  // round trip: a value of the line's largest exponent is exact through fx_split and fx_double
  for (int q = 0; q < 20000; ++q) {
    const double v = std::ldexp(uniform(), (int)(rng() % 1800) - 900);
    if (v == 0.0) continue;
    const int E = fx_exponent(fx_mag(v));
    int h, l;
    fx_split(v, E, h, l);
    const long long x = ((long long)h << FX_LIMB) + l;
    if (fx_double(x, E - 56) != v || fx_double(x * 16, E - 60) != v) return 1;
    // against the largest value of a line 2^k above it: the bits above 2^-56 of that value
    const int k = (int)(rng() % 70);
    fx_split(v, E + k, h, l);
    const long double unit = std::ldexp(1.0L, E + k - 1023 - 56);
    const long double got = (((long long)h << FX_LIMB) + l) * unit;
    if (!(std::fabs(got - (long double)v) < unit && std::fabs(got) <= std::fabs((long double)v))) return 2;
  }
  int h, l;
  for (double z : {0.0, -0.0, 5e-324, -1e-310}) {
    fx_split(z, FX_EMIN, h, l);
    if (((long long)h << FX_LIMB) + l != 0) return 5;
  }
  for (double b : {(double)INFINITY, (double)NAN, 1.7e308, 1e-300, 1e-310})
    if (!fx_bad(fx_mag(b))) return 6;
  if (fx_bad(0u) || fx_bad(fx_mag(1e-280)) || fx_bad(fx_mag(1e290))) return 7;
  // conversion of any 62-bit integer: to nearest, at most two units lost
  for (int q = 0; q < 200000; ++q) {
    const long long R = (long long)(rng() >> 2 >> (rng() % 62)) * ((rng() & 1) ? 1 : -1);
    const double d = fx_double(R, 1023);
    if (std::fabs((long double)d - (long double)R) > 2.0L + 0x1p-53L * std::fabs((long double)R)) return 8;
  }
  all<2>(), all<3>(), all<4>(), all<5>(), all<6>(), all<7>(), all<8>(), all<9>(), all<10>(), all<11>();
  return 0;
}
