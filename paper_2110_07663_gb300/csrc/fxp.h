// FP64-accurate line contractions on the integer pipe (block floating point).
//
// GB300 executes 2 FP64 FMAs per clock and SM, but about 36 32 x 32 + 64 bit integer multiply-adds
// (IMAD.WIDE, measured with independent chains: 36 lanes/clk/SM against 1.6-2 of DFMA).  A
// contraction out_i = sum_l M_il v_l whose inputs share one binary scale is therefore cheaper in
// fixed point: three integer multiply-adds per term instead of one DFMA, 6 times the rate.
//
//   value      x = v 2^(56 - e), |x| < 2^57, e the (unbiased) exponent of the largest |v| of the
//              line or element: kept as x = h 2^28 + l, |l| < 2^28, h and l of the sign of v
//              (fx_split; bits below 2^-56 of the largest value are dropped, and what is
//              dropped whole contracts to exactly 0)
//   matrix     M' = M 2^k rounded to an integer, |M'| < 2^59, kept as mh 2^28 + ml with
//              -2^27 <= ml < 2^27 (fx_limbs), its row sums bounded so that the sums below fit;
//              k is the matrix's, or each row's own (fx_fold_rows)
//   product    hi = sum mh h, mid = sum (mh l + ml h), 64-bit sums that cannot overflow
//              (|hi|, |mid| < 2^63); the ml l terms (below 2^-59 of the largest
//              possible sum, and without a bias because ml has both signs) are left out.
//              R = hi + round(mid / 2^28) is the result in units of 2^(e - k)
//   back       the double nearest to R 2^(e - k) (fx_double): one rounding to 53 bits
//
// Before the final rounding every error is below 2^-55 of (largest value on the scale) x (largest row
// sum of M); an FP64 dot product rounds each of its terms to 2^-53 of the running sum.  Exponents outside
// [FX_EMIN, FX_EMAX] (infinities, NaN, values whose results could leave the normal range) are not
// representable: kernels test for them and compute such lines, or elements, in FP64.
//
// The arithmetic also compiles as host code, so that its accuracy can be checked without a GPU.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define SE_FX __host__ __device__ __forceinline__
#else
#define SE_FX inline
#endif

namespace se {

constexpr int FX_LIMB = 28;
constexpr long long FX_HALF = 1ll << (FX_LIMB - 1);  // where a middle sum starts: its cut rounds
constexpr int FX_EMIN = 70, FX_EMAX = 2020;  // biased exponents of the largest value

// Folded tables of a centro-(anti)symmetric N x N matrix M, M[N-1-k][N-1-l] = sym * M[k][l]:
// with e_l = v_l + v_{N-1-l}, o_l = v_l - v_{N-1-l} (l < N/2; for odd N also e_m = v_m, m = N/2)
//   2 (M v)_k       =  E_k + O_k         E_k = sum_l (M_kl + M_k,N-1-l) e_l   (middle: 2 M_km e_m)
//   2 (M v)_{N-1-k} = sym (E_k - O_k)    O_k = sum_l (M_kl - M_k,N-1-l) o_l
// The tables hold 2^k (M_kl +- M_k,N-1-l) as limbs; `k` includes the factor 2.  A kernel takes
// them as a parameter, so that every multiplier is a constant-bank operand.
template <int NR, int NC>
struct FxFold {
  static constexpr int RE = (NR + 1) / 2;  // rows computed (the others follow by symmetry)
  static constexpr int CE = (NC + 1) / 2, CO = NC / 2;
  int eh[RE * CE], el[RE * CE];
  int oh[RE * (CO > 0 ? CO : 1)], ol[RE * (CO > 0 ? CO : 1)];
  int k;
};

// ------------------------------------------------------------------ word operations
SE_FX void fx_words(double v, unsigned& hi, unsigned& lo) {
#ifdef __CUDA_ARCH__
  hi = (unsigned)__double2hiint(v);
  lo = (unsigned)__double2loint(v);
#else
  unsigned long long b;
  std::memcpy(&b, &v, 8);
  hi = (unsigned)(b >> 32);
  lo = (unsigned)b;
#endif
}
SE_FX double fx_from_words(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const unsigned long long b = ((unsigned long long)hi << 32) | lo;
  double v;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
// High word of (hi, lo) << n and low word of (hi, lo) >> n, n modulo 32.
SE_FX unsigned fx_funnel_l(unsigned lo, unsigned hi, int n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, n);
#else
  return (unsigned)(((((unsigned long long)hi << 32) | lo) << (n & 31)) >> 32);
#endif
}
SE_FX unsigned fx_funnel_r(unsigned lo, unsigned hi, int n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, n);
#else
  return (unsigned)((((unsigned long long)hi << 32) | lo) >> (n & 31));
#endif
}
// x >> n; 0 (or the sign) for n >= 64.
SE_FX unsigned long long fx_shr(unsigned long long x, int n) {
#ifdef __CUDA_ARCH__
  asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(n));
  return x;
#else
  return n > 63 ? 0ull : x >> n;
#endif
}
SE_FX long long fx_shr(long long x, int n) {
#ifdef __CUDA_ARCH__
  asm("shr.s64 %0, %0, %1;" : "+l"(x) : "r"(n));
  return x;
#else
  return x >> (n > 63 ? 63 : n);
#endif
}
// Position of the leading bit, -1 for 0.
SE_FX int fx_bfind(unsigned x) {
#ifdef __CUDA_ARCH__
  int p;
  asm("bfind.u32 %0, %1;" : "=r"(p) : "r"(x));
  return p;
#else
  return x ? 31 - __builtin_clz(x) : -1;
#endif
}

// ------------------------------------------------------------------ tables
// Limbs of an integer |m| < 2^59 - 2^27.
SE_FX void fx_limbs(long long m, int& mh, int& ml) {
  const long long h = (m + (1ll << (FX_LIMB - 1))) >> FX_LIMB;
  mh = (int)h;
  ml = (int)(m - (h << FX_LIMB));
}

// Row r (and its mirror image) of the folded tables of M: M times f, halves averaged.
template <int NR, int NC>
inline void fx_fold_row(FxFold<NR, NC>& t, const double* M, int sym, int r, double f) {
  auto fix = [&](int c) {
    const double m = M[r * NC + c] * f * 0.5, w = sym * M[(NR - 1 - r) * NC + (NC - 1 - c)] * f * 0.5;
    return (long long)(m < 0 ? m - 0.5 : m + 0.5) + (long long)(w < 0 ? w - 0.5 : w + 0.5);
  };
  for (int c = 0; c < t.CE; ++c) fx_limbs(fix(c) + fix(NC - 1 - c), t.eh[r * t.CE + c], t.el[r * t.CE + c]);
  for (int c = 0; c < t.CO; ++c) fx_limbs(fix(c) - fix(NC - 1 - c), t.oh[r * t.CO + c], t.ol[r * t.CO + c]);
}

// Largest k, f = 2^k, with `rows` f below 2^rows_log2 and folded entries (at most twice `most` f,
// and the tables hold twice the average) below 2^59; at most FX_EMIN - 2, so that
// FX_EMIN - (k + 1) is an exponent fx_double takes.
inline int fx_fold_scale(double rows, double most, int rows_log2, double* f) {
  double lim = 1.0;
  for (int q = 0; q < rows_log2; ++q) lim *= 2.0;
  auto fits = [&](double g) { return rows * g < lim && 2.0 * most * g < 0x1p59 - 0x1p27; };
  int k = 0;
  *f = 1.0;
  while (!fits(*f)) *f *= 0.5, --k;
  while (k < FX_EMIN - 2 && fits(2.0 * *f)) *f *= 2.0, ++k;
  return k;
}

// Largest row sum and entry of rows r0 .. r1 - 1 of M.
template <int NC>
inline void fx_row_sizes(const double* M, int r0, int r1, double* rows, double* most) {
  for (int r = r0; r < r1; ++r) {
    double s = 0.0;
    for (int c = 0; c < NC; ++c) {
      const double m = M[r * NC + c] < 0 ? -M[r * NC + c] : M[r * NC + c];
      s += m;
      *most = m > *most ? m : *most;
    }
    *rows = s > *rows ? s : *rows;
  }
}

// Folded fixed-point tables of M (row-major NR x NC, M[NR-1-r][NC-1-c] = sym M[r][c] up to rounding:
// both entries are averaged), host.  rows_log2: the largest row sum of |M'| stays below 2^rows_log2,
// at most 60; entries stay below 2^59.  |R| < 2^(rows_log2 + 2) for |x| < 2^57.
template <int NR, int NC>
inline FxFold<NR, NC> fx_fold_tables(const double* M, int sym, int rows_log2) {
  FxFold<NR, NC> t{};
  double rows = 0.0, most = 0.0, f;
  fx_row_sizes<NC>(M, 0, NR, &rows, &most);
  t.k = fx_fold_scale(rows, most, rows_log2, &f) + 1;
  for (int r = 0; r < t.RE; ++r) fx_fold_row(t, M, sym, r, f);
  return t;
}

// The same with a scale per row.  The rows of a derivative matrix differ by up to 2^5 in size and the
// small ones lose those bits on a common scale (error of the operator at p = 10 on smooth fields, over that
// of FP64 dot products: 1.09 with one scale, 0.47 with a scale per row).
template <int NR, int NC>
struct FxFoldRows : FxFold<NR, NC> {
  int kr[FxFold<NR, NC>::RE];
  SE_FX int row_k(int r) const { return kr[r < FxFold<NR, NC>::RE ? r : NR - 1 - r]; }
};
template <int NR, int NC>
inline FxFoldRows<NR, NC> fx_fold_rows(const double* M, int sym) {
  FxFoldRows<NR, NC> t{};
  for (int r = 0; r < t.RE; ++r) {
    double rows = 0.0, most = 0.0, f;
    fx_row_sizes<NC>(M, r, r + 1, &rows, &most);
    fx_row_sizes<NC>(M, NR - 1 - r, NR - r, &rows, &most);
    t.kr[r] = fx_fold_scale(rows, most, 60, &f) + 1;
    fx_fold_row(t, M, sym, r, f);
  }
  return t;
}

// ------------------------------------------------------------------ values
// High word without the sign: orders doubles by magnitude.
SE_FX unsigned fx_mag(double v) {
  unsigned hi, lo;
  fx_words(v, hi, lo);
  return hi & 0x7fffffffu;
}

// Biased exponent of an element whose largest fx_mag is `mag`, and whether it can be represented
// (one of zeros is; so, by the high word alone, is one whose largest value is below 2^-1042: kernels look
// at the low words where the largest high word is 0).
SE_FX int fx_exponent(unsigned mag) {
  const int e = (int)(mag >> 20);
  return e > FX_EMIN ? e : FX_EMIN;
}
SE_FX bool fx_bad(unsigned mag) {
  return mag != 0u && (unsigned)((int)(mag >> 20) - FX_EMIN) > (unsigned)(FX_EMAX - FX_EMIN);
}

// v in units of 2^(E - 1023 - (XB - 1)), |x| < 2^XB, E >= every value's biased exponent.  XB = 57, or
// 58 where lines are not folded (a folded sum needs the bit).  NEAR: |l| <= 2^27 of either sign, which
// halves the low x low products that a contraction leaves out, for one more operation; a folded sum of
// two low limbs needs their sign to be the value's.
template <int XB = 57, bool NEAR = XB == 58>
SE_FX void fx_split(double v, int E, int& h, int& l) {
  unsigned hi, lo;
  fx_words(v, hi, lo);
  const int s = (int)hi >> 31;
  const int sh = E - (int)((hi >> 20) & 0x7ffu);
  // XB + 4 bit magnitude, led by the implicit one (a zero or subnormal is shifted out: sh >= 70)
  constexpr int UP = XB - 49;
  const unsigned one = 1u << (20 + UP);
  const unsigned top = (fx_funnel_l(lo, hi, UP) & (one - 1u)) | one;
  const unsigned long long x = fx_shr(((unsigned long long)top << 32) | (lo << UP), sh);
  // both limbs take the sign: a zero, or a value shifted out, has two zero limbs whatever its sign
  const unsigned xl = (unsigned)x;
  if constexpr (NEAR) {
    h = ((int)((unsigned)(x >> 32) + (xl >> 31)) ^ s) - s;
    l = (((int)xl >> 4) ^ s) - s;
  } else {
    h = ((int)(unsigned)(x >> 32) ^ s) - s;
    l = ((int)(xl >> 4) ^ s) - s;
  }
}

// The double nearest to R 2^(eb - 1023), |R| < 2^63; eb >= 1 and eb + 63 < 2046 (callers bound
// the exponents).  Normalisation by the position of the leading bit, rounding by adding half a
// unit before the cut (a carry moves into the exponent field).  Up to two units of R are dropped:
// one where R < 0 (|R| as the one's complement), one where |R| < 2^32.  No branches: the
// conversions of a line's results interleave.
SE_FX double fx_double(long long R, int eb) {
  const unsigned s = (unsigned)((int)(R >> 32) >> 31);
  const unsigned rh = (unsigned)((unsigned long long)R >> 32) ^ s, rl = (unsigned)R ^ s;
  const bool small = rh == 0u;
  unsigned h = small ? rl >> 1 : rh, l = small ? 0u : rl;
  const int p = small ? eb : eb + 31;
  const int pos = fx_bfind(h);
  const int n = 30 - pos;
  const unsigned mh0 = fx_funnel_l(l, h, n);
  l <<= n & 31;  // leading bit at bit 62 of (mh0, l)
  const unsigned long long m = (((unsigned long long)mh0 << 32) | l) + 0x200u;
  const unsigned mh = (unsigned)(m >> 32);
  const unsigned lo = fx_funnel_r((unsigned)m, mh, 10);
  const unsigned hi = (mh >> 10) + ((unsigned)(p + pos) << 20);
  return fx_from_words(h ? hi | (s & 0x80000000u) : 0u, h ? lo : 0u);
}

// ------------------------------------------------------------------ renormalisation of 64-bit results
// |R| by its high word (one less for negative R).
SE_FX unsigned fx_high(long long R) {
  const int h = (int)(R >> 32);
  return (unsigned)(h ^ (h >> 31));
}

// Left shift that brings values whose largest high word is `high` to 63 bits.
SE_FX int fx_norm(unsigned high) { return high ? 30 - fx_bfind(high) : 30; }

// Limbs of R after a left shift by n to 63 bits: x = R 2^n / 2^(63 - XB), |x| < 2^XB, |l| <= 2^27.
template <int XB = 57>
SE_FX void fx_renorm(long long R, int n, int& h, int& l) {
  const unsigned long long x = (unsigned long long)R << n;
  const int xh = (int)(x >> 32);
  constexpr int UP = 63 - XB + FX_LIMB - 32;  // bits of x's high word below h
  const unsigned w = fx_funnel_r((unsigned)x, (unsigned)xh, UP);  // l, and bits below it, at the top
  h = (xh >> UP) + (int)(w >> 31);
  l = (int)w >> (32 - FX_LIMB);
}

// Limbs of x 2^-(s + 1), s >= 0, rounded; |l| <= 2^27.
SE_FX void fx_shift_limbs(long long x, int s, int& h, int& l) {
  const long long y = (fx_shr(x, s) + 1) >> 1;
  const unsigned w = (unsigned)y << (32 - FX_LIMB);
  h = (int)(y >> FX_LIMB) + (int)(w >> 31);
  l = (int)w >> (32 - FX_LIMB);
}

#ifdef __CUDACC__
// Starts moving n doubles at p towards L2 (whole 16-byte units inside [p - 1, p + n)).
__device__ __forceinline__ void fx_prefetch(const double* p, int n) {
  const unsigned long long a = (unsigned long long)p & ~15ull;
  const unsigned bytes = (unsigned)(((unsigned long long)(p + n) - a) & ~15ull);
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(bytes) : "memory");
}
#endif

// R of the folded contraction of the line (h, l): out(k, R) for k < NR.  SYM = -1: M is
// centro-antisymmetric (derivatives), +1: centro-symmetric (interpolation).
template <int NR, int NC, int SYM, class Out>
SE_FX void fx_contract(const FxFold<NR, NC>& t, const int (&h)[NC], const int (&l)[NC],
                                            Out&& out) {
  constexpr int RE = FxFold<NR, NC>::RE, CE = FxFold<NR, NC>::CE, CO = FxFold<NR, NC>::CO;
  int eh[CE], el[CE], oh[CE], ol[CE];
#pragma unroll
  for (int c = 0; c < CO; ++c) {
    eh[c] = h[c] + h[NC - 1 - c];
    el[c] = l[c] + l[NC - 1 - c];
    oh[c] = h[c] - h[NC - 1 - c];
    ol[c] = l[c] - l[NC - 1 - c];
  }
  if constexpr (CE > CO) {
    eh[CO] = h[CO];
    el[CO] = l[CO];
  }
#pragma unroll
  for (int r = 0; r < RE; ++r) {
    const bool mid = NR % 2 == 1 && r == RE - 1;  // the middle row is its own mirror image
    long long hE = 0, mE = FX_HALF, hO = 0, mO = FX_HALF;
    if (!(mid && SYM < 0)) {
#pragma unroll
      for (int c = 0; c < CE; ++c) {
        hE += (long long)t.eh[r * CE + c] * eh[c];
        mE += (long long)t.eh[r * CE + c] * el[c];
        mE += (long long)t.el[r * CE + c] * eh[c];
      }
    }
    if (!(mid && SYM > 0)) {
#pragma unroll
      for (int c = 0; c < CO; ++c) {
        hO += (long long)t.oh[r * CO + c] * oh[c];
        mO += (long long)t.oh[r * CO + c] * ol[c];
        mO += (long long)t.ol[r * CO + c] * oh[c];
      }
    }
    if (mid) {
      out(r, SYM < 0 ? hO + (mO >> FX_LIMB) : hE + (mE >> FX_LIMB));
    } else {
      const long long E = hE + (mE >> FX_LIMB), O = hO + (mO >> FX_LIMB);
      out(r, E + O);
      out(NR - 1 - r, SYM < 0 ? O - E : E - O);
    }
  }
}

}  // namespace se
