// FP64 fast-diagonalisation solves in block floating point (fxp.h): the apply of fdm.cu,
// z = (S_z x S_y x S_x) D^-1 (S_z^T x S_y^T x S_x^T) R_e r, with its six line contractions on the
// integer pipe.  S and S^T of each direction are split once per block into limbs on the scale of
// the matrix's largest entry.
//
// The window of pbar^3 points lives in one shared array per element, updated in place line by line
// (each thread reads its whole line, contracts it, and writes over it).  Between two contractions
// the values are 64-bit integers on a scale common to the element; the largest magnitude of a
// phase, gathered while its results are produced, gives the shift by which the next phase's
// readers renormalise to 58 bits, so no phase loses headroom.  The z lines (forward, D^-1, and
// backward) belong to one thread: their intermediate values stay in registers, D^-1 is applied in
// FP64, and the lines meet again on a common scale after the backward z contraction.  Lines whose
// results become doubles (forward z, backward x) are read on their own scale: their leading bits cost
// two instructions per value and no shift back.  Results leave as doubles, 1/multiplicity taken from
// the exponent.
//
// Measured on GB300 (us per launch; in brackets the FP64 kernel this one replaced, at 91% of the FP64
// pipe): 24^3 elements p = 7 377 [1190], p = 5 158 [460], p = 3 59 [150]; 16^3 p = 9 236 [700].  The
// multiply-adds keep their pipe (32 lanes/clk/SM) 64% busy; a result's two sums in a row beat all results' sums
// input by input (more chains in flight, 500 instead of 406 at p = 7: the accumulator stays in the
// pipe), and 64 registers beat 80 and 96 (440).
//
// Error against extended precision (2-norm, host emulation, p = 2 to 10), over that of the FP64 solve with
// the same S: 0.31 to 0.43 for random and 0.33 to 0.44 for smooth residuals, 0.34 to 0.70 where the
// residual decays by eight decades across the window, 0.41 to 0.99 around one value 10^8 times the
// others.  FP64 keeps the products of S's small entries in full, this kernel on the scale of S's
// largest entry and of the window, so the error relative to each value by itself is up to 1.5 and 1.8
// times FP64's (geometric mean) in the last two.  58-bit values, low limbs with both signs, in S and in
// the values, and rounded middle sums matter: with 57 bits and unsigned limbs the dropped products had a
// bias and the error was 3 to 5 times FP64's; with unsigned limbs of the values it was up to 1.5
// times around a large value, and the masks cost 24 us at p = 7 (400).
//
// An element whose values cannot share a scale (infinities, NaN, magnitudes at the ends of the range) is
// solved in FP64 (fdm_slow_block); the others of its block keep their bits.
#include <climits>

#include "fdm_window.h"
#include "fxp.h"
#include "se_internal.h"

namespace se {

template <int PB>
struct FdmFxDims {
  static constexpr int RS = PB % 2 ? PB : PB + 1;          // odd row stride: lines do not conflict
  static constexpr int PS = RS * PB;
  static constexpr int VOL = (RS * PB * PB + 1) / 2 * 2;    // 16-byte multiple
  static constexpr int PBP = (PB + 1) / 2 * 2;              // padded matrix row (16-byte loads of two entries)
  static constexpr int SMAT = PB * PBP;                     // one matrix
  static constexpr int META = 36;                           // magnitudes, exponents, fallback, neighbours (ints)
  static constexpr size_t BYTES = (VOL + 6 * SMAT) * 8 + META * 4;
};

size_t fdm_fx_smem_per_element(int p) {
  switch (p) {
#define SE_FDMFX_SM(PP) \
  case PP: return FdmFxDims<PP + 3>::BYTES;
    SE_FDMFX_SM(1) SE_FDMFX_SM(2) SE_FDMFX_SM(3) SE_FDMFX_SM(4) SE_FDMFX_SM(5)
    SE_FDMFX_SM(6) SE_FDMFX_SM(7) SE_FDMFX_SM(8) SE_FDMFX_SM(9) SE_FDMFX_SM(10)
#undef SE_FDMFX_SM
    default: return 0;
  }
}

struct FdmFxArgs {
  int64_t E;
  int NE;
  const int* nbr;
  const double *in, *S, *dinv;
  const uint8_t* pflag;
  double* out;
};

// Largest value of a group of lanes of one element, collected in *dst (one atomic per group).
__device__ __forceinline__ void fx_group_max(unsigned peers, unsigned v, unsigned* dst) {
  v = __reduce_max_sync(peers, v);
  if ((threadIdx.x & 31) == (unsigned)(__ffs(peers) - 1)) atomicMax(dst, v);
}

// R of one row of limbs (16-byte aligned, two entries per load) against the line (h, l).
template <int PB>
__device__ __forceinline__ long long fx_dot_row(const int2* __restrict__ row, const int (&h)[PB], const int (&l)[PB]) {
  long long hi = 0, mid = FX_HALF;
#pragma unroll
  for (int c = 0; c + 1 < PB; c += 2) {
    const int4 s = *reinterpret_cast<const int4*>(row + c);
    hi += (long long)s.x * h[c];
    mid += (long long)s.x * l[c];
    mid += (long long)s.y * h[c];
    hi += (long long)s.z * h[c + 1];
    mid += (long long)s.z * l[c + 1];
    mid += (long long)s.w * h[c + 1];
  }
  if constexpr (PB % 2 == 1) {
    const int2 s = row[PB - 1];
    hi += (long long)s.x * h[PB - 1];
    mid += (long long)s.x * l[PB - 1];
    mid += (long long)s.y * h[PB - 1];
  }
  return hi + (mid >> FX_LIMB);
}

// fx_double for any exponent (under- and overflow as FP64 has them).
__device__ __forceinline__ double fx_double_any(long long R, int eb) {
  if ((unsigned)(eb - 1) < 1980u) return fx_double(R, eb);
  return scalbn(fx_double(R, 1023), eb - 1023);
}

// 2^-log2(multiplicity) of a local point.
__device__ __forceinline__ int fdm_mult_log2(const uint8_t* pflag, int64_t li) { return __ffs(pflag[li] & 0x0F) - 1; }

constexpr int FDM_SLOW = 7;  // index, among an element's ints, of the mark of one without a scale

// The solve in FP64 of the block's marked elements.  Every thread of the block calls it.
template <int P, int MODE>
__device__ __noinline__ void fdm_slow_block(const FdmFxArgs& a, int ne, int64_t e0, double* W0, const int* I0,
                                            size_t stride) {
  constexpr int N = P + 1, PB = P + 3, PB2 = PB * PB, PB3 = PB2 * PB;
  constexpr int C0 = MODE == FDM_RAS ? 1 : 0, NC = MODE == FDM_RAS ? N : PB;
  using Dm = FdmFxDims<PB>;
  const int tid = threadIdx.x, le = tid / PB2, ql = tid - le * PB2, p = ql % PB, q = ql / PB;
  const int es = le < ne ? le : 0;
  double* W = reinterpret_cast<double*>(reinterpret_cast<char*>(W0) + es * stride);
  const int* I = reinterpret_cast<const int*>(reinterpret_cast<const char*>(I0) + es * stride);
  const int* nb = I + 8;
  const bool on = le < ne && I[FDM_SLOW] != 0;
  const int64_t e = e0 + le;
  __syncthreads();
  if (on) {
#pragma unroll 1
    for (int c = 0; c < PB; ++c) {
      double v = 0.0;
      if constexpr (MODE == FDM_EXT_IN) {
        v = a.in[e * PB3 + p + PB * q + PB2 * c];
      } else {
        const int64_t src = window_source<P>(nb, e, p, q, c);
        if (src >= 0) v = a.in[src];
      }
      W[p + Dm::RS * q + Dm::PS * c] = v;
    }
  }
  __syncthreads();
  // phase f: direction of the lines, transposed or not
#pragma unroll 1
  for (int f = 0; f < 6; ++f) {
    const int d = f < 3 ? f : 5 - f;
    const int st = d == 0 ? 1 : (d == 1 ? Dm::RS : Dm::PS);
    const int base = d == 0 ? Dm::RS * p + Dm::PS * q : (d == 1 ? p + Dm::PS * q : p + Dm::RS * q);
    if (on) {
      double v[PB];
#pragma unroll
      for (int m = 0; m < PB; ++m) v[m] = W[base + st * m];
      const double* S = a.S + (3 * e + d) * PB2;
#pragma unroll 1
      for (int o = 0; o < PB; ++o) {
        double acc = 0.0;
#pragma unroll
        for (int m = 0; m < PB; ++m) acc = fma(f < 3 ? S[m * PB + o] : S[o * PB + m], v[m], acc);
        if (f == 2) acc *= a.dinv[e * PB3 + p + PB * q + PB2 * o];
        W[base + st * o] = acc;
      }
    }
    __syncthreads();
  }
  if (on && p >= C0 && p < C0 + NC && q >= C0 && q < C0 + NC) {
#pragma unroll 1
    for (int c = C0; c < C0 + NC; ++c) {
      const double v = W[p + Dm::RS * q + Dm::PS * c];
      if constexpr (MODE == FDM_RAS) {
        const int64_t li = e * (N * N * N) + (p - 1) + N * ((q - 1) + N * (c - 1));
        a.out[li] = scalbn(v, -fdm_mult_log2(a.pflag, li));
      } else {
        a.out[e * PB3 + p + PB * q + PB2 * c] = v;
      }
    }
  }
}

template <int P>
constexpr int fdm_fx_regs() { return P == 8 || P == 9 ? 72 : 64; }

template <int P, int MODE>
__global__ void __maxnreg__(fdm_fx_regs<P>()) fdm_fx_kernel(const __grid_constant__ FdmFxArgs a) {
  constexpr int N = P + 1, PB = P + 3, PB2 = PB * PB, PB3 = PB2 * PB;
  constexpr int C0 = MODE == FDM_RAS ? 1 : 0, NC = MODE == FDM_RAS ? N : PB;  // outputs kept per direction
  using Dm = FdmFxDims<PB>;
  constexpr int RS = Dm::RS, PS = Dm::PS, PBP = Dm::PBP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int64_t e0 = (int64_t)blockIdx.x * a.NE;
  const int ne = (int)(a.E - e0 < a.NE ? a.E - e0 : a.NE);
  const int tid = threadIdx.x;
  auto base_of = [&](int le) { return smem_raw + (size_t)le * Dm::BYTES; };
  auto W_of = [&](int le) { return reinterpret_cast<double*>(base_of(le)); };
  auto M_of = [&](int le) { return reinterpret_cast<int2*>(base_of(le)) + Dm::VOL; };  // S^T x 3, S x 3
  // ints: [0..2] largest high words (fx_mag) of S_x, S_y, S_z, [3] of the window, [4] of phase x,
  // [5] phase y, [6] exponent after z, [7] without a scale (FDM_SLOW), [8..34] neighbours
  auto I_of = [&](int le) { return reinterpret_cast<int*>(M_of(le) + 6 * Dm::SMAT); };
  for (int q = tid; q < ne * 8; q += blockDim.x) I_of(q >> 3)[q & 7] = (q & 7) == 6 ? INT_MIN : 0;
  for (int q = tid; q < ne * 27; q += blockDim.x) I_of(q / 27)[8 + q % 27] = a.nbr[27 * e0 + q];
  const int le = tid / PB2, ql = tid - le * PB2;
  const bool on = le < ne;
  const int es = on ? le : 0;            // element whose shared data the thread reads
  const int lp = ql % PB, lq = ql / PB;
  const unsigned peers = __match_any_sync(__activemask(), on ? le : -1);
  double* W = W_of(es);
  long long* WR = reinterpret_cast<long long*>(W);
  int2* ST = M_of(es);
  int2* SR = ST + 3 * Dm::SMAT;
  int* I = I_of(es);
  unsigned* mag = reinterpret_cast<unsigned*>(I);
  const int64_t e = e0 + es;
  if (on && ql == 0) fx_prefetch(a.dinv + e * PB3, PB3);  // needed after the forward contractions
  double s3[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) s3[d] = on ? a.S[(3 * e + d) * PB2 + ql] : 0.0;
  __syncthreads();
  // shift that brings a line of results to 63 bits
  auto line_norm = [](const long long* w, int st) {
    unsigned high = 0u;
#pragma unroll
    for (int q = 0; q < PB; ++q) {
      const int x = reinterpret_cast<const int*>(w + st * q)[1];
      high |= (unsigned)(x ^ (x >> 31));
    }
    return fx_norm(high);
  };
  // ---- gather the window (thread: (a, b), loop over c), the matrices' largest entries
  if (on) {
#pragma unroll
    for (int c = 0; c < PB; ++c) {
      double v = 0.0;
      if constexpr (MODE == FDM_EXT_IN) {
        v = a.in[e * PB3 + ql + PB2 * c];
      } else {
        const int64_t src = window_source<P>(I + 8, e, lp, lq, c);
        if (src >= 0) v = a.in[src];
      }
      W[lp + RS * lq + PS * c] = v;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) fx_group_max(peers, fx_mag(s3[d]), mag + d);
  }
  __syncthreads();
  double v[PB];
  bool bad = false;   // of the thread's element: S or the window without a scale
  unsigned low = 0u;  // low words of a line whose high words are all 0
  {
    unsigned m = 0u;
#pragma unroll
    for (int q = 0; q < PB; ++q) {
      v[q] = W[RS * lp + PS * lq + q];
      m = max(m, fx_mag(v[q]));
    }
    if (m == 0u) {
#pragma unroll
      for (int q = 0; q < PB; ++q) low |= (unsigned)__double2loint(v[q]);
    }
    if (on) {
      fx_group_max(peers, m, mag + 3);
      // limbs of S (row lq, column lp) and of its transpose
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const unsigned ms = mag[d];
        bad |= fx_bad(ms);
        int h, l;
        fx_split<57, true>(s3[d], fx_exponent(ms), h, l);
        SR[d * Dm::SMAT + lq * PBP + lp] = make_int2(h, l);
        ST[d * Dm::SMAT + lp * PBP + lq] = make_int2(h, l);
      }
    }
  }
  __syncthreads();
  bad |= fx_bad(mag[3]) || (mag[3] == 0u && low != 0u);
  if (on && bad) I[FDM_SLOW] = 1;
  int E = fx_exponent(mag[3]);  // x in units of 2^(E - 1023 - 57)
  auto kS = [&](int d) { return 1079 - fx_exponent(mag[d]); };
  int h[PB], l[PB];
  // ---- S_x^T along a (line (b, c))
  if (on) {
#pragma unroll
    for (int q = 0; q < PB; ++q) fx_split<58>(v[q], E, h[q], l[q]);
    unsigned m = 0u;
#pragma unroll
    for (int o = 0; o < PB; ++o) {
      const long long r = fx_dot_row<PB>(ST + o * PBP, h, l);
      WR[RS * lp + PS * lq + o] = r;
      m = max(m, fx_high(r));
    }
    fx_group_max(peers, m, mag + 4);
  }
  E -= kS(0);
  bool slow = __syncthreads_or(on && bad);  // some element of the block
  // ---- S_y^T along b (line (alpha, c))
  {
    const int n = fx_norm(mag[4]);
    E += 61 - n;
    if (on) {
#pragma unroll
      for (int q = 0; q < PB; ++q) fx_renorm<58>(WR[lp + RS * q + PS * lq], n, h[q], l[q]);
      unsigned m = 0u;
#pragma unroll
      for (int o = 0; o < PB; ++o) {
        const long long r = fx_dot_row<PB>(ST + Dm::SMAT + o * PBP, h, l);
        WR[lp + RS * o + PS * lq] = r;
        m = max(m, fx_high(r));
      }
      fx_group_max(peers, m, mag + 5);
    }
    E -= kS(1);
  }
  __syncthreads();
  // ---- S_z^T along c, D^-1, S_z (line (alpha, beta)); the line's own scale
  {
    const int n = line_norm(WR + lp + RS * lq, PS);
    E += 61 - n;
    long long r3[NC];
    int sft = 0, nl = 0;
    if (on) {
      double dv[PB];
#pragma unroll
      for (int q = 0; q < PB; ++q) dv[q] = a.dinv[e * PB3 + ql + PB2 * q];
#pragma unroll
      for (int q = 0; q < PB; ++q) fx_renorm<58>(WR[lp + RS * lq + PS * q], n, h[q], l[q]);
      unsigned m = 0u;
#pragma unroll
      for (int o = 0; o < PB; ++o) {
        v[o] = fx_double_any(fx_dot_row<PB>(ST + 2 * Dm::SMAT + o * PBP, h, l), E - 1 - kS(2)) * dv[o];
        m = max(m, fx_mag(v[o]));
      }
      if (fx_bad(m)) I[FDM_SLOW] = 1;
      const int E2 = fx_exponent(m);
#pragma unroll
      for (int q = 0; q < PB; ++q) fx_split<58>(v[q], E2, h[q], l[q]);
      unsigned high = 0u, any = 0u;
#pragma unroll
      for (int o = 0; o < NC; ++o) {
        r3[o] = fx_dot_row<PB>(SR + 2 * Dm::SMAT + (C0 + o) * PBP, h, l);
        high = max(high, fx_high(r3[o]));
        any |= (unsigned)r3[o];
      }
      // the line's largest value has its leading bit at 62 - nl, exponent 62 - nl + E2 - k
      nl = fx_norm(high);
      sft = E2 - 1 - kS(2);
      if (high | any) atomicMax(I + 6, 62 - nl + sft);
    }
    slow |= __syncthreads_or(on && I[FDM_SLOW] != 0);
    E = I[6] == INT_MIN ? FX_EMIN : I[6];
    if (on) {
      // x = r3 2^(sft - E + 57): left to 63 bits, then right (by 5 at least)
      const int right = nl - (sft - E + 57);
#pragma unroll
      for (int o = 0; o < NC; ++o) {
        int xh, xl;
        fx_shift_limbs((long long)((unsigned long long)r3[o] << nl), right - 1, xh, xl);
        reinterpret_cast<int2*>(W)[lp + RS * lq + PS * (C0 + o)] = make_int2(xh, xl);
      }
    }
  }
  __syncthreads();
  // ---- S_y along beta (line (alpha, c'), PB NC lines per element)
  {
    const int le2 = tid / (PB * NC), q2 = tid - le2 * PB * NC;
    const bool on2 = le2 < ne;
    const int e2 = on2 ? le2 : 0;
    const int al = q2 % PB, c = C0 + q2 / PB;
    if (on2) {
      const int2* Wl = reinterpret_cast<const int2*>(W_of(e2));
      const int2* Sy = M_of(e2) + 4 * Dm::SMAT;
#pragma unroll
      for (int q = 0; q < PB; ++q) {
        const int2 x = Wl[al + RS * q + PS * c];
        h[q] = x.x;
        l[q] = x.y;
      }
#pragma unroll
      for (int o = 0; o < NC; ++o)
        reinterpret_cast<long long*>(W_of(e2))[al + RS * (C0 + o) + PS * c] = fx_dot_row<PB>(Sy + (C0 + o) * PBP, h, l);
    }
  }
  __syncthreads();
  // ---- S_x along alpha (line (b', c'), NC^2 lines per element), write out
  const int le3 = tid / (NC * NC), q3 = tid - le3 * NC * NC;
  if (le3 < ne && I_of(le3)[FDM_SLOW] == 0) {
    const int b = C0 + q3 % NC, c = C0 + q3 / NC;
    const int* I3 = I_of(le3);
    const unsigned* mag3 = reinterpret_cast<const unsigned*>(I3);
    const int Em = I3[6] == INT_MIN ? FX_EMIN : I3[6];
    const long long* Wl = reinterpret_cast<const long long*>(W_of(le3)) + RS * b + PS * c;
    const int n = line_norm(Wl, 1);
    const int eb = Em - (1079 - fx_exponent(mag3[1])) + 60 - n - (1079 - fx_exponent(mag3[0]));
    const int2* Sx = M_of(le3) + 3 * Dm::SMAT;
#pragma unroll
    for (int q = 0; q < PB; ++q) fx_renorm<58>(Wl[q], n, h[q], l[q]);
    const int64_t eo = e0 + le3;
#pragma unroll
    for (int o = 0; o < NC; ++o) {
      const long long r = fx_dot_row<PB>(Sx + (C0 + o) * PBP, h, l);
      if constexpr (MODE == FDM_RAS) {
        const int64_t li = eo * (N * N * N) + o + N * ((b - 1) + N * (c - 1));
        a.out[li] = fx_double_any(r, eb - fdm_mult_log2(a.pflag, li));  // x 1/multiplicity
      } else {
        a.out[eo * PB3 + o + PB * (b + PB * c)] = fx_double_any(r, eb);
      }
    }
  }
  if (slow) fdm_slow_block<P, MODE>(a, ne, e0, W_of(0), I_of(0), Dm::BYTES);
}

template <int P, int MODE>
static int launch_fdm_fx(const Level& lv, const double* in, double* out, int NE, cudaStream_t s) {
  constexpr int PB = P + 3;
  FdmFxArgs a{lv.E, NE, lv.nbr, in, lv.S64, lv.fdm_dinv64, lv.pflag, out};
  const int threads = (NE * PB * PB + 31) / 32 * 32;
  const size_t smem = NE * FdmFxDims<PB>::BYTES;
  static const cudaError_t attr = cudaFuncSetAttribute(
      fdm_fx_kernel<P, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  SE_CUDA(attr);
  fdm_fx_kernel<P, MODE><<<(unsigned)((lv.E + NE - 1) / NE), threads, smem, s>>>(a);
  SE_LAUNCH_CHECK();
  return SE_OK;
}

int fdm_fx_apply(const Level& lv, int mode, const double* in, double* out, int NE, cudaStream_t s) {
  switch (lv.p) {
#define SE_FDMFX_CASE(PP)                                                            \
  case PP:                                                                           \
    if (mode == FDM_RAS) return launch_fdm_fx<PP, FDM_RAS>(lv, in, out, NE, s);      \
    if (mode == FDM_FULL) return launch_fdm_fx<PP, FDM_FULL>(lv, in, out, NE, s);    \
    return launch_fdm_fx<PP, FDM_EXT_IN>(lv, in, out, NE, s);
    SE_FDMFX_CASE(1) SE_FDMFX_CASE(2) SE_FDMFX_CASE(3) SE_FDMFX_CASE(4) SE_FDMFX_CASE(5)
    SE_FDMFX_CASE(6) SE_FDMFX_CASE(7) SE_FDMFX_CASE(8) SE_FDMFX_CASE(9) SE_FDMFX_CASE(10)
#undef SE_FDMFX_CASE
    default: set_error("fdm: unsupported p=%d", lv.p); return SE_EINVAL;
  }
}

}  // namespace se
