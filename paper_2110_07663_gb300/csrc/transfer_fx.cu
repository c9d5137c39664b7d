// FP64 p-multigrid transfers in block floating point (fxp.h), every pair of orders:
//   prolongation e_f = (J x J x J) e_c,  restriction (J^T x J^T x J^T)(r_f / mult_f)
// element by element (transfer.cu adds QQ^T on the coarse level).  Both GLL point sets are symmetric
// about 0, so J is centro-symmetric and its lines fold.
//
// Each thread takes one line per direction and contracts it on the line's own scale.  The first
// direction's line is read straight from memory (NI consecutive values); its results, and the second
// direction's, are kept in shared memory as 64-bit integers on a scale common to the element, which
// starts from the element's largest value and then only takes the fixed bound of a contraction
// (|R| < 2^62): interpolation hardly changes magnitudes, so no renormalisation by value is needed.
// The last direction leaves as doubles, stored from its lines (a warp's lanes hold consecutive
// (a, b): each plane of an element is a contiguous store).
//
// Measured on GB300 (us per launch, restriction / prolongation; in brackets the FP64 kernels this one
// replaced, bound by the FP64 pipe): 32^3 elements p = 7 -> 5 96 / 86 [346 / 383], 5 -> 3 40 / 35
// [117 / 127], 3 -> 1 13 / 12 [23 / 25]; 20^3 9 -> 5 48 / 42 [135 / 140]; even orders (not folded
// before) 20^3 8 -> 4 34 / 29.  Memory needs 33 us of the 96; the rest is integer issue.
//
// Error against extended precision (2-norm) over the FP64 contraction's: 0.35 to 0.75 for random and
// smooth values, 0.7 to 2.7 for values that decay by eight decades across the element.  One scale per
// element for all three directions needed 40% fewer integer operations, but was 1.4 to 2.6 times less
// exact than FP64 in the restriction.
//
// Elements without a common scale (infinities, NaN, magnitudes at the ends of the range) send their
// block to transfer_slow_block, the same contraction in FP64.
#include "fxp.h"
#include "reduce.h"
#include "se_internal.h"

namespace se {

struct TransferFxArgs {
  int64_t E;
  const double *in, *J;
  const uint8_t* pflag;  // restriction: multiplicities of the input points
  double* out;
  int accumulate;        // out += instead of out =
};

template <int NF, int NC, bool RESTRICT>
struct TransferFxDims {
  static constexpr int NI = RESTRICT ? NF : NC, NO = RESTRICT ? NC : NF;
  static constexpr int L1 = NI * NI, L2 = NO * NI, L3 = NO * NO;  // lines per direction
  static constexpr int MOST = L1 > L3 ? L1 : L3;
  static constexpr int NE = MOST >= 256 ? 1 : (256 / MOST > 16 ? 16 : 256 / MOST);
  static constexpr int THREADS = (NE * MOST + 31) / 32 * 32;
  static constexpr int RB = NO % 2 ? NO : NO + 1;   // row stride of the first result
  static constexpr int B = RB * NI * NI, A = NO * NO * NI;
  static constexpr size_t SMEM = (size_t)NE * ((A + B) * 8 + 8);
};

// The line operator: J, or J^T for the restriction (host).
template <int NF, int NC, bool RESTRICT>
using TransferFxTable = FxFold<TransferFxDims<NF, NC, RESTRICT>::NO, TransferFxDims<NF, NC, RESTRICT>::NI>;

template <int NF, int NC, bool RESTRICT>
static TransferFxTable<NF, NC, RESTRICT> transfer_fx_table() {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  double J[NF * NC], M[NF * NC];
  interp_matrix(NF - 1, NC - 1, J);
  for (int o = 0; o < D::NO; ++o)
    for (int i = 0; i < D::NI; ++i) M[o * D::NI + i] = RESTRICT ? J[i * NC + o] : J[o * NC + i];
  return fx_fold_tables<D::NO, D::NI>(M, 1, 60);
}

__device__ __forceinline__ double transfer_fx_input(const TransferFxArgs& a, int64_t gi, bool weighted) {
  double v = a.in[gi];
  if (weighted) v = scale_pow2(v, mult_log2(a.pflag[gi]));
  return v;
}

template <int NF, int NC, bool RESTRICT>
__device__ __noinline__ void transfer_slow_block(const TransferFxArgs& a, int64_t e0, int ne, double* bufA, double* bufB) {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  constexpr int NI = D::NI, NO = D::NO;
  auto m = [&](int o, int i) { return RESTRICT ? a.J[i * NC + o] : a.J[o * NC + i]; };
  __syncthreads();
#pragma unroll 1
  for (int q = threadIdx.x; q < ne * NO * D::L1; q += blockDim.x) {
    const int le = q / (NO * D::L1), r = q - le * NO * D::L1, o = r % NO, jk = r / NO;
    double acc = 0.0;
#pragma unroll 1
    for (int i = 0; i < NI; ++i)
      acc = fma(m(o, i), transfer_fx_input(a, (e0 + le) * (NI * NI * NI) + i + NI * jk, RESTRICT), acc);
    bufB[le * D::B + o + D::RB * jk] = acc;
  }
  __syncthreads();
#pragma unroll 1
  for (int q = threadIdx.x; q < ne * NO * D::L2; q += blockDim.x) {
    const int le = q / (NO * D::L2), r = q - le * NO * D::L2, x = r % NO, b = (r / NO) % NO, k = r / (NO * NO);
    double acc = 0.0;
#pragma unroll 1
    for (int j = 0; j < NI; ++j) acc = fma(m(b, j), bufB[le * D::B + x + D::RB * (j + NI * k)], acc);
    bufA[le * D::A + x + NO * (b + NO * k)] = acc;
  }
  __syncthreads();
#pragma unroll 1
  for (int q = threadIdx.x; q < ne * NO * D::L3; q += blockDim.x) {
    const int le = q / (NO * D::L3), r = q - le * NO * D::L3, ab = r % D::L3, c = r / D::L3;
    double acc = 0.0;
#pragma unroll 1
    for (int k = 0; k < NI; ++k) acc = fma(m(c, k), bufA[le * D::A + ab + D::L3 * k], acc);
    double* out = a.out + (e0 + le) * (NO * NO * NO) + r;
    *out = a.accumulate ? *out + acc : acc;
  }
}

template <int NF, int NC, bool RESTRICT>
__global__ void __launch_bounds__(TransferFxDims<NF, NC, RESTRICT>::THREADS)
    transfer_fx_kernel(const __grid_constant__ TransferFxArgs a,
                       const __grid_constant__ TransferFxTable<NF, NC, RESTRICT> m) {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  constexpr int NI = D::NI, NO = D::NO, NE = D::NE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* bufB = reinterpret_cast<long long*>(smem_raw);  // first direction's results
  long long* bufA = bufB + NE * D::B;                         // second direction's
  unsigned* mags = reinterpret_cast<unsigned*>(bufA + NE * D::A);
  const int tid = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * NE;
  const int ne = (int)(a.E - e0 < NE ? a.E - e0 : NE);
  if (tid < NE) mags[tid] = 0u;
  __syncthreads();
  int h[NI], l[NI];
  // ---- direction r: lines (j, k)
  bool bad = false;
  {
    const int le = tid / D::L1, jk = tid - le * D::L1;
    const bool on = le < ne;
    int E = FX_EMIN;
    if (on) {
      double v[NI];
      unsigned mag = 0u;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        v[i] = transfer_fx_input(a, (e0 + le) * (NI * NI * NI) + i + NI * jk, RESTRICT);
        mag = max(mag, fx_mag(v[i]));
      }
      if (mag) atomicMax(mags + le, mag);
      bad = fx_bad(mag);
      E = fx_exponent(mag);
#pragma unroll
      for (int i = 0; i < NI; ++i) fx_split(v[i], E, h[i], l[i]);
    }
    __syncthreads();
    if (on) {
      const int back = fx_exponent(mags[le]) - E;
      long long* B = bufB + le * D::B + D::RB * jk;
      fx_contract<NO, NI, 1>(m, h, l, [&](int o, long long r) { B[o] = fx_shr(r, back); });
    }
  }
  bad = __syncthreads_or(bad);
  if (bad) {
    transfer_slow_block<NF, NC, RESTRICT>(a, e0, ne, reinterpret_cast<double*>(bufA), reinterpret_cast<double*>(bufB));
    return;
  }
  // a line of results on its own scale: R 2^n / 2^6
  auto line = [&](const long long* p, int st) {
    unsigned high = 0u;
    long long r[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      r[i] = p[st * i];
      high = max(high, fx_high(r[i]));
    }
    const int n = fx_norm(high);
#pragma unroll
    for (int i = 0; i < NI; ++i) fx_renorm(r[i], n, h[i], l[i]);
    return n;
  };
  // ---- direction s: lines (a, k); |R| < 2^62 needs n >= 1, the common scale is that of n = 1
  {
    const int le = tid / D::L2, r2 = tid - le * D::L2, k = r2 / NO, x = r2 - k * NO;
    if (le < ne) {
      const int back = line(bufB + le * D::B + x + D::RB * NI * k, D::RB) - 1;
      long long* A = bufA + le * D::A + x + D::L3 * k;
      fx_contract<NO, NI, 1>(m, h, l, [&](int o, long long r) { A[NO * o] = fx_shr(r, back); });
    }
  }
  __syncthreads();
  // ---- direction t: lines (a, b), stored to memory
  {
    const int le = tid / D::L3, ab = tid - le * D::L3;
    if (le < ne) {
      const int n = line(bufA + le * D::A + ab, D::L3);
      // x in units 2^(E - 1079) gives R in units 2^(E - 1023 - k); R 2^n / 2^6 has E + 62 - n - k
      const int eb = fx_exponent(mags[le]) - m.k + 61 - m.k + 62 - n - m.k;
      double* out = a.out + (e0 + le) * (NO * NO * NO) + ab;
      fx_contract<NO, NI, 1>(m, h, l, [&](int o, long long r) {
        const double v = fx_double(r, eb);
        out[D::L3 * o] = a.accumulate ? out[D::L3 * o] + v : v;
      });
    }
  }
}

template <int NF, int NC, bool RESTRICT>
static int launch_transfer_fx(int64_t E, const double* J, const double* in, const uint8_t* pflag, double* out,
                              bool accumulate, cudaStream_t s) {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  static_assert(D::SMEM <= 96 * 1024, "transfer block: shared memory");
  static const TransferFxTable<NF, NC, RESTRICT> table = transfer_fx_table<NF, NC, RESTRICT>();
  static const cudaError_t attr = cudaFuncSetAttribute(
      transfer_fx_kernel<NF, NC, RESTRICT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  SE_CUDA(attr);
  const TransferFxArgs a{E, in, J, pflag, out, accumulate};
  transfer_fx_kernel<NF, NC, RESTRICT><<<(unsigned)((E + D::NE - 1) / D::NE), D::THREADS, D::SMEM, s>>>(a, table);
  SE_LAUNCH_CHECK();
  return SE_OK;
}

template <int NF, int NC>
static int transfer_fx_pair(int Nc, bool restrict_, int64_t E, const double* J, const double* in,
                            const uint8_t* pflag, double* out, bool accumulate, cudaStream_t s) {
  if (Nc == NC)
    return restrict_ ? launch_transfer_fx<NF, NC, true>(E, J, in, pflag, out, accumulate, s)
                     : launch_transfer_fx<NF, NC, false>(E, J, in, pflag, out, accumulate, s);
  if constexpr (NC + 1 < NF) return transfer_fx_pair<NF, NC + 1>(Nc, restrict_, E, J, in, pflag, out, accumulate, s);
  set_error("transfer: unsupported orders %d, %d", NF - 1, Nc - 1);
  return SE_EINVAL;
}

int transfer_fx(const Level& f, const Level& c, bool restrict_, const double* J, const double* in, double* out,
                bool accumulate, cudaStream_t s) {
  switch (f.N) {
#define SE_TRFX_CASE(NN) \
  case NN: return transfer_fx_pair<NN, 2>(c.N, restrict_, f.E, J, in, f.pflag, out, accumulate, s);
    SE_TRFX_CASE(3) SE_TRFX_CASE(4) SE_TRFX_CASE(5) SE_TRFX_CASE(6) SE_TRFX_CASE(7)
    SE_TRFX_CASE(8) SE_TRFX_CASE(9) SE_TRFX_CASE(10) SE_TRFX_CASE(11)
#undef SE_TRFX_CASE
    default: set_error("transfer: unsupported order %d", f.p); return SE_EINVAL;
  }
}

}  // namespace se
