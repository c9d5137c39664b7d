// FP64 p-multigrid transfers in block floating point (fxp.h), every pair of orders:
//   prolongation e_f = (J x J x J) e_c,  restriction (J^T x J^T x J^T)(r_f / mult_f)
// element by element (transfer.cu adds QQ^T on the coarse level).  Both GLL point sets are symmetric
// about 0, so J is centro-symmetric and its lines fold.
//
// Each thread takes one line per direction and contracts it on the line's own scale; between the
// directions the values are doubles in shared memory.  The first direction's line is read straight
// from memory (NI consecutive values), the last direction's results are stored from its lines (a
// warp's lanes hold consecutive (a, b): each plane of an element is a contiguous store).
//
// The two point sets share their end points (and for two odd counts the middle one), where J's rows are
// unit vectors: prolongation copies those values and contracts the others; restriction adds them to
// their one result and contracts the inner points only.  So a value is never cut on the scale of values
// that do not enter its result, and a face of the prolonged vector depends on the face's values
// alone: both copies of an interface point get the same bits.
//
// Measured on GB300 (us per launch, restriction / prolongation; in brackets the FP64 kernels this one
// replaced, bound by the FP64 pipe): 32^3 elements p = 7 -> 5 99 / 88 [346 / 383], 5 -> 3 41 / 34
// [117 / 127], 3 -> 1 13 / 11 [23 / 25]; 20^3 9 -> 5 50 / 43 [135 / 140]; even orders (not folded
// before) 20^3 8 -> 4 33 / 27.  Memory needs 33 us of the 99; the rest is integer issue.  64-bit
// integers on the element's scale between the directions were 0 to 6% faster (96 / 86, 40 / 35), but
// cut every value on its element's largest one, and left the copies of an interface point
// unequal.
//
// Error against extended precision (2-norm, host emulation), over the FP64 contraction's: 0.43 to 0.89
// for random values, 0.40 to 1.0 for smooth ones, 0.33 to 0.78 for values that decay by eight decades
// across the element, 0.28 to 1.01 around one value 10^8 times the others (2 -> 1, whose rows have two
// entries of 1/2: 1.0 to 1.19, the conversion rounds ties upwards).
//
// A line without a scale (infinities, NaN, magnitudes at the ends of the range) is contracted in FP64 by
// itself.
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
  static constexpr size_t SMEM = (size_t)NE * (A + B) * 8;
  // what is contracted: prolongation all inputs to the inner outputs, restriction the inner inputs
  static constexpr int I0 = RESTRICT ? 1 : 0, O0 = RESTRICT ? 0 : 1, NL = NI - 2 * I0, NR = NO - 2 * O0;
  static constexpr bool MID = NI % 2 == 1 && NO % 2 == 1;  // a middle point in common
};

// The line operator without its unit rows: rows of J, or columns of J^T for the restriction (host).
template <int NF, int NC, bool RESTRICT>
using TransferFxTable = FxFold<TransferFxDims<NF, NC, RESTRICT>::NR, TransferFxDims<NF, NC, RESTRICT>::NL>;

template <int NF, int NC, bool RESTRICT>
static TransferFxTable<NF, NC, RESTRICT> transfer_fx_table() {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  double J[NF * NC], M[D::NR * D::NL];
  interp_matrix(NF - 1, NC - 1, J);
  for (int o = 0; o < D::NR; ++o)
    for (int i = 0; i < D::NL; ++i)
      M[o * D::NL + i] = RESTRICT ? J[(i + D::I0) * NC + o] : J[(o + D::O0) * NC + i];
  return fx_fold_tables<D::NR, D::NL>(M, 1, 60);
}

__device__ __forceinline__ double transfer_fx_input(const TransferFxArgs& a, int64_t gi, bool weighted) {
  double v = a.in[gi];
  if (weighted) v = scale_pow2(v, mult_log2(a.pflag[gi]));
  return v;
}

// out(o, value) of the line v, on its own scale; false where it has none.
template <int NF, int NC, bool RESTRICT, class Out>
__device__ __forceinline__ bool transfer_fx_line(const TransferFxTable<NF, NC, RESTRICT>& m,
                                                 const double (&v)[TransferFxDims<NF, NC, RESTRICT>::NI], Out&& out) {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  constexpr int NI = D::NI, NO = D::NO, NL = D::NL;
  // the value that only adds to its own result
  auto apart = [](int i) { return RESTRICT && D::MID && i == NI / 2; };
  unsigned mag = 0u, rest = 0u;
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const bool in = i >= D::I0 && i < NI - D::I0 && !apart(i);
    (in ? mag : rest) = max(in ? mag : rest, fx_mag(v[i]));
  }
  if (fx_bad(mag) || fx_bad(max(mag, rest))) return false;
  if (mag == 0u) {  // zeros, or values so small that their high words are
    unsigned low = 0u;
#pragma unroll
    for (int i = D::I0; i < NI - D::I0; ++i) low |= (unsigned)__double2loint(v[i]);
    if (low != 0u) return false;
  }
  const int E = fx_exponent(mag);
  int h[NL], l[NL];
#pragma unroll
  for (int i = 0; i < NL; ++i) {
    fx_split(v[i + D::I0], E, h[i], l[i]);
    if (apart(i + D::I0)) h[i] = l[i] = 0;
  }
  if constexpr (!RESTRICT) {
    out(0, v[0]);
    out(NO - 1, v[NI - 1]);
    if constexpr (D::MID) out(NO / 2, v[NI / 2]);
  }
  fx_contract<D::NR, NL, 1>(m, h, l, [&](int q, long long r) {
    const int o = q + D::O0;
    const double w = fx_double(r, E - m.k);
    if (RESTRICT && o == 0) out(o, w + v[0]);
    else if (RESTRICT && o == NO - 1) out(o, w + v[NI - 1]);
    else if (RESTRICT && D::MID && o == NO / 2) out(o, w + v[NI / 2]);
    else if (!(!RESTRICT && D::MID && o == NO / 2)) out(o, w);
  });
  return true;
}

template <int NF, int NC, bool RESTRICT>
__global__ void __launch_bounds__(TransferFxDims<NF, NC, RESTRICT>::THREADS)
    transfer_fx_kernel(const __grid_constant__ TransferFxArgs a,
                       const __grid_constant__ TransferFxTable<NF, NC, RESTRICT> m) {
  using D = TransferFxDims<NF, NC, RESTRICT>;
  constexpr int NI = D::NI, NO = D::NO, NE = D::NE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* bufB = reinterpret_cast<double*>(smem_raw);  // first direction's results
  double* bufA = bufB + NE * D::B;                     // second direction's
  const int tid = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * NE;
  const int ne = (int)(a.E - e0 < NE ? a.E - e0 : NE);
  // a line: in(i) read once, results to out(o, value)
  auto line = [&](auto&& in, auto&& out) {
    double v[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) v[i] = in(i);
    if (!transfer_fx_line<NF, NC, RESTRICT>(m, v, out)) {
#pragma unroll 1
      for (int o = 0; o < NO; ++o) {
        double acc = 0.0;
#pragma unroll
        for (int i = 0; i < NI; ++i) acc = fma(RESTRICT ? a.J[i * NC + o] : a.J[o * NC + i], v[i], acc);
        out(o, acc);
      }
    }
  };
  // ---- direction r: lines (j, k)
  {
    const int le = tid / D::L1, jk = tid - le * D::L1;
    if (le < ne) {
      double* B = bufB + le * D::B + D::RB * jk;
      line([&](int i) { return transfer_fx_input(a, (e0 + le) * (NI * NI * NI) + i + NI * jk, RESTRICT); },
           [&](int o, double w) { B[o] = w; });
    }
  }
  __syncthreads();
  // ---- direction s: lines (a, k)
  {
    const int le = tid / D::L2, r2 = tid - le * D::L2, k = r2 / NO, x = r2 - k * NO;
    if (le < ne) {
      const double* B = bufB + le * D::B + x + D::RB * NI * k;
      double* A = bufA + le * D::A + x + D::L3 * k;
      line([&](int i) { return B[D::RB * i]; }, [&](int o, double w) { A[NO * o] = w; });
    }
  }
  __syncthreads();
  // ---- direction t: lines (a, b), stored to memory
  {
    const int le = tid / D::L3, ab = tid - le * D::L3;
    if (le < ne) {
      const double* A = bufA + le * D::A + ab;
      double* out = a.out + (e0 + le) * (NO * NO * NO) + ab;
      line([&](int i) { return A[D::L3 * i]; },
           [&](int o, double w) { out[D::L3 * o] = a.accumulate ? out[D::L3 * o] + w : w; });
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
