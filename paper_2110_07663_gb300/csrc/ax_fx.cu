// FP64 local Ax with folded line contractions in block floating point (fxp.h), every N.
//
// Sum factorisation: (ur, us, ut) = (D_r u, D_s u, D_t u);  w = G (ur, us, ut);
// y = D_r^T wr + D_s^T ws + D_t^T wt.  The six contractions run on the integer pipe: every line, of u
// and of w, is split into fixed point on the scale of its own largest value, so that a result's error is
// relative to its lines, as in FP64.  The gradients come back as doubles for the pointwise product
// with G (9 FP64 instructions per point, what is left on the FP64 pipe); the three parts of y stay
// 64-bit integers with the scale of their line, are added on the largest of the three scales and
// rounded to double once.  The derivative matrix is centro-antisymmetric, so a line of N values costs
// N^2/2 terms.
//
// NE elements per block, N^2 threads per element; each thread owns one line per direction.  Per
// element three arrays U, R, S in shared memory (rows of N padded to an odd stride, so that lines
// along every direction are read without bank conflicts; the padding holds the lines' scales), each
// updated in place: a thread writes a line's results over the line, and the column (i, j, 0..N-1)
// it owns holds wt in U.
//
// FOLD: the block's elements are consecutive in the element numbering, so neighbours along x
// (same row of the lattice, nx elements per row) are usually in the same block.  The kernel then
// also does the x part of QQ^T for them: both copies of each such x-interface node get
// left + right (the same bits on both sides), and it applies the Dirichlet mask (bit f of `bits`:
// face f = x0, x1, y0, y1, z0, z1 is Dirichlet); the x-interfaces between consecutive blocks are
// left to gs_fold_fixup_x.
//
// Measured on GB300 (us per launch; in brackets the even-odd FP64 kernel this one replaced, which ran at
// the FP64 pipe's 2 FMA/clk/SM): 32^3 elements p = 7 408 [1420], p = 5 203 [525], p = 3 54 [138]; even
// orders (unfolded in FP64) 20^3 p = 8 179 [725].  Memory needs 158 us of the 408 and the 9 FP64
// instructions per point 240; what bounds it is about 498 instructions per 32 points, 72 of them
// multiply-adds of 3.5 cycles each, at the 32 warps that its registers and shared memory allow (no
// pipe is full, each waits for the others in turn).  64 registers beat 48, 56, 72 and more;
// prefetching G to L2 costs more instructions than it saves waits.  w on one scale per element was 0.5%
// faster at p = 7 (406), but a small value then lost the bits below 2^-56 of the element's largest one,
// though no line joins them; the parts of y as doubles, added in FP64, cost about 470.
//
// Error against extended precision (2-norm, host emulation on plain and perturbed meshes, p = 2, 3, 7, 8
// and 10), over that of the FP64 dot products: 0.40 to 0.78 for random values, 0.40 to 0.50 for smooth
// ones, 0.32 to 0.67 for values that decay by eight decades across the element, 0.29 to 0.74 around one
// value 10^8 times the others; away from that value's lines the points keep FP64's accuracy.
//
// A line whose values cannot share a scale (infinities, NaN, magnitudes at the ends of the range) is
// contracted in FP64 (ax_slow_line); what does not touch it keeps its bits.
#include <climits>

#include "fxp.h"
#include "se_internal.h"

namespace se {

struct AxFxArgs {
  int64_t E, L;
  int NE;
  const double *u, *G, *D, *sub, *dinv;
  const uint8_t* pflag;
  double* y;
  int mask_in;             // zero the Dirichlet values of u as they are read
  int nx, ny, nz, bits;    // FOLD
};

// Splits the line p[0], p[st], ... on its own scale E; false where it has none (infinities, NaN,
// largest value at an end of the range).
template <int N>
__device__ __forceinline__ bool fx_split_line(const double* p, int st, int (&h)[N], int (&l)[N], int& E) {
  double v[N];
  unsigned mag = 0u;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    v[q] = p[st * q];
    mag = max(mag, fx_mag(v[q]));
  }
  bool scaled = !fx_bad(mag);
  if (mag == 0u) {  // zeros, or values so small that their high words are
    unsigned low = 0u;
#pragma unroll
    for (int q = 0; q < N; ++q) low |= (unsigned)__double2loint(v[q]);
    scaled = low == 0u;
  }
  E = fx_exponent(mag);
#pragma unroll
  for (int q = 0; q < N; ++q) fx_split(v[q], E, h[q], l[q]);
  return scaled;
}

// out = M in along a line without a scale, in FP64: M = D, or D^T.  in and out may be the same line.
template <int N>
__device__ __noinline__ void ax_slow_line(const double* D, bool transposed, const double* in, double* out, int st) {
  double v[N];
#pragma unroll
  for (int q = 0; q < N; ++q) v[q] = in[st * q];
#pragma unroll 1
  for (int k = 0; k < N; ++k) {
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < N; ++q) acc = fma(D[transposed ? q * N + k : k * N + q], v[q], acc);
    out[st * k] = acc;
  }
}

template <int N>
struct AxFxDims {
  static constexpr int NP = N % 2 ? N : N + 1;     // padded row: odd, so 8-byte lines do not conflict
  static constexpr int PLANE = NP * N, VOL = NP * N * N;
  // scales of the r- and s-lines of w: even N in the padding of R's and S's rows, odd N behind the arrays
  static constexpr int SIZE = 3 * VOL + (N % 2 ? (2 * N * N + 1) / 2 : 0);  // doubles per element
};

constexpr int FX_NO_SCALE = INT_MAX;  // of a line whose results are doubles

// Scale of line (c, k) of an array's N^2 lines, c the coordinate across and k = 0 .. N - 1 the plane.
template <int N>
__device__ __forceinline__ int* ax_line_scale(double* U, int array, int c, int k) {
  using Dm = AxFxDims<N>;
  if constexpr (N % 2) return reinterpret_cast<int*>(U + 3 * Dm::VOL) + (array - 1) * N * N + c + N * k;
  else return reinterpret_cast<int*>(U + array * Dm::VOL + Dm::NP * c + Dm::PLANE * k + N);
}

// A column's place in the lattice (FOLD): its element and its Dirichlet points (bit k).
struct AxLattice {
  int ex, ey, ez;
  unsigned zmask;
};
template <int N>
__device__ __forceinline__ AxLattice ax_lattice(const AxFxArgs& a, int e, int i, int j) {
  AxLattice r;
  r.ex = e % a.nx;
  r.ey = (e / a.nx) % a.ny;
  r.ez = e / (a.nx * a.ny);
  const bool dxy = ((a.bits & 1) && i == 0 && r.ex == 0) || ((a.bits & 2) && i == N - 1 && r.ex == a.nx - 1) ||
                   ((a.bits & 4) && j == 0 && r.ey == 0) || ((a.bits & 8) && j == N - 1 && r.ey == a.ny - 1);
  r.zmask = dxy ? (1u << N) - 1u : 0u;
  if ((a.bits & 16) && r.ez == 0) r.zmask |= 1u;
  if ((a.bits & 32) && r.ez == a.nz - 1) r.zmask |= 1u << (N - 1);
  return r;
}

// Input value of a local point: u, or D^-1 u, zero on masked points.
__device__ __forceinline__ double ax_fx_input(const AxFxArgs& a, int64_t gi, bool zero) {
  double v = a.u[gi];
  if (a.dinv) v *= a.dinv[gi];
  return zero ? 0.0 : v;
}

// The three parts of a result, each on its own scale, added on the largest of them (what a smaller one
// loses there is below 2^-60 of the sum's largest part) and rounded to double once.
__device__ __forceinline__ double ax_sum(long long t, int et, long long r, int er, long long s, int es, int k) {
  const int m = max(et, max(er, es));
  return fx_double(fx_shr(t, m - et) + fx_shr(r, m - er) + fx_shr(s, m - es), m - k);
}

// The last step of a column (i, j) where the column or a line through it has no scale (in a function of
// its own, out of the kernel's instruction stream): points without such a line get the same bits as ever.
template <int N>
__device__ __noinline__ void ax_slow_column(const double* D, const FxFold<N, N>& tT, double* U, int i, int j) {
  using Dm = AxFxDims<N>;
  constexpr int PL = Dm::PLANE;
  double* u = U + i + Dm::NP * j;
  int h[N], l[N], E;
  if (fx_split_line<N>(u, PL, h, l, E)) {
    fx_contract<N, N, -1>(tT, h, l, [&](int q, long long r) { reinterpret_cast<long long*>(u)[PL * q] = r; });
  } else {
    ax_slow_line<N>(D, true, u, u, PL);
    E = FX_NO_SCALE;
  }
  auto value = [&](const double* p, int e) {
    return e == FX_NO_SCALE ? *p : fx_double(*reinterpret_cast<const long long*>(p), e - tT.k);
  };
#pragma unroll 1
  for (int q = 0; q < N; ++q) {
    double *t = u + PL * q, *r = t + Dm::VOL, *s = r + Dm::VOL;
    const int er = *ax_line_scale<N>(U, 1, j, q), es = *ax_line_scale<N>(U, 2, i, q);
    if (max(E, max(er, es)) != FX_NO_SCALE)
      *t = ax_sum(*reinterpret_cast<const long long*>(t), E, *reinterpret_cast<const long long*>(r), er,
                  *reinterpret_cast<const long long*>(s), es, tT.k);
    else
      *t = value(t, E) + (value(r, er) + value(s, es));
  }
}

// Registers: the kernel waits on memory, shared memory and dependent integer operations in turn, so
// resident warps are worth more than registers up to the point where lines spill.
template <int N>
constexpr int ax_fx_regs() { return N <= 9 ? 64 : (N == 10 ? 72 : 96); }

template <int N, bool FOLD>
__global__ void __maxnreg__(ax_fx_regs<N>())
    ax_fx_kernel(const __grid_constant__ AxFxArgs a, const __grid_constant__ FxFoldRows<N, N> tD,
                 const __grid_constant__ FxFold<N, N> tT) {
  constexpr int N2 = N * N, N3 = N2 * N, NP = AxFxDims<N>::NP, PL = AxFxDims<N>::PLANE, VOL = AxFxDims<N>::VOL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int le = threadIdx.x / N2;
  const int t = threadIdx.x - le * N2;
  const int i = t % N, j = t / N;  // the thread's column; also (j, k) of its r-line, (i, k) of its s-line
  double* U = reinterpret_cast<double*>(smem_raw) + (size_t)le * AxFxDims<N>::SIZE;
  double* R = U + VOL;
  double* S = R + VOL;
  const int64_t e = (int64_t)blockIdx.x * a.NE + le;
  const bool valid = e < a.E;
  const int64_t eb = e * N3 + t;
  const int col = i + NP * j, rl = NP * i + PL * j, sl = i + PL * j;  // lines: column, (j=i,k=j), (i,k=j)
  // the column's place in the lattice (E < 2^31): needed last, worth registers until then for small N
  constexpr bool EARLY = FOLD && N < 8;
  AxLattice at{};
  if constexpr (EARLY) at = ax_lattice<N>(a, (int)e, i, j);
  // Dirichlet points of the column (bit k), to mask the input
  unsigned zin = 0u;
  if (a.mask_in && valid) {
    if constexpr (FOLD) {
      zin = EARLY ? at.zmask : ax_lattice<N>(a, (int)e, i, j).zmask;
    } else {
#pragma unroll
      for (int k = 0; k < N; ++k)
        if (!(a.pflag[eb + N2 * k] & PF_FREE)) zin |= 1u << k;
    }
  }
#pragma unroll
  for (int k = 0; k < N; ++k) U[col + PL * k] = valid ? ax_fx_input(a, eb + N2 * k, (zin >> k) & 1u) : 0.0;
  __syncthreads();
  // a line of doubles contracted on its own scale, st apart: in and out may be the same line
  auto contract = [&](const FxFoldRows<N, N>& m, bool transposed, const double* in, double* out, int st) {
    int h[N], l[N], E;
    if (fx_split_line<N>(in, st, h, l, E))
      fx_contract<N, N, -1>(m, h, l, [&](int q, long long r) { out[st * q] = fx_double(r, E - m.row_k(q)); });
    else
      ax_slow_line<N>(a.D, transposed, in, out, st);
  };
  // r-lines and s-lines
  contract(tD, false, U + rl, R + rl, 1);
  contract(tD, false, U + sl, S + sl, NP);
  __syncthreads();
  // t-lines and the pointwise factors: the thread's column.  From N = 8 the factors have a loop of
  // their own, two points at a time behind a barrier (which the compiler does not move loads across),
  // so that the contraction and the loads in flight do not compete for registers: p = 7 429 -> 406 us,
  // p = 8 192 -> 182, p = 9 283 -> 271; p = 5 and 6 are 8% faster fused (198, 138)
  constexpr bool SPLIT = N >= 8;
  const double* g = a.G + (valid ? eb : (int64_t)t);
  auto pointwise = [&](int q, double ut) {
    const double* gq = g + N2 * q;
    const double grr = gq[0], grs = gq[a.L], grt = gq[2 * a.L], gss = gq[3 * a.L], gst = gq[4 * a.L], gtt = gq[5 * a.L];
    const double ur = R[col + PL * q], us = S[col + PL * q];
    R[col + PL * q] = fma(grt, ut, fma(grs, us, grr * ur));
    S[col + PL * q] = fma(gst, ut, fma(gss, us, grs * ur));
    U[col + PL * q] = fma(gtt, ut, fma(gst, us, grt * ur));
  };
  if constexpr (SPLIT) {
    contract(tD, false, U + col, U + col, PL);
    __syncthreads();
#pragma unroll 2
    for (int q = 0; q < N; ++q) pointwise(q, U[col + PL * q]);
  } else {
    int h[N], l[N], E;
    if (fx_split_line<N>(U + col, PL, h, l, E)) {
      fx_contract<N, N, -1>(tD, h, l, [&](int q, long long r) { pointwise(q, fx_double(r, E - tD.row_k(q))); });
    } else {
      ax_slow_line<N>(a.D, false, U + col, U + col, PL);
#pragma unroll 1
      for (int q = 0; q < N; ++q) pointwise(q, U[col + PL * q]);
    }
  }
  __syncthreads();
  // r-lines and s-lines of w, in place: 64-bit integers on the line's own scale, or the doubles of a line
  // without one
  auto transposed = [&](double* w, int st) {
    int h[N], l[N], E;
    if (fx_split_line<N>(w, st, h, l, E)) {
      fx_contract<N, N, -1>(tT, h, l, [&](int q, long long r) { reinterpret_cast<long long*>(w)[st * q] = r; });
    } else {
      ax_slow_line<N>(a.D, true, w, w, st);
      E = FX_NO_SCALE;
    }
    return E;
  };
  const int Er = transposed(R + rl, 1), Es = transposed(S + sl, NP);
  *ax_line_scale<N>(U, 1, i, j) = Er;
  *ax_line_scale<N>(U, 2, i, j) = Es;
  const bool slow = __syncthreads_or(max(Er, Es) == FX_NO_SCALE);
  // t-lines, and the three parts added
  {
    int h[N], l[N], E;
    const bool scaled = fx_split_line<N>(U + col, PL, h, l, E);
    if (scaled && !slow) {
      fx_contract<N, N, -1>(tT, h, l, [&](int q, long long r) {
        U[col + PL * q] = ax_sum(r, E, reinterpret_cast<const long long*>(R)[col + PL * q], *ax_line_scale<N>(U, 1, j, q),
                                 reinterpret_cast<const long long*>(S)[col + PL * q], *ax_line_scale<N>(U, 2, i, q), tT.k);
      });
    } else {
      ax_slow_column<N>(a.D, tT, U, i, j);
    }
  }
  // U: A_L u, each thread's own column
  if constexpr (FOLD) {
    // residual form: each copy's b / multiplicity - (A_L u); a copy on an interior interface
    // normal to a direction has 2 copies along it, so the weight is a power of two, built from its
    // exponent bits
    double yv[N];
#pragma unroll
    for (int k = 0; k < N; ++k) yv[k] = U[col + PL * k];
    if constexpr (!EARLY) at = ax_lattice<N>(a, (int)e, i, j);
    if (a.sub) {
      const int xy = (int)((i == 0 && at.ex > 0) || (i == N - 1 && at.ex < a.nx - 1)) +
                     (int)((j == 0 && at.ey > 0) || (j == N - 1 && at.ey < a.ny - 1));
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int zi = (int)((k == 0 && at.ez > 0) || (k == N - 1 && at.ez < a.nz - 1));
        const double w = __longlong_as_double((long long)(1023 - xy - zi) << 52);
        yv[k] = valid ? a.sub[eb + N2 * k] * w - yv[k] : 0.0;
      }
    }
    // x-interfaces inside the block: (N - 1, j, k) of element lp and (0, j, k) of lp + 1 when both
    // lie in one row; both copies get left + right.  Each pair is added once, by one lane of
    // densely packed warps (a warp-wide FP64 instruction costs the same with 2 or 32 lanes active)
    const bool left = i == N - 1 && le + 1 < a.NE && e + 1 < a.E && at.ex < a.nx - 1;
    const bool right = i == 0 && le > 0 && at.ex > 0;
    if (left || right) {
#pragma unroll
      for (int k = 0; k < N; ++k) U[col + PL * k] = yv[k];
    }
    __syncthreads();
    const int64_t e0 = (int64_t)blockIdx.x * a.NE;
    for (int idx = threadIdx.x; idx < (a.NE - 1) * N2; idx += blockDim.x) {
      const int lp = idx / N2, jk = idx - lp * N2;
      const int el = (int)(e0 + lp);
      if (el + 1 < a.E && el % a.nx < a.nx - 1) {
        double* p = reinterpret_cast<double*>(smem_raw) + (size_t)lp * AxFxDims<N>::SIZE + NP * jk + N - 1;
        double* q = p + AxFxDims<N>::SIZE - (N - 1);
        const double v = *p + *q;
        *p = v;
        *q = v;
      }
    }
    __syncthreads();
    if (left || right) {
#pragma unroll
      for (int k = 0; k < N; ++k) yv[k] = U[col + PL * k];
    }
    if (valid) {
#pragma unroll
      for (int k = 0; k < N; ++k) a.y[eb + N2 * k] = ((at.zmask >> k) & 1u) ? 0.0 : yv[k];
    }
  } else {
    if (valid) {
#pragma unroll
      for (int k = 0; k < N; ++k) a.y[eb + N2 * k] = ax_output(U[col + PL * k], a.sub, a.pflag, eb + N2 * k);
    }
  }
}

// The x-interfaces that ax_fx_kernel<FOLD> leaves: element e = (b + 1) NE - 1, the last of block b,
// and e + 1, the first of block b + 1, when both lie in one row.  Thread: (boundary, point (j, k)
// of the face).  Masked copies are zero on both sides (a node's copies are all masked or none).
template <int N>
__global__ void gs_fold_fixup_x(int64_t E, int NE, int nx, double* __restrict__ y) {
  constexpr int N2 = N * N, N3 = N2 * N;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nbnd = (E + NE - 1) / NE - 1;
  if (t >= nbnd * N2) return;
  const int64_t b = t / N2;
  const int jk = (int)(t - b * N2);
  const int64_t e = (b + 1) * NE - 1;
  if (e + 1 >= E || (int)(e % nx) == nx - 1) return;
  const int64_t ia = e * N3 + (N - 1) + (int64_t)N * jk;  // (N - 1, j, k) of e
  const int64_t ib = (e + 1) * N3 + (int64_t)N * jk;      // (0, j, k) of e + 1
  const double v = y[ia] + y[ib];
  y[ia] = v;
  y[ib] = v;
}

template <int N>
struct AxFxTables {
  FxFoldRows<N, N> D;
  FxFold<N, N> T;  // D^T: three results are added in 64 bits
  explicit AxFxTables(const double* d) : D(fx_fold_rows<N, N>(d, -1)) {
    double t[N * N];
    for (int r = 0; r < N; ++r)
      for (int c = 0; c < N; ++c) t[r * N + c] = d[c * N + r];
    T = fx_fold_tables<N, N>(t, -1, 59);
  }
};

template <int N>
static int launch_ax_fx(const Level& lv, const double* u, double* y, bool mask_in, const double* sub,
                        const double* dinv, int NE, bool fold, cudaStream_t s) {
  static_assert(sizeof(FxFoldRows<N, N>) <= 1536, "two folded tables and the arguments fit the 4 KB of parameters");
  // the tables depend on the order only: formed once per process
  static const AxFxTables<N> tab(lv.basis.D);
  AxFxArgs a{};
  a.E = lv.E;
  a.L = lv.L;
  a.NE = NE;
  a.u = u;
  a.G = lv.G64;
  a.D = lv.D64;
  a.sub = sub;
  a.dinv = dinv;
  a.pflag = lv.pflag;
  a.y = y;
  a.mask_in = mask_in;
  const int threads = NE * N * N;
  const size_t smem = (size_t)NE * AxFxDims<N>::SIZE * sizeof(double);
  const unsigned blocks = (unsigned)((lv.E + NE - 1) / NE);
  if (fold) {
    a.nx = lv.nel[0];
    a.ny = lv.nel[1];
    a.nz = lv.nel[2];
    for (int f = 0; f < 6; ++f)
      if (lv.bc[f] == SE_BC_DIRICHLET) a.bits |= 1 << f;
    static const cudaError_t attr = cudaFuncSetAttribute(
        ax_fx_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    SE_CUDA(attr);
    ax_fx_kernel<N, true><<<blocks, threads, smem, s>>>(a, tab.D, tab.T);
  } else {
    static const cudaError_t attr = cudaFuncSetAttribute(
        ax_fx_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    SE_CUDA(attr);
    ax_fx_kernel<N, false><<<blocks, threads, smem, s>>>(a, tab.D, tab.T);
  }
  SE_LAUNCH_CHECK();
  return SE_OK;
}

// y = A_L (dinv .* u), or sub / multiplicity minus it.  fold: with the x-interface sums of the
// block's elements and the mask of the box lattice (NE elements per block).
int ax_local_fx(const Level& lv, const double* u, double* y, bool mask_in, const double* sub,
                const double* dinv, int NE, bool fold, cudaStream_t s) {
  switch (lv.N) {
#define SE_AXFX_CASE(NN) \
  case NN: return launch_ax_fx<NN>(lv, u, y, mask_in, sub, dinv, NE, fold, s);
    SE_AXFX_CASE(2) SE_AXFX_CASE(3) SE_AXFX_CASE(4) SE_AXFX_CASE(5) SE_AXFX_CASE(6)
    SE_AXFX_CASE(7) SE_AXFX_CASE(8) SE_AXFX_CASE(9) SE_AXFX_CASE(10) SE_AXFX_CASE(11)
#undef SE_AXFX_CASE
    default: set_error("ax: unsupported N=%d", lv.N); return SE_EINVAL;
  }
}

int gs_fold_fixup(const Level& lv, double* y, int NE, cudaStream_t s) {
  const int64_t nbnd = (lv.E + NE - 1) / NE - 1;
  if (nbnd <= 0 || lv.nel[0] <= 1) return SE_OK;
  const int64_t n = nbnd * lv.N * lv.N;
  switch (lv.N) {
#define SE_FIX_CASE(NN)                                                                      \
  case NN:                                                                                   \
    gs_fold_fixup_x<NN><<<grid_for(n, 256), 256, 0, s>>>(lv.E, NE, lv.nel[0], y);            \
    break;
    SE_FIX_CASE(2) SE_FIX_CASE(3) SE_FIX_CASE(4) SE_FIX_CASE(5) SE_FIX_CASE(6)
    SE_FIX_CASE(7) SE_FIX_CASE(8) SE_FIX_CASE(9) SE_FIX_CASE(10) SE_FIX_CASE(11)
#undef SE_FIX_CASE
    default: set_error("gs_fold_fixup: unsupported N=%d", lv.N); return SE_EINVAL;
  }
  SE_LAUNCH_CHECK();
  return SE_OK;
}

}  // namespace se
