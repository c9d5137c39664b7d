// The extended Schwarz window (Fig. 1b): modes of the FDM kernels and where a window point lives.
#pragma once
#include <cstdint>

namespace se {

enum { FDM_RAS = 0, FDM_FULL = 1, FDM_EXT_IN = 2, FDM_GATHER = 3 };

// Window point (a, b, c) of element e: index in the L-vector, -1 outside the domain.
template <int P>
__device__ __forceinline__ int64_t window_source(const int* __restrict__ nb, int64_t e, int a,
                                                 int b, int c) {
  constexpr int N = P + 1, PB = P + 3;
  const int da = a == 0 ? -1 : (a == PB - 1 ? 1 : 0);
  const int db = b == 0 ? -1 : (b == PB - 1 ? 1 : 0);
  const int dc = c == 0 ? -1 : (c == PB - 1 ? 1 : 0);
  int64_t src = e;
  if (da | db | dc) {
    src = nb[(da + 1) + 3 * (db + 1) + 9 * (dc + 1)];
    if (src < 0) return -1;
  }
  const int ia = da < 0 ? P - 1 : (da > 0 ? 1 : a - 1);
  const int ib = db < 0 ? P - 1 : (db > 0 ? 1 : b - 1);
  const int ic = dc < 0 ? P - 1 : (dc > 0 ? 1 : c - 1);
  return src * (N * N * N) + ia + N * (ib + N * ic);
}

}  // namespace se
