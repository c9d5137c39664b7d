// Values of the per-block flags of the register-resident coarse solver (coarse.cu).  A block publishes
// coarse_flag(it) once its w of iteration `it` is in memory; a block whose stencil reaches it waits
// for that value.  Flags only grow: a waiter may poll late, when its neighbour is one iteration
// further or has left the loop, and must then find its generation passed, not missing.
// Compiles as host code, so that the order can be checked without a GPU.
#pragma once

#ifdef __CUDACC__
#define SE_FLAG __host__ __device__ __forceinline__
#else
#define SE_FLAG inline
#endif

namespace se {

// Generation of iteration `it` (0: nothing published yet).
SE_FLAG unsigned coarse_flag(int it) { return (unsigned)it + 1u; }

// What a block that left the loop after `it` updates publishes with its last arrival: nothing waits
// for a further generation, but a neighbour may not have polled for that of `it` yet.
SE_FLAG unsigned coarse_flag_final(int it) { return coarse_flag(it); }

SE_FLAG bool coarse_flag_reached(unsigned flag, unsigned want) { return (int)(flag - want) >= 0; }

}  // namespace se
