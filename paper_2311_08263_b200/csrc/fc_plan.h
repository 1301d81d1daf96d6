// Integer arithmetic of the launch plans and of the waits, without CUDA types (the tests compile it with the host compiler).
#pragma once

#ifdef __CUDACC__
#define FC_HD __host__ __device__ inline
#else
#define FC_HD inline
#endif

namespace fc {

// A ring of `stages` stages into which `issued` copies have been requested, copy j into stage j % stages: the parity of the phase that
// the last copy into `stage` completes (stage < issued).
FC_HD unsigned int last_copy_parity(int issued, int stages, int stage) { return (unsigned int)((issued - 1 - stage) / stages) & 1u; }

}  // namespace fc
