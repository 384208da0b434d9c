// State of a conjugate-gradient solve that runs on the device (krr.cu).
#pragma once

#if defined(__CUDACC__)
#define HDF_CG_FN __host__ __device__ inline
#else
#define HDF_CG_FN inline
#endif

namespace hdf {

constexpr int kCgRunning = 0x7fffffff;

// Iteration it reads rz[(it - 1) & 1] and writes rz[it & 1].
struct CgState {
    double rz[2];
    double nb, rtol;             // norm of the right-hand side
    double res;                  // relative residual after iteration `it`
    int it, bad;                 // bad: p . q <= 0
    int last;                    // the last iteration, kCgRunning until it is known
};

// Whether a kernel of iteration it returns at once.  Kernels of iteration it write it into `last` and
// nothing smaller, while blocks of the same launch are still starting: both values mean "go on" for
// that launch, so every thread of it decides alike (a flag that the launch itself sets would let some
// threads of a block leave and the others wait for them at a barrier).
HDF_CG_FN bool cg_past_end(int last, int it) { return last < it; }

}  // namespace hdf
