// Shared device helpers of libstagger: mesh geometry, periodic indexing,
// the staggered operator weights of eqs. (deriv)/(interp), and error macros.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/stagger.h"

namespace stg {

// Interpolation weights, eq. (interpcoef): a = 1/2 - b - c.
#define STG_IA (150.0 / 256.0)
#define STG_IB (-25.0 / 256.0)
#define STG_IC (3.0 / 256.0)
// Derivative weights, eq. (derivcoef): c = 3/640, b = -25/384, a = 1 - 3b - 5c.
#define STG_DA (225.0 / 192.0)
#define STG_DB (-25.0 / 384.0)
#define STG_DC (3.0 / 640.0)

// Low-storage RK3 constants, eq. (tconst), as printed.
static const double RK_ALPHA[3] = {0.0, -0.641874, -1.31021};
static const double RK_BETA[3] = {0.46173, 0.924087, 0.390614};

struct Geo {
  int nx, ny, nz;
  long long sy;   // stride of y (= nx)
  long long sz;   // stride of z (= nx*ny)
  long long n;    // cells
};

inline Geo make_geo(int nx, int ny, int nz) {
  Geo g;
  g.nx = nx; g.ny = ny; g.nz = nz;
  g.sy = nx; g.sz = (long long)nx * ny; g.n = g.sz * nz;
  return g;
}

// Periodic wrap of j into [0, n).  Fast path for the usual |offset| < n.
__host__ __device__ __forceinline__ int wrap(int j, int n) {
  if (j >= 0 && j < n) return j;
  if (j < 0 && j >= -n) return j + n;
  if (j >= n && j < 2 * n) return j - n;
  j %= n;
  return j < 0 ? j + n : j;
}

// Linear index of (i+di, j+dj, k+dk) with periodic wrap.
__host__ __device__ __forceinline__ long long lin(const Geo& g, int i, int j, int k) {
  return (long long)k * g.sz + (long long)j * g.sy + i;
}

// Programmatic dependent launch.  A kernel launched by launch_dep may be put on
// the SMs while the one before it in the stream drains; dep_wait, the first
// thing it does, returns once that kernel has finished and its writes are
// visible, and only then lets the next kernel be put on the SMs (so a kernel
// never starts before the one two places ahead of it has finished, and the L1
// invalidation at its start drops whatever that one had cached).  It returns 0;
// the cell index of a thread is formed with it, because a read-only load whose
// address did not depend on the wait could be scheduled above it.  Every kernel
// that launch_dep launches calls it; in a plain launch it does nothing.
// A 131 x 97 x 75 right-hand side of 13 launches takes 397 us so, 422 without.
// Under stream capture the launches are plain: a CUDA graph of programmatic
// edges replays slower than one of full dependencies (64^3 step 246 against 220
// us, 32^3 FP64 adjoint 2963 against 2617).
__device__ __forceinline__ int dep_wait() {
  int zero = 0;
#ifdef __CUDA_ARCH__
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(zero)::"memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
  return zero;
}
#ifdef __CUDACC__   // (a host build brings launch and launch_dep of its own)
template <class... P, class... A>
inline void launch(void (*kern)(P...), dim3 grid, dim3 block, cudaStream_t s, A&&... args) {
  kern<<<grid, block, 0, s>>>(static_cast<P>(args)...);
}
template <class... P, class... A>
inline void launch_dep(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       A&&... args) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cap);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}
#endif

// The status of a failed device allocation, whose error the next check of the
// launches must not report.
inline int no_memory() {
  cudaGetLastError();
  return STAGGER_EOOM;
}

// Grid and parameter checks of stagger_create (STAGGER_OK or STAGGER_EINVAL).
int validate_inputs(const stagger_grid* g, const stagger_params* p);

}  // namespace stg

#define STG_CUDA_OK(call)                                   \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) { return STAGGER_ECUDA; }        \
  } while (0)
