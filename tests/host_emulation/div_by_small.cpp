// Host build of the op graph's division by a spacing, div_by(v, h, 1/h), on values so
// small that the remainder of the product is not representable, subnormal ones
// included: within two units in the last place of v / h (in units of the smallest
// subnormal where the quotient is one).  From the size that the comment at div_by
// states on, the division's own bits.  Exit status: whether a value is outside.
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#undef __global__
#undef __device__
#undef __host__
#undef __forceinline__
#undef __launch_bounds__
#undef __shared__
#define __global__
#define __device__
#define __host__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __shared__ static
#define __syncthreads()
uint3 blockIdx, threadIdx;
dim3 blockDim, gridDim;
static inline float __fdividef(float a, float b) { return a / b; }
using std::fabs;
using std::fma;
#include "../../paper_2405_02483_gb300/csrc/graph_kernels.cuh"
using namespace stg;


template <typename T>
static int check(int lo, int hi, int exact_from) {
  std::mt19937_64 rng(9);
  std::uniform_real_distribution<double> e(lo, hi), m(1.0, 2.0), s(std::log(1e-5), std::log(1e3));
  double worst = 0;
  long long bad = 0;
  for (int i = 0; i < 4000000; ++i) {
    const T h = (T)std::exp(s(rng));
    const int ex = (int)std::floor(e(rng));
    const T v = std::ldexp((T)((i & 1 ? -1 : 1) * m(rng)), ex);
    const T q = div_by<T>(v, h, (T)1 / h), w = v / h;
    if (!std::isfinite(w)) continue;
    const T ulp = std::nextafter(std::fabs(w), (T)INFINITY) - std::fabs(w);
    worst = std::max(worst, (double)(std::fabs((long double)q - (long double)w) / (long double)ulp));
    if (ex >= exact_from) bad += !(q == w);
  }
  printf("FP%d: %.2f units at most, %lld differing where exact\n", (int)(8 * sizeof(T)), worst, bad);
  return worst > 2.0 || bad > 0;
}

int main() { return check<float>(-149, -80, -102) + check<double>(-1074, -900, -966); }
