// Host build of the op graph's division by a spacing: div_by(v, h, 1/h) equals
// v / h bit for bit over random values and spacings, and returns what the
// division returns for zeros, infinities, NaN and overflows.  Exit status: the
// number of differing values.
#include <cuda_runtime.h>
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
static long long check(double lo, double hi) {
  std::mt19937_64 rng(5);
  std::uniform_real_distribution<double> e(lo, hi), m(1.0, 2.0), s(std::log(1e-5), std::log(1e3));
  long long bad = 0;
  auto one = [&](T v, T h) {
    const T a = div_by<T>(v, h, (T)1 / h), b = v / h;
    bad += !(std::memcmp(&a, &b, sizeof(T)) == 0 || (a != a && b != b));
  };
  for (int i = 0; i < 4000000; ++i)
    one((T)((i & 1 ? -1 : 1) * m(rng) * std::exp2(e(rng))), (T)std::exp(s(rng)));
  const T inf = (T)INFINITY, big = sizeof(T) == 4 ? (T)3e38 : (T)1e308;
  for (T h : {(T)0.1, (T)(1.0 / 3.0), (T)7.5, (T)1})
    for (T v : {(T)0, -(T)0, inf, -inf, (T)NAN, big, -big}) one(v, h);
  return bad;
}

int main() {
  const long long f = check<float>(-60, 60), d = check<double>(-400, 400);
  printf("FP32 %lld differing, FP64 %lld differing\n", f, d);
  return f || d;
}
