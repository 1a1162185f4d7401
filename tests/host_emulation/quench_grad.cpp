// Host build of the quench's ratio q and its derivatives (q_val): the same bits as the
// chain rule written out with one division for each quotient, a zero stress (whose
// den^2 would underflow) included.  Exit status: the number of differing values.
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
static long long check() {
  std::mt19937_64 rng(3);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  long long bad = 0;
  auto s = [](T a) { return (T)((a > 0) - (a < 0)); };
  for (int i = 0; i < 200000; ++i) {
    T t[3];
    for (T& x : t) x = i < 8 ? (T)0 : (T)(U(rng) * (i % 3 ? 1.0 : 1e-6));
    const T iq = (T)1 / (T)8, eps = i & 1 ? (T)1e-4 : (T)-1;
    T dq[3];
    const T q = q_val<T>(t[0], t[1], t[2], iq, eps, dq);
    const T d2 = (t[2] - (T)2 * t[1]) + t[0], a2 = fabs(d2);
    const T m0 = std::max(fabs(t[0]), fabs(t[1])), m = std::max(m0, fabs(t[2]));
    const T M = eps < 0 ? m : fabs(t[1]) + eps * m, den = (M + a2 * iq) + (T)1e-30;
    const T ratio = a2 / den, qd = ratio / den, da = (T)1 / den - iq * qd;
    // the weights of |T| in the maximum: an even split on ties, the inner pair first
    const T a = fabs(t[0]), b = fabs(t[1]), c = fabs(t[2]);
    const T wi = m0 > c ? (T)1 : m0 == c ? (T)0.5 : (T)0, wa = a > b ? (T)1 : a == b ? (T)0.5 : (T)0;
    const T w[3] = {wi * wa, wi * ((T)1 - wa), (T)1 - wi};
    const T cM = eps < 0 ? (T)1 : eps, cP = eps < 0 ? (T)0 : (T)1;
    for (int k = 0; k < 3; ++k) {
      const T g = da * s(d2) * (k == 1 ? (T)-2 : (T)1) - qd * (cM * w[k] + (k == 1 ? cP : (T)0)) * s(t[k]);
      bad += !(g == dq[k]);
    }
    bad += !(q == ratio);
  }
  return bad;
}

int main() {
  const long long f = check<float>(), d = check<double>();
  printf("FP32 %lld differing, FP64 %lld differing\n", f, d);
  return f || d;
}
