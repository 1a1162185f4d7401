// Op-graph kernels (see graph.cuh): the forward and the hand-written
// transpose (vector-Jacobian) kernel of every primitive, as templates over the
// sweep's precision.  Included by the executor (graph.cu) and by the C ABI
// (api.cu, for the 16-byte access helpers of its RK combinations); plain C++
// apart from the CUDA qualifiers, so that a host build can run them too.
#pragma once

#include <math.h>

#include "graph.cuh"

namespace stg {

// The launch shape of the one-node kernels (threads along x, y, z).
#ifndef GBX
#define GBX 32
#endif
#ifndef GBY
#define GBY 2
#endif
#ifndef GBZ
#define GBZ 4
#endif
#define GZU 1   // planes a thread of the one-node kernels takes

// Roundings that do not depend on how the compiler contracts: the product a b
// rounded, and a b + c rounded once (the host build rounds twice, like the graph of
// one node per primitive it is compared with).  The reverse takes the branches of
// max and |.| at these values, so a last bit can route a cell's gradient elsewhere.
template <typename T>
__device__ __forceinline__ T mul_rn(T a, T b) {
#ifdef __CUDA_ARCH__
  if constexpr (sizeof(T) == sizeof(float)) return __fmul_rn(a, b);
  else return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
template <typename T>
__device__ __forceinline__ T mad(T a, T b, T c) {
#ifdef __CUDA_ARCH__
  return fma(a, b, c);
#else
  return a * b + c;
#endif
}

// The cells of a thread.  W 4: the consecutive x-cells i .. i + 3 of row (j, k) (needs
// nx a multiple of 4 and 16-byte aligned arrays: each tap is then one 16-byte load and
// the index work is shared by four cells).  W 1: one cell.  W 3, for rows of other
// lengths: the cells (i, j) of planes k, k + blockDim.z and k + 2 blockDim.z, which share
// the offsets of the taps along x and y and the reads of the node's constants (indexed
// reads of the launch's parameters: with one cell a thread the unit that serves them is
// 69% busy and the rest of the SM waits on it); a cell past the last plane is the
// first one again.  FP32 adjoint step, viscous, one plane / three: 90^3 7.64 / 5.02
// ms, 199 x 150 x 150 41.4 / 25.2, 251 x 250 x 250 140 / 75.8 (one launch a node on
// four streams: 6.0, 27.8 and 87.8; two planes 5.59, 27.2, 89.6).  Every cell takes the
// same arithmetic, so the values do not depend on W.
struct GCell {
  int i, j, k;
  int idx;       // (a box has less than 2^31 cells)
  int dk[4];     // planes from k to each cell (0 for W 4), the most of them,
  int dmax;
  int off[4];    // and cells from idx
};

template <int W>
__device__ __forceinline__ bool gcell_at(GCell& c, int kb, const Geo& g) {
  constexpr int WX = W == 4 ? 4 : 1, WZ = W / WX;
  c.i = WX * (int)(blockIdx.x * blockDim.x + threadIdx.x + dep_wait());
  c.j = blockIdx.y * blockDim.y + threadIdx.y;
  c.k = kb * (WZ * (int)blockDim.z) + (int)threadIdx.z;
  if (c.i >= g.nx || c.j >= g.ny || c.k >= g.nz) return false;
  c.idx = c.k * (int)g.sz + c.j * (int)g.sy + c.i;
  c.dmax = 0;
#pragma unroll
  for (int l = 0; l < W; ++l) {
    c.dk[l] = WZ > 1 && c.k + l * (int)blockDim.z < g.nz ? l * (int)blockDim.z : 0;
    c.off[l] = c.dk[l] * (int)g.sz;
    c.dmax = c.dk[l] > c.dmax ? c.dk[l] : c.dmax;
  }
  return true;
}
template <int W>
__device__ __forceinline__ bool gcell(GCell& c, const Geo& g) {
  return gcell_at<W>(c, (int)blockIdx.z, g);
}

// A node's constant in the sweep's precision: the FP32 kernels read the
// float copies made when the graph was built (a conversion from double, or
// a double comparison, runs on the FP64 pipe, which is narrow on this GPU).
template <typename T>
__device__ __forceinline__ T kc(double d, float f) {
  if constexpr (sizeof(T) == sizeof(float)) return f;
  else return d;
}

// W consecutive elements i .. as 16-byte loads and stores (W = 4) or one.
template <typename T>
__device__ __forceinline__ void ld4(const T* p, long long i, T (&v)[4]) {
  if constexpr (sizeof(T) == sizeof(float)) {
    const float4 x = *reinterpret_cast<const float4*>(p + i);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  } else {
    const double2 x = *reinterpret_cast<const double2*>(p + i);
    const double2 y = *reinterpret_cast<const double2*>(p + i + 2);
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
  }
}
template <typename T>
__device__ __forceinline__ void st4(T* p, long long i, const T (&v)[4]) {
  if constexpr (sizeof(T) == sizeof(float)) {
    *reinterpret_cast<float4*>(p + i) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    *reinterpret_cast<double2*>(p + i) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + i + 2) = make_double2(v[2], v[3]);
  }
}
// The thread's cells, o elements further on.
template <typename T, int W>
__device__ __forceinline__ void ldw(const T* p, const GCell& c, int o, T (&v)[W]) {
  if constexpr (W == 4) ld4(p, c.idx + o, v);
  else
#pragma unroll
    for (int l = 0; l < W; ++l) v[l] = p[c.idx + o + c.off[l]];
}
template <typename T, int W>
__device__ __forceinline__ void stw(T* p, const GCell& c, const T (&v)[W]) {
  if constexpr (W == 4) st4(p, c.idx, v);
  else
#pragma unroll
    for (int l = 0; l < W; ++l) p[c.idx + c.off[l]] = v[l];
}

// Stride, position and length of an axis.
struct GAxis {
  int st, pos, n;
};
__device__ __forceinline__ GAxis gaxis(const GCell& c, int axis, const Geo& g) {
  return {axis == 0 ? 1 : axis == 1 ? (int)g.sy : (int)g.sz, axis == 0 ? c.i : axis == 1 ? c.j : c.k,
          axis == 0 ? g.nx : axis == 1 ? g.ny : g.nz};
}
// f at offset o along the axis from each of the thread's cells, with the wrapped index.
template <int W, typename T>
__device__ __forceinline__ void tap_wrap(const T* f, const GCell& c, int axis, const GAxis& a, int o,
                                         T (&v)[W]) {
  if (W > 1 && W < 4 && axis == 2) {   // the cells wrap on their own
#pragma unroll
    for (int l = 0; l < W; ++l) {
      const int q = a.pos + c.dk[l];
      v[l] = f[c.idx + c.off[l] + (wrap(q + o, a.n) - q) * a.st];
    }
  } else {
    ldw<T, W>(f, c, (wrap(a.pos + o, a.n) - a.pos) * a.st, v);
  }
}
// Whether the offsets lo .. hi from each of the thread's cells stay in the box.
template <int W>
__device__ __forceinline__ bool inner(const GCell& c, int axis, const GAxis& a, int lo, int hi) {
  return a.pos + lo >= 0 && a.pos + (W > 1 && W < 4 && axis == 2 ? c.dmax : 0) + hi < a.n;
}

// t[o + K][l]: f at cell (i + l, j, k) + o e_axis, o = -K .. K (K <= 3):
// plain strides away from the periodic seam, wrapped indices next to it.
template <int K, int W, typename T>
__device__ __forceinline__ void taps(const T* f, const GCell& c, int axis, const Geo& g,
                                     T (&t)[2 * K + 1][W]) {
  if (W == 4 && axis == 0) {
    T L[W], M[W], R[W];
    ldw<T, W>(f, c, wrap(c.i - 4, g.nx) - c.i, L);
    ldw<T, W>(f, c, 0, M);
    ldw<T, W>(f, c, wrap(c.i + 4, g.nx) - c.i, R);
#pragma unroll
    for (int o = -K; o <= K; ++o)
#pragma unroll
      for (int l = 0; l < W; ++l) {
        const int q = 4 + l + o;   // in the 12-cell window i - 4 .. i + 7
        t[o + K][l] = q < 4 ? L[q & (W - 1)] : q < 8 ? M[(q - 4) & (W - 1)] : R[(q - 8) & (W - 1)];
      }
  } else {
    const GAxis a = gaxis(c, axis, g);
    if (W == 1 || W == 4) {
      const bool in = inner<W>(c, axis, a, -K, K);
#pragma unroll
      for (int o = -K; o <= K; ++o)
        ldw<T, W>(f, c, (in ? o : wrap(a.pos + o, a.n) - a.pos) * a.st, t[o + K]);
    } else if (inner<W>(c, axis, a, -K, K)) {
#pragma unroll
      for (int o = -K; o <= K; ++o) ldw<T, W>(f, c, o * a.st, t[o + K]);
    } else {
#pragma unroll
      for (int o = -K; o <= K; ++o) tap_wrap<W>(f, c, axis, a, o, t[o + K]);
    }
  }
}

// v[l]: f at cell (i + l, j, k) + o e_axis; with W = 4 along x |o| <= 3.
template <int W, typename T>
__device__ __forceinline__ void tap(const T* f, const GCell& c, int axis, int o, const Geo& g,
                                    T (&v)[W]) {
  if (W == 4 && axis == 0) {
    T t[7][W];
    taps<3, W>(f, c, 0, g, t);
#pragma unroll
    for (int l = 0; l < W; ++l)
      v[l] = o == -1 ? t[2][l] : o == 1 ? t[4][l] : o == 0 ? t[3][l] : o == -2 ? t[1][l]
           : o == 2 ? t[5][l] : o == -3 ? t[0][l] : t[6][l];
  } else {
    tap_wrap<W>(f, c, axis, gaxis(c, axis, g), o, v);
  }
}

// The six taps of a stencil: t[q][l] is f at cell (i + l, j, k) + (q - 2 - dn) e_axis
// (c - 2 .. c + 3 for the upward kinds, c - 3 .. c + 2 for the downward ones).
template <int W, typename T>
__device__ __forceinline__ void taps6(const T* f, const GCell& c, int axis, int dn, const Geo& g,
                                      T (&t)[6][W]) {
  if (W == 4 && axis == 0) {
    T w[3][W];   // the 12-cell window i - 4 .. i + 7
    ldw<T, W>(f, c, wrap(c.i - 4, g.nx) - c.i, w[0]);
    ldw<T, W>(f, c, 0, w[1]);
    ldw<T, W>(f, c, wrap(c.i + 4, g.nx) - c.i, w[2]);
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
      for (int l = 0; l < W; ++l) {
        const int u = 2 + q + l, d = 1 + q + l;
        t[q][l] = dn ? w[d / 4][d & (W - 1)] : w[u / 4][u & (W - 1)];
      }
  } else {
    const GAxis a = gaxis(c, axis, g);
    const int lo = -2 - dn;
    if (inner<W>(c, axis, a, lo, lo + 5)) {
#pragma unroll
      for (int q = 0; q < 6; ++q) ldw<T, W>(f, c, (lo + q) * a.st, t[q]);
    } else {
#pragma unroll
      for (int q = 0; q < 6; ++q) tap_wrap<W>(f, c, axis, a, lo + q, t[q]);
    }
  }
}

// A node's first and second stencil's spacing and its reciprocal.
template <typename T> struct Spc { T h, ih; };
template <typename T> __device__ __forceinline__ Spc<T> sp1(const GNode& nd) {
  return {kc<T>(nd.c0, nd.f0), kc<T>(nd.ic0, nd.fi0)};
}
template <typename T> __device__ __forceinline__ Spc<T> sp2(const GNode& nd) {
  return {kc<T>(nd.h2, nd.fh2), kc<T>(nd.ih2, nd.fih2)};
}

// v / h from the rounded reciprocal ih of h, rounded as a division rounds it while the
// remainder of the product can be represented (|v| above 2e-31 in FP32, 2e-291 in FP64;
// within two units in the last place below): the product and one correction by its
// exact remainder (Markstein, IBM J. Res. Dev. 34, 1990).  The product itself where
// it is exact (a zero keeps its sign) or where it or the remainder is not finite.
template <typename T>
__device__ __forceinline__ T div_by(T v, T h, T ih) {
  const T q = v * ih;
  const T r = fma(-q, h, v);
  const T most = sizeof(T) == 4 ? (T)3.4028235e38 : (T)1.7976931348623157e308;
  return r != (T)0 && fabs(r) <= most ? fma(r, ih, q) : q;
}

// A stencil (kind, spacing h, its reciprocal ih) from its six taps: up/dn are eq.
// (interp) to i+1/2 and i-1/2, ddup/dddn eq. (deriv) to i+1/2 and i-1/2.  One
// form for the four kinds, sums for the interpolations and differences for the
// derivatives by the factor s (the kind is known at run time only, and a
// switch over four forms was a third of the sweeps' instructions).  The division
// by the spacing was half the work of an FP64 derivative on the narrow FP64 pipe.
template <int W, typename T>
__device__ __forceinline__ void st_comb(int kind, const Spc<T>& sp, const T (&t)[6][W], T (&v)[W]) {
  const bool d = kind >= ST_DDUP;
  const T s = d ? (T)-1 : (T)1;
  const T a = d ? (T)STG_DA : (T)STG_IA, b = d ? (T)STG_DB : (T)STG_IB, e = d ? (T)STG_DC : (T)STG_IC;
#pragma unroll
  for (int l = 0; l < W; ++l) {
    const T x = a * (t[3][l] + s * t[2][l]) + b * (t[4][l] + s * t[1][l]) + e * (t[5][l] + s * t[0][l]);
    v[l] = d ? div_by(x, sp.h, sp.ih) : x;
  }
}
__device__ __forceinline__ int st_down(int kind) { return kind & 1; }   // ST_DN, ST_DDDN
// The stencil (kind, axis, spacing) of f at the thread's cells.
template <int W, typename T>
__device__ __forceinline__ void stencil(const T* f, const GCell& c, int axis, int kind,
                                        const Spc<T>& sp, const Geo& g, T (&v)[W]) {
  T t[6][W];
  taps6<W>(f, c, axis, st_down(kind), g, t);
  st_comb<W>(kind, sp, t, v);
}
// The stencil of the product f (h - s): one tap array live, the product
// formed as its second factor arrives.
template <int W, typename T>
__device__ __forceinline__ void stencil_mul(const T* f, const T* h, T s, const GCell& c, int axis,
                                            int kind, const Spc<T>& sp, const Geo& g, T (&v)[W]) {
  T t[6][W];
  taps6<W>(f, c, axis, st_down(kind), g, t);
  {
    T u[6][W];
    taps6<W>(h, c, axis, st_down(kind), g, u);
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
      for (int l = 0; l < W; ++l) t[q][l] = mul_rn(t[q][l], u[q][l] - s);
  }
  st_comb<W>(kind, sp, t, v);
}

// Transposed kind and sign of a stencil: up^T = dn, dn^T = up, ddup^T =
// -dddn, dddn^T = -ddup (periodic summation by parts).
__device__ __forceinline__ int st_transpose(int kind) {
  return kind == ST_UP ? ST_DN : kind == ST_DN ? ST_UP : kind == ST_DDUP ? ST_DDDN : ST_DDUP;
}
__device__ __forceinline__ bool st_negates(int kind) { return kind == ST_DDUP || kind == ST_DDDN; }

// ---------------------------------------------------------------------------
// Quench, eq. (quench) with reading R8, as one node: out = T min(fac, qlim),
// fac = the max over the node's axes of max3 along the axis of
// q = |D2 T| / ((M + |D2 T| / qmax) + 1e-30), D2 T = T(+1) - 2 T + T(-1) and
// M = |T| + eps max3 |T| (eps = c2 >= 0), or M = max3 |T| (c2 < 0).  Its
// transpose follows the rules of the primitive nodes it stands for: a max
// splits the gradient evenly on a tie (pairwise, the inner pair first),
// |x|' = sign x with sign 0 = 0, the clamp passes the gradient where
// fac <= qlim.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void max_w(T a, T b, T& wa, T& wb) {
  wa = a > b ? (T)1 : (a == b ? (T)0.5 : (T)0);
  wb = b > a ? (T)1 : (a == b ? (T)0.5 : (T)0);
}
template <typename T>
__device__ __forceinline__ T sgn(T a) {
  return a > (T)0 ? (T)1 : (a < (T)0 ? (T)-1 : (T)0);
}

// The quench's divisions: the fast intrinsic in FP32 (within 2 ulp; the
// divisors are >= 1e-30 and far below 2^126), IEEE division in FP64.
template <typename T>
__device__ __forceinline__ T qdiv(T a, T b) {
  if constexpr (sizeof(T) == sizeof(float)) return __fdividef(a, b);
  else return a / b;
}

// q at z = c + s e_ax from T at z - 1, z, z + 1 (vm, v0, vp), and (dq) its
// derivatives with respect to those (through D2 T and through M).
template <typename T>
__device__ __forceinline__ T q_val(T vm, T v0, T vp, T iq, T eps, T* dq) {
  const T d2 = (vp - (T)2 * v0) + vm, a2 = fabs(d2);
  const T am = fabs(vm), a0 = fabs(v0), ap = fabs(vp);
  const T inner = am >= a0 ? am : a0;
  const T M3 = inner >= ap ? inner : ap;
  // M = cM max3|T| + cP |T|.
  const T cM = eps < (T)0 ? (T)1 : eps, cP = eps < (T)0 ? (T)0 : (T)1;
  const T M = eps < (T)0 ? M3 : a0 + eps * M3;
  const T den = (M + a2 * iq) + (T)1e-30;
  const T q = qdiv(a2, den);
  if (dq) {
    T wim, wi0, woi, wop;
    max_w(am, a0, wim, wi0);
    max_w(inner, ap, woi, wop);
    // a2 / den^2 as q / den, one rounding: den^2 underflows in FP32 where T and
    // D2 T are both zero (den = 1e-30), and 0 / 0 would poison the cotangent.
    const T qd = qdiv(q, den);
    const T dq_da2 = qdiv((T)1, den) - iq * qd;
    const T dq_dM = -qd;
    const T sd = sgn(d2);
    dq[0] = dq_da2 * sd + dq_dM * (cM * (woi * wim)) * sgn(vm);
    dq[1] = dq_da2 * sd * (T)-2 + dq_dM * (cM * (woi * wi0) + cP) * sgn(v0);
    dq[2] = dq_da2 * sd + dq_dM * (cM * wop) * sgn(vp);
  }
  return q;
}
// fac at c, and (when wq) the weights of the three q of each axis in fac:
// wq[3 t + p + 1] for axis t and position p.  qf(t, ax, s) is q at
// c + s e_ax (axis slot t): formed from T, or read from the transpose's
// per-cell q arrays.
template <typename T, class QF>
__device__ __forceinline__ T quench_fac(QF qf, int a0, int a1, T* wq) {
  T m[2] = {0, 0}, w[2][3];
  for (int t = 0; t < 2; ++t) {
    const int ax = t == 0 ? a0 : a1;
    if (ax < 0) continue;
    const T qm = qf(t, ax, -1), q0 = qf(t, ax, 0), qp = qf(t, ax, 1);
    const T inner = qm >= q0 ? qm : q0;
    m[t] = inner >= qp ? inner : qp;
    T wim, wi0, woi, wop;
    max_w(qm, q0, wim, wi0);
    max_w(inner, qp, woi, wop);
    w[t][0] = woi * wim;
    w[t][1] = woi * wi0;
    w[t][2] = wop;
  }
  T fac = m[0], wf0 = 1, wf1 = 0;
  if (a1 >= 0) {
    fac = m[0] >= m[1] ? m[0] : m[1];
    max_w(m[0], m[1], wf0, wf1);
  }
  if (wq)
    for (int p = 0; p < 3; ++p) {
      wq[p] = wf0 * w[0][p];
      wq[3 + p] = a1 >= 0 ? wf1 * w[1][p] : (T)0;
    }
  return fac;
}

// Transpose, q pass (per cell z, per axis slot t): q(z) and its derivatives
// with respect to T at z - 1, z, z + 1, into Q[(4 t + 0 .. 3) n + z], formed
// once here instead of at every tap of the two passes that follow.
template <typename T, int W>
__device__ __forceinline__ void quench_q(const GNode& nd, const T* A, T* Q, const GCell& c,
                                         const Geo& g) {
  const T iq = (T)1 / kc<T>(nd.c0, nd.f0), eps = kc<T>(nd.c2, nd.f2);
  for (int t = 0; t < 2; ++t) {
    const int ax = t == 0 ? nd.axis : nd.sk;
    if (ax < 0) continue;
    T ta[3][W], q[W], d0[W], d1[W], d2[W];
    taps<1, W>(A, c, ax, g, ta);
#pragma unroll
    for (int l = 0; l < W; ++l) {
      T dq[3];
      q[l] = q_val(ta[0][l], ta[1][l], ta[2][l], iq, eps, dq);
      d0[l] = dq[0];
      d1[l] = dq[1];
      d2[l] = dq[2];
    }
    stw<T, W>(Q + (long long)(4 * t) * g.n, c, q);
    stw<T, W>(Q + (long long)(4 * t + 1) * g.n, c, d0);
    stw<T, W>(Q + (long long)(4 * t + 2) * g.n, c, d1);
    stw<T, W>(Q + (long long)(4 * t + 3) * g.n, c, d2);
  }
}

// Transpose, first pass (per output cell y): S0 = gbar C (the product's own
// term) and S[1 + 3 t + p + 1] = gbar T dC/dfac dfac/dq, the cotangent each
// q of axis t at position p receives from y.
template <typename T, int W>
__device__ __forceinline__ void quench_b1(const GNode& nd, const T* A, const T* Q, const T* gout,
                                          T* S, const GCell& c, const Geo& g) {
  const T qlim = kc<T>(nd.c1, nd.f1);
  T tq[2][3][W];   // q at offsets -1 .. 1 along each axis slot
  taps<1, W>(Q, c, nd.axis, g, tq[0]);
  if (nd.sk >= 0) taps<1, W>(Q + 4 * g.n, c, nd.sk, g, tq[1]);
  T a[W], gg[W], s0[W], sw[6][W];
  ldw<T, W>(A, c, 0, a);
  ldw<T, W>(gout, c, 0, gg);
#pragma unroll
  for (int l = 0; l < W; ++l) {
    T wq[6];
    const T fac = quench_fac<T>([&](int t, int, int s) { return tq[t][s + 1][l]; }, nd.axis,
                                nd.sk, wq);
    const T C = fac > qlim ? qlim : fac;
    const T dC = fac <= qlim ? (T)1 : (T)0;
    const T base = gg[l] * a[l] * dC;
    s0[l] = gg[l] * C;
#pragma unroll
    for (int j = 0; j < 6; ++j) sw[j][l] = base * wq[j];
  }
  stw<T, W>(S, c, s0);
#pragma unroll
  for (int j = 0; j < 6; ++j)
    if (j < 3 || nd.sk >= 0) stw<T, W>(S + (long long)(1 + j) * g.n, c, sw[j]);
}

// Transpose, second pass (per input cell x): Tbar(x) = S0(x) + the sum over
// the axes and the three q positions z = x + r e_a whose stencils hold x of
// qbar(z) dq(z)/dT(x), qbar(z) = sum_p S[.. p](z - p e_a).  Reads Q and S only.
template <typename T, int W>
__device__ __forceinline__ void quench_b3(const GNode& nd, const T* Q, const T* S, const GCell& c,
                                          const Geo& g, T (&acc)[W]) {
  ldw<T, W>(S, c, 0, acc);
  for (int t = 0; t < 2; ++t) {
    const int ax = t == 0 ? nd.axis : nd.sk;
    if (ax < 0) continue;
    T ts[3][5][W];   // S of q position p = -1 .. 1 at offsets -2 .. 2
#pragma unroll
    for (int p = 0; p < 3; ++p) taps<2, W>(S + (long long)(1 + 3 * t + p) * g.n, c, ax, g, ts[p]);
    T td[3][W];      // d q(z) / d T at its tap 1 - r, z at offsets r = -1 .. 1
#pragma unroll
    for (int r = -1; r <= 1; ++r)
      tap<W>(Q + (long long)(4 * t + 2 - r) * g.n, c, ax, r, g, td[r + 1]);
#pragma unroll
    for (int r = -1; r <= 1; ++r)
#pragma unroll
      for (int l = 0; l < W; ++l) {
        T qbar = 0;
#pragma unroll
        for (int p = -1; p <= 1; ++p) qbar += ts[p + 1][r - p + 2][l];
        acc[l] += qbar * td[r + 1][l];
      }
  }
}

// y = st (op) b of a G_STBIN node (side 1: b first).
template <typename T>
__device__ __forceinline__ T stbin_val(const GNode& nd, T st, T b) {
  if (nd.iop == G_MUL) return st * b;
  if (nd.iop == G_ADD) return nd.side ? b + st : st + b;
  return nd.side ? b - st : st - b;     // G_SUB
}

// The ops whose value at a cell reads only that cell of their operands.
__host__ __device__ __forceinline__ bool pointwise_op(int op) {
  constexpr unsigned mask = 1u << G_ADD | 1u << G_SUB | 1u << G_MUL | 1u << G_DIV | 1u << G_MAX |
                            1u << G_EXP | 1u << G_LOG | 1u << G_LOG1P | 1u << G_SQRT |
                            1u << G_ABS | 1u << G_AXPB | 1u << G_CLAMPMIN | 1u << G_CLAMPMAX |
                            1u << G_STEP | 1u << G_CONST;
  return (mask >> op) & 1u;
}

// A pointwise op's value from its operands' values a, b at the cell.
template <typename T>
__device__ __forceinline__ T pw_value(int op, const GNode& nd, T a, T b) {
  switch (op) {
    case G_ADD: return a + b;
    case G_SUB: return a - b;
    case G_MUL: return a * b;
    case G_DIV: return a / b;
    case G_MAX: return a >= b ? a : b;
    case G_EXP: return exp(a);
    case G_LOG: return log(a);
    case G_LOG1P: return log1p(a);
    case G_SQRT: return sqrt(a);
    case G_ABS: return fabs(a);
    case G_AXPB: return kc<T>(nd.c0, nd.f0) * a + kc<T>(nd.c1, nd.f1);
    case G_CLAMPMIN: return a < kc<T>(nd.c0, nd.f0) ? kc<T>(nd.c0, nd.f0) : a;
    case G_CLAMPMAX: return a > kc<T>(nd.c0, nd.f0) ? kc<T>(nd.c0, nd.f0) : a;
    case G_STEP: return a > kc<T>(nd.c0, nd.f0) ? (T)1 : (T)0;
    default: return kc<T>(nd.c0, nd.f0);  // G_CONST
  }
}

// The folded sum and the epilogue of a node's value v (C's value cv).
template <typename T>
__device__ __forceinline__ T finish(const GNode& nd, T v, T cv) {
  if (nd.pop) v = nd.pop == 1 ? v + cv : nd.pop == 2 ? v - cv : cv - v;
  return nd.ep ? kc<T>(nd.ps, nd.fps) * v + kc<T>(nd.pt, nd.fpt) : v;
}

// The value of a node (every op but G_INPUT and G_PMEAN) at the thread's cells.
template <typename T, int W>
__device__ __forceinline__ void node_value(int op, const GNode& nd, const T* A, const T* B,
                                           const T* mesh, const GCell& c, const Geo& g,
                                           T (&r)[W]) {
  if (pointwise_op(op)) {
    T a[W] = {}, b[W] = {};
    if (A) ldw<T, W>(A, c, 0, a);
    if (B) ldw<T, W>(B, c, 0, b);
#pragma unroll
    for (int l = 0; l < W; ++l) r[l] = pw_value(op, nd, a[l], b[l]);
    return;
  }
  switch (op) {
    case G_STENCIL: stencil<W>(A, c, nd.axis, nd.sk, sp1<T>(nd), g, r); break;
    case G_STEXP:
      stencil<W>(A, c, nd.axis, nd.sk, sp1<T>(nd), g, r);
#pragma unroll
      for (int l = 0; l < W; ++l) r[l] = exp(r[l]);
      break;
    case G_STBIN: {
      T b[W];
      stencil<W>(A, c, nd.axis, nd.sk, sp1<T>(nd), g, r);
      ldw<T, W>(B, c, 0, b);
#pragma unroll
      for (int l = 0; l < W; ++l) r[l] = stbin_val(nd, r[l], b[l]);
      break;
    }
    case G_STMUL: stencil_mul<W>(A, B, (T)0, c, nd.axis, nd.sk, sp1<T>(nd), g, r); break;
    case G_ST2: {   // one after the other: one tap array live
      T s2[W];
      stencil<W>(A, c, nd.axis, nd.sk, sp1<T>(nd), g, r);
      stencil<W>(B, c, nd.axis2, nd.sk2, sp2<T>(nd), g, s2);
#pragma unroll
      for (int l = 0; l < W; ++l) r[l] = nd.iop == G_ADD ? r[l] + s2[l] : r[l] - s2[l];
      break;
    }
    case G_NB3: {
      T m[W], z[W], p[W];
      tap<W>(A, c, nd.axis, nd.sk, g, m);
      ldw<T, W>(A, c, 0, z);
      tap<W>(A, c, nd.axis, -nd.sk, g, p);
#pragma unroll
      for (int l = 0; l < W; ++l) {
        const T in = m[l] >= z[l] ? m[l] : z[l];
        r[l] = nd.iop == G_ADD ? (m[l] + z[l]) + p[l] : in >= p[l] ? in : p[l];
      }
      break;
    }
    case G_SHIFT: tap<W>(A, c, nd.axis, nd.sk, g, r); break;
    case G_QUENCH: {   // out = T min(fac, qlim)
      const T iq = (T)1 / kc<T>(nd.c0, nd.f0), qlim = kc<T>(nd.c1, nd.f1);
      const T eps = kc<T>(nd.c2, nd.f2);
      T ta[2][5][W];   // T at offsets -2 .. 2 along each axis slot
      taps<2, W>(A, c, nd.axis, g, ta[0]);
      if (nd.sk >= 0) taps<2, W>(A, c, nd.sk, g, ta[1]);
#pragma unroll
      for (int l = 0; l < W; ++l) {
        const T fac = quench_fac<T>(
            [&](int t, int, int s) {
              return q_val(ta[t][s + 1][l], ta[t][s + 2][l], ta[t][s + 3][l], iq, eps, (T*)nullptr);
            },
            nd.axis, nd.sk, (T*)nullptr);
        r[l] = ta[0][2][l] * (fac > qlim ? qlim : fac);
      }
      break;
    }
    default: {   // G_ZFIELD
#pragma unroll
      for (int l = 0; l < W; ++l) r[l] = mesh[(long long)nd.sk * g.nz + c.k + c.dk[l]];
    }
  }
}
// ... with its folded sum and epilogue, stored.
template <typename T, int W>
__device__ __forceinline__ void node_forward(int op, const GNode& nd, const T* A, const T* B,
                                             const T* C, T* out, const T* mesh, const GCell& c,
                                             const Geo& g) {
  T r[W], cv[W] = {};
  if (nd.pop) ldw<T, W>(C, c, 0, cv);
  if (op == G_MUL && nd.pop) {   // a b and its folded sum, rounded once
    T a[W], b[W];
    ldw<T, W>(A, c, 0, a);
    ldw<T, W>(B, c, 0, b);
#pragma unroll
    for (int l = 0; l < W; ++l) {
      const T v = mad(nd.pop == 3 ? -a[l] : a[l], b[l], nd.pop == 2 ? -cv[l] : cv[l]);
      r[l] = nd.ep ? kc<T>(nd.ps, nd.fps) * v + kc<T>(nd.pt, nd.fpt) : v;
    }
  } else {
    node_value<T, W>(op, nd, A, B, mesh, c, g, r);
#pragma unroll
    for (int l = 0; l < W; ++l) r[l] = finish(nd, r[l], cv[l]);
  }
  stw<T, W>(out, c, r);
}

// A pointwise op's cotangents of a and b from y = its value and gg = y's
// cotangent (before the folded sum's sign and the epilogue's factor, which
// the kernel applies; exp reads ps exp(a) = y - pt itself).
template <typename T>
__device__ __forceinline__ void pw_grad(int op, const GNode& nd, T a, T b, T y, T gg, T& ca,
                                        T& cb) {
  ca = 0;
  cb = 0;
  switch (op) {
    case G_ADD: ca = gg; cb = gg; break;
    case G_SUB: ca = gg; cb = -gg; break;
    case G_MUL: ca = gg * b; cb = gg * a; break;
    case G_DIV:
      ca = gg / b;
      cb = -gg * a / (b * b);
      break;
    case G_MAX:
      ca = a > b ? gg : (a == b ? gg / (T)2 : (T)0);
      cb = b > a ? gg : (a == b ? gg / (T)2 : (T)0);
      break;
    case G_EXP: ca = gg * (y - kc<T>(nd.pt, nd.fpt)); break;   // ps exp(a) = y - pt
    case G_LOG: ca = gg / a; break;
    case G_LOG1P: ca = gg / ((T)1 + a); break;
    case G_SQRT: ca = gg / ((T)2 * y); break;
    case G_ABS: ca = a > (T)0 ? gg : (a < (T)0 ? -gg : (T)0); break;
    case G_AXPB: ca = kc<T>(nd.c0, nd.f0) * gg; break;
    case G_CLAMPMIN: ca = a >= kc<T>(nd.c0, nd.f0) ? gg : (T)0; break;
    case G_CLAMPMAX: ca = a <= kc<T>(nd.c0, nd.f0) ? gg : (T)0; break;
    default: break;
  }
}

// What a node (operands' values A, B, its own value Y, its cotangent G) passes
// to one of its operands: role 0 to a, 1 to b, 2 to the folded sum's c, 3 G
// itself (an identity, or an array that already holds the contribution).
// Pointwise rules follow the usual subgradient choices: |x|' = sign(x) with
// sign(0) = 0; clamp passes the gradient where the bound holds with equality;
// max(a, b) splits it evenly on ties.
enum { R_A = 0, R_B, R_C, R_COPY };
template <typename T, int W>
__device__ __forceinline__ void pull(int op, int role, const GNode& nd, const T* A, const T* B,
                                     const T* Y, const T* G, const GCell& c, const Geo& g,
                                     T (&v)[W]) {
  // The factors of the epilogue and the folded sum: every transpose is linear
  // in G, and c's cotangent is +-ps G at the cell.
  const T sv = kc<T>(nd.ps, nd.fps) * (nd.pop == 3 ? (T)-1 : (T)1);
  if (role >= R_C) {
    const T sc = role == R_C ? kc<T>(nd.ps, nd.fps) * (nd.pop == 2 ? (T)-1 : (T)1) : (T)1;
    ldw<T, W>(G, c, 0, v);
#pragma unroll
    for (int l = 0; l < W; ++l) v[l] = sc * v[l];
    return;
  }
  if (pointwise_op(op)) {
    T a[W] = {}, b[W] = {}, y[W], gg[W];
    if (A) ldw<T, W>(A, c, 0, a);
    if (B) ldw<T, W>(B, c, 0, b);
    ldw<T, W>(Y, c, 0, y);
    ldw<T, W>(G, c, 0, gg);
#pragma unroll
    for (int l = 0; l < W; ++l) {
      T ca, cb;
      pw_grad(op, nd, a[l], b[l], y[l], gg[l], ca, cb);
      v[l] = role == R_A ? ca : cb;
    }
  } else {
    const int tk = st_transpose(nd.sk);
    bool ng = st_negates(nd.sk);
    if (op == G_STBIN && nd.iop == G_MUL) {
      // y = st(a) b
      if (role == R_A) {
        stencil_mul<W>(G, B, (T)0, c, nd.axis, tk, sp1<T>(nd), g, v);
      } else {
        T gg[W];
        stencil<W>(A, c, nd.axis, nd.sk, sp1<T>(nd), g, v);
        ldw<T, W>(G, c, 0, gg);
#pragma unroll
        for (int l = 0; l < W; ++l) v[l] = gg[l] * v[l];
        ng = false;
      }
    } else if (op == G_STBIN && role == R_B) {
      ldw<T, W>(G, c, 0, v);
      ng = nd.iop == G_SUB && !nd.side;                    // st - b
    } else if (op == G_STEXP) {
      // y = ps exp(st(a)) + pt: the stencil's transpose of g (y - pt), the
      // epilogue's factor included (it is in y).
      stencil_mul<W>(G, Y, kc<T>(nd.pt, nd.fpt), c, nd.axis, tk, sp1<T>(nd), g, v);
    } else if (op == G_NB3) {
      // Gather over the three outputs y = x - o, x, x + o (o = sk) that read x
      // as their a(y + o), a(y), a(y - o); a max passes g by the primitive
      // nodes' rule (an even split on a tie, the inner pair first).
      const int ax = nd.axis, o = nd.sk;
      T gm[W], g0[W], gp[W];
      tap<W>(G, c, ax, -o, g, gm);
      ldw<T, W>(G, c, 0, g0);
      tap<W>(G, c, ax, o, g, gp);
      if (nd.iop == G_ADD) {
#pragma unroll
        for (int l = 0; l < W; ++l) v[l] = (gm[l] + g0[l]) + gp[l];
      } else {
        T a0[W], am[W], am2[W], ap[W], ap2[W];
        ldw<T, W>(A, c, 0, a0);
        tap<W>(A, c, ax, -o, g, am);
        tap<W>(A, c, ax, -2 * o, g, am2);
        tap<W>(A, c, ax, o, g, ap);
        tap<W>(A, c, ax, 2 * o, g, ap2);
#pragma unroll
        for (int l = 0; l < W; ++l) {
          T wm, wz, wi, wp;
          max_w(a0[l], am[l], wm, wz);   // y = x - o: (a0 op am) op am2, x in the inner first slot
          max_w(a0[l] >= am[l] ? a0[l] : am[l], am2[l], wi, wp);
          T acc = gm[l] * (wi * wm);
          max_w(ap[l], a0[l], wm, wz);   // y = x: (ap op a0) op am, x in the inner second slot
          max_w(ap[l] >= a0[l] ? ap[l] : a0[l], am[l], wi, wp);
          acc += g0[l] * (wi * wz);
          max_w(ap2[l], ap[l], wm, wz);  // y = x + o: (ap2 op ap) op a0, x the outer second slot
          max_w(ap2[l] >= ap[l] ? ap2[l] : ap[l], a0[l], wi, wp);
          v[l] = acc + gp[l] * wp;
        }
      }
      ng = false;
    } else if (op == G_SHIFT) {
      tap<W>(G, c, nd.axis, -nd.sk, g, v);
      ng = false;
    } else if (op == G_ST2 && role == R_B) {
      // y = st1(a) +- st2(b)
      stencil<W>(G, c, nd.axis2, st_transpose(nd.sk2), sp2<T>(nd), g, v);
      ng = st_negates(nd.sk2) != (nd.iop == G_SUB);
    } else {
      // The transposed stencil of G: STENCIL, ST2 and STBIN (a sum) to a; STMUL,
      // y = st(a b), times the other factor.
      stencil<W>(G, c, nd.axis, tk, sp1<T>(nd), g, v);
      if (op == G_STBIN && nd.iop == G_SUB && nd.side) ng = !ng;   // b - st
      if (op == G_STMUL) {
        T f[W];
        ldw<T, W>(role == R_A ? B : A, c, 0, f);
#pragma unroll
        for (int l = 0; l < W; ++l) v[l] = (ng ? -v[l] : v[l]) * f[l];
        ng = false;
      }
    }
    if (ng) {
#pragma unroll
      for (int l = 0; l < W; ++l) v[l] = -v[l];
    }
  }
  // exp's transposes take the epilogue's factor from their own value.
  if ((nd.ep && op != G_EXP && op != G_STEXP) || nd.pop == 3) {
#pragma unroll
    for (int l = 0; l < W; ++l) v[l] *= sv;
  }
}

// ---------------------------------------------------------------------------
// The sweeps' kernels.  A launch runs a batch of nodes that do not depend on
// one another, their blocks interleaved along the launch's z extent (tasks of
// one batch share operands); block-uniform switches pick the op.  A node alone
// is a few microseconds of work (8 MB at 128^3), much of it the launch, its ramp
// and its tail: one launch a node took 9.5 ms for an adjoint step at 128^3 and
// 3.4 ms at 64^3 (on four streams), batches of 24 take 7.4 and 1.5 ms, batches
// of 6 7.6 and 1.6.  The reverse gathers: the thread sums what every consumer
// passes to the node's cells and stores once, where a sweep by consumer reads
// and rewrites the gradient for each of them.
// ---------------------------------------------------------------------------
// x / n as the high word of x times recip32(n), exact for x < 65536, n <= 64.
inline unsigned recip32(int n) { return n == 1 ? 0u : 0xffffffffu / (unsigned)n + 1u; }
__device__ __forceinline__ int div_small(unsigned x, int n, unsigned rn) {
#ifdef __CUDA_ARCH__
  return n == 1 ? (int)x : (int)__umulhi(x, rn);
#else
  return n == 1 ? (int)x : (int)(((unsigned long long)x * rn) >> 32);
#endif
}
// Nodes and terms a batch holds.
#ifndef STG_FWD_MAX
#define STG_FWD_MAX 24
#endif
#ifndef STG_REV_MAX
#define STG_REV_MAX 32
#endif
template <typename T>
struct FwdTask {
  GNode nd;
  const T *A, *B, *C;
  T* out;
};
template <typename T>
struct FwdBatch {
  static constexpr int MAX = STG_FWD_MAX;
  int n;         // tasks
  unsigned rn;   // recip32(n)
  FwdTask<T> t[MAX];
};
template <typename T>
struct RevTerm {
  GNode nd;
  int role;
  const T *A, *B, *Y, *G;
};
// What becomes of dst's old value: replaced, the start of the sum (a sum in
// parts), or added to the sum (the caller's input cotangents).
enum { ADD_NO = 0, ADD_FIRST, ADD_LAST };
template <typename T>
struct RevTask {
  T* dst;
  int first, n, add;   // its terms
};
template <typename T>
struct RevBatch {
  static constexpr int MAX = STG_REV_MAX;
  int n, nterm;
  unsigned rn;
  RevTask<T> t[MAX];
  RevTerm<T> c[MAX];
};
template <typename T>
struct QuenchBatch {
  static constexpr int MAX = 3;
  int n;
  unsigned rn;
  GNode nd[MAX];
  const T* A[MAX];
  T* G[MAX];        // the node's cotangent, replaced by its operand's contribution
  T* scr[MAX];      // 15 arrays each: S (7), Q (8)
};

// Both sweeps wait on their loads and on instruction issue (a stencil of four
// cells is 6 loads, 28 operations and about as many for its indices), so warps
// count until the values no longer fit the registers.  FP32 adjoint step at
// 128^3, blocks an SM for (forward, reverse): (4, 4) 8.27 ms, (5, 5) 7.52,
// (6, 6) 7.60, (6, 5) 7.46-7.53, (6, 4) 7.62, (7, 6) 7.88, (6, 7) 8.03; two planes
// of four cells a thread slower.  FP64 is bound by its own pipe (1 to 4 blocks: the same).
#define STG_GRAPH_LB(T, b32) __launch_bounds__(256, sizeof(T) == 4 ? b32 : 2)

// f(integral constant) for the op of a task or term (uniform over the block).
template <int OP> struct OpC { static constexpr int value = OP; };
template <class F>
__device__ __forceinline__ void for_op(int op, F f) {
  switch (op) {
#define STG_OP(X) case X: f(OpC<X>()); break;
    STG_OP(G_STENCIL) STG_OP(G_STBIN) STG_OP(G_STMUL) STG_OP(G_ST2) STG_OP(G_STEXP) STG_OP(G_NB3)
    STG_OP(G_SHIFT) STG_OP(G_ADD) STG_OP(G_SUB) STG_OP(G_MUL) STG_OP(G_DIV) STG_OP(G_MAX)
    STG_OP(G_EXP) STG_OP(G_LOG) STG_OP(G_LOG1P) STG_OP(G_SQRT) STG_OP(G_ABS) STG_OP(G_AXPB)
    STG_OP(G_CLAMPMIN) STG_OP(G_CLAMPMAX) STG_OP(G_STEP) STG_OP(G_CONST) STG_OP(G_QUENCH)
    default: f(OpC<G_ZFIELD>()); break;
#undef STG_OP
  }
}

template <typename T, int W>
__global__ void STG_GRAPH_LB(T, 6) g_level_fwd(const __grid_constant__ FwdBatch<T> b, const T* mesh,
                                            Geo g) {
  const int kb = div_small(blockIdx.z, b.n, b.rn);
  GCell c;
  if (!gcell_at<W>(c, kb, g)) return;
  const FwdTask<T>& t = b.t[(int)blockIdx.z - kb * b.n];
  for_op(t.nd.op, [&](auto op) {
    node_forward<T, W>(decltype(op)::value, t.nd, t.A, t.B, t.C, t.out, mesh, c, g);
  });
}

template <typename T, int W>
__global__ void STG_GRAPH_LB(T, 5) g_level_rev(const __grid_constant__ RevBatch<T> b, Geo g) {
  const int kb = div_small(blockIdx.z, b.n, b.rn);
  GCell c;
  if (!gcell_at<W>(c, kb, g)) return;
  const RevTask<T>& t = b.t[(int)blockIdx.z - kb * b.n];
  T acc[W];
  if (t.add == ADD_FIRST) ldw<T, W>((const T*)t.dst, c, 0, acc);
  for (int q = 0; q < t.n; ++q) {
    const RevTerm<T>& r = b.c[t.first + q];
    T v[W];
    for_op(r.nd.op, [&](auto op) {
      pull<T, W>(decltype(op)::value, r.role, r.nd, r.A, r.B, r.Y, r.G, c, g, v);
    });
#pragma unroll
    for (int l = 0; l < W; ++l) acc[l] = q == 0 && t.add != ADD_FIRST ? v[l] : acc[l] + v[l];
  }
  if (t.add == ADD_LAST) {
    T o[W];
    ldw<T, W>((const T*)t.dst, c, 0, o);
#pragma unroll
    for (int l = 0; l < W; ++l) acc[l] = o[l] + acc[l];
  }
  stw<T, W>(t.dst, c, acc);
}

// The quench's transpose: PASS 0 q and its derivatives, 1 the cotangents the q
// receive, 2 the operand's contribution over the node's own cotangent.  The passes
// stream 4 to 15 arrays a node and wait on them: blocks an SM for FP32 (quenched
// adjoint step at 128^3): uncapped 9.99 ms, 3 9.71, 4 9.57, 5 9.46, 6 9.51.
template <typename T, int W, int PASS>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 1)
    g_level_quench(const __grid_constant__ QuenchBatch<T> b, Geo g) {
  const int kb = div_small(blockIdx.z, b.n, b.rn);
  const int ti = (int)blockIdx.z - kb * b.n;
  GCell c;
  if (!gcell_at<W>(c, kb, g)) return;
  const GNode& nd = b.nd[ti];
  T* S = b.scr[ti];
  T* Q = S + 7 * g.n;
  if (PASS == 0) quench_q<T, W>(nd, b.A[ti], Q, c, g);
  if (PASS == 1) quench_b1<T, W>(nd, b.A[ti], Q, b.G[ti], S, c, g);
  if (PASS == 2) {
    T acc[W];
    quench_b3<T, W>(nd, Q, S, c, g, acc);
    stw<T, W>(b.G[ti], c, acc);
  }
}

// ---------------------------------------------------------------------------
// One node per launch (op a template constant), the reverse by consumer: not run by
// the library, whose host tests sweep the merged graph and the graph of one node per
// primitive with it.
// ---------------------------------------------------------------------------
template <typename T, int OP>
__global__ void g_forward(GNode nd, const T* A, const T* B, const T* C, T* out, const T* mesh,
                          Geo g) {
  GCell c;
  if (gcell<1>(c, g)) node_forward<T, 1>(OP, nd, A, B, C, out, mesh, c, g);
}
template <typename T, int OP>
__global__ void g_forward4(GNode nd, const T* A, const T* B, const T* C, T* out, const T* mesh,
                           Geo g) {
  GCell c;
  if (gcell<4>(c, g)) node_forward<T, 4>(OP, nd, A, B, C, out, mesh, c, g);
}
// A flat launch over n cells, four at a time with vec.
template <typename T, int OP>
__global__ void g_forward_pw(GNode nd, const T* A, const T* B, const T* C, T* out, long long n,
                             int vec) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const Geo g{};
  GCell c{};
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < (vec ? n / 4 : n);
       t += stride) {
    c.idx = vec ? 4 * t : t;
    if (vec) node_forward<T, 4>(OP, nd, A, B, C, out, nullptr, c, g);
    else node_forward<T, 1>(OP, nd, A, B, C, out, nullptr, c, g);
  }
}
// The operands' contributions, a's first; the first a gradient receives
// writes it (wA, wB, wC), later ones add.
template <typename T, int W>
__device__ __forceinline__ void push_cell(int op, const GNode& nd, const T* A, const T* B,
                                          const T* out, const T* gout, T* gA, T* gB, T* gC, int wA,
                                          int wB, int wC, const GCell& c, const Geo& g) {
  T* dst[3] = {gA, gB, gC};
  const int w[3] = {wA, wB, wC};
  for (int r = 0; r < 3; ++r) {
    if (!dst[r]) continue;
    T v[W], o[W];
    pull<T, W>(op, r, nd, A, B, out, gout, c, g, v);
    if (!w[r]) {
      ldw<T, W>((const T*)dst[r], c, 0, o);
      for (int l = 0; l < W; ++l) v[l] = o[l] + v[l];
    }
    stw<T, W>(dst[r], c, v);
  }
}
template <typename T, int OP>
__global__ void g_backward(GNode nd, const T* A, const T* B, const T* out, const T* gout,
                           T* gA, T* gB, T* gC, int wA, int wB, int wC, Geo g) {
  GCell c;
  if (gcell<1>(c, g)) push_cell<T, 1>(OP, nd, A, B, out, gout, gA, gB, gC, wA, wB, wC, c, g);
}
template <typename T, int OP>
__global__ void g_backward4(GNode nd, const T* A, const T* B, const T* out, const T* gout, T* gA,
                            T* gB, T* gC, int wA, int wB, int wC, Geo g) {
  GCell c;
  if (gcell<4>(c, g)) push_cell<T, 4>(OP, nd, A, B, out, gout, gA, gB, gC, wA, wB, wC, c, g);
}
template <typename T, int OP>
__global__ void g_backward_pw(GNode nd, const T* A, const T* B, const T* out, const T* gout,
                              T* gA, T* gB, T* gC, int wA, int wB, int wC, long long n, int vec) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const Geo g{};
  GCell c{};
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < (vec ? n / 4 : n);
       t += stride) {
    c.idx = vec ? 4 * t : t;
    if (vec) push_cell<T, 4>(OP, nd, A, B, out, gout, gA, gB, gC, wA, wB, wC, c, g);
    else push_cell<T, 1>(OP, nd, A, B, out, gout, gA, gB, gC, wA, wB, wC, c, g);
  }
}
template <typename T>
__global__ void g_quench_f(GNode nd, const T* A, T* out, Geo g) {
  GCell c;
  if (gcell<1>(c, g)) node_forward<T, 1>(G_QUENCH, nd, A, nullptr, nullptr, out, nullptr, c, g);
}
template <typename T>
__global__ void g_quench_f4(GNode nd, const T* A, T* out, Geo g) {
  GCell c;
  if (gcell<4>(c, g)) node_forward<T, 4>(G_QUENCH, nd, A, nullptr, nullptr, out, nullptr, c, g);
}
template <typename T>
__global__ void g_quench_q(GNode nd, const T* A, T* Q, Geo g) {
  GCell c;
  if (gcell<1>(c, g)) quench_q<T, 1>(nd, A, Q, c, g);
}
template <typename T>
__global__ void g_quench_q4(GNode nd, const T* A, T* Q, Geo g) {
  GCell c;
  if (gcell<4>(c, g)) quench_q<T, 4>(nd, A, Q, c, g);
}
template <typename T>
__global__ void g_quench_b1(GNode nd, const T* A, const T* Q, const T* gout, T* S, Geo g) {
  GCell c;
  if (gcell<1>(c, g)) quench_b1<T, 1>(nd, A, Q, gout, S, c, g);
}
template <typename T>
__global__ void g_quench_b1_4(GNode nd, const T* A, const T* Q, const T* gout, T* S, Geo g) {
  GCell c;
  if (gcell<4>(c, g)) quench_b1<T, 4>(nd, A, Q, gout, S, c, g);
}
template <typename T, int W>
__device__ __forceinline__ void quench_put(const GNode& nd, const T* Q, const T* S, T* gA, int wA,
                                           const GCell& c, const Geo& g) {
  T acc[W], o[W];
  quench_b3<T, W>(nd, Q, S, c, g, acc);
  if (!wA) {
    ldw<T, W>((const T*)gA, c, 0, o);
    for (int l = 0; l < W; ++l) acc[l] = o[l] + acc[l];
  }
  stw<T, W>(gA, c, acc);
}
template <typename T>
__global__ void g_quench_b3(GNode nd, const T* Q, const T* S, T* gA, int wA, Geo g) {
  GCell c;
  if (gcell<1>(c, g)) quench_put<T, 1>(nd, Q, S, gA, wA, c, g);
}
template <typename T>
__global__ void g_quench_b3_4(GNode nd, const T* Q, const T* S, T* gA, int wA, Geo g) {
  GCell c;
  if (gcell<4>(c, g)) quench_put<T, 4>(nd, Q, S, gA, wA, c, g);
}

// Horizontal-plane mean (G_PMEAN): one block per z sums its plane in a fixed
// order; the broadcast writes sum / (nx ny).  The mean is linear and symmetric, so
// its transpose is the same mean, of the node's cotangent in place.
template <typename T>
__global__ void g_plane_sum(const T* A, T* psum, Geo g) {
  __shared__ T sm[256];
  const int kz = blockIdx.x;
  const long long m = (long long)g.nx * g.ny;
  T acc = 0;
  for (long long i = threadIdx.x; i < m; i += blockDim.x) acc += A[(long long)kz * g.sz + i];
  sm[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sm[threadIdx.x] += sm[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) psum[kz] = sm[0];
}

template <typename T>
__global__ void g_plane_bcast(const T* psum, T* out, Geo g) {
  GCell c;
  if (!gcell<1>(c, g)) return;
  out[c.idx] = psum[c.k] / (T)((double)g.nx * g.ny);
}

}  // namespace stg
