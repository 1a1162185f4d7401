// Host build of the op graph's executor (graph.cu): its batched sweeps, the launches
// run one thread at a time on host memory, against the graph of one node per primitive
// swept node by node with the one-cell kernels.  Forward outputs must be equal bit for
// bit; gradients, added to what the caller's arrays hold, within 1e-12 (FP64) or
// 1e-5 (FP32) of each field's largest.  Every device array starts as NaN, so a
// cotangent array read before it is written, or reused too early, shows.  Built with
// the library's batch sizes and with small ones, which split the sums of nodes with
// many consumers.  Also: the lean layout of an init whose allocations fail gives the
// same bits, and one without room for that is not ready.  Exit status: the number of
// failing cases.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <random>
#include <vector>
#undef __global__
#undef __device__
#undef __host__
#undef __forceinline__
#undef __launch_bounds__
#undef __shared__
#undef __grid_constant__
#define __global__
#define __device__
#define __host__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __shared__ static
#define __grid_constant__
#define __ldg(p) (*(p))
#define __syncthreads()
uint3 blockIdx, threadIdx;
dim3 blockDim, gridDim;
static inline float __fdividef(float a, float b) { return a / b; }

// Device memory: host memory, NaN-filled, up to a limit.
static size_t g_limit = ~(size_t)0, g_used = 0;
static std::map<void*, size_t> g_sizes;
extern "C" cudaError_t CUDARTAPI cudaMalloc(void** p, size_t n) {
  if (g_used + n > g_limit) return cudaErrorMemoryAllocation;
  *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
  std::memset(*p, 0xff, n);
  g_used += g_sizes[*p] = n;
  return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaFree(void* p) {
  g_used -= g_sizes[p];
  g_sizes.erase(p);
  std::free(p);
  return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaGetLastError() { return cudaSuccess; }

namespace stg {
static int g_badgrid = 0;
// The threads of a block from the last to the first: a tree reduction in shared
// memory, whose thread t reads what threads above it left, then comes out right.
template <class... P, class... A>
static void launch(void (*kern)(P...), dim3 gd, dim3 bd, cudaStream_t, A&&... args) {
  gridDim = gd;
  blockDim = bd;
  g_badgrid += gd.y > 65535 || gd.z > 65535 || bd.x * bd.y * bd.z > 256;
  for (unsigned bz = 0; bz < gd.z; ++bz)
    for (unsigned by = 0; by < gd.y; ++by)
      for (unsigned bx = 0; bx < gd.x; ++bx) {
        blockIdx = make_uint3(bx, by, bz);
        for (int t = (int)(bd.x * bd.y * bd.z) - 1; t >= 0; --t) {
          threadIdx = make_uint3(t % bd.x, t / bd.x % bd.y, t / (bd.x * bd.y));
          kern(static_cast<P>(args)...);
        }
      }
}
template <class... P, class... A>
static void launch_dep(void (*kern)(P...), dim3 gd, dim3 bd, size_t, cudaStream_t s, A&&... args) {
  launch(kern, gd, bd, s, args...);
}
}  // namespace stg
#include "../../paper_2405_02483_gb300/csrc/graph.cu"
#include "../../paper_2405_02483_gb300/csrc/graph_build.cu"
using namespace stg;

template <typename T> using Fields = std::vector<std::vector<T>>;

// One node per primitive, one node after another, each by its one-cell kernel.
template <typename T>
static void reference(const GraphDef& d, const Geo& g, const Fields<T>& in, const Fields<T>& seed,
                      Fields<T>& out, Fields<T>& gin) {
  const int nn = (int)d.nodes.size();
  std::vector<std::vector<T>> v(nn), gr;
  const std::vector<T> mesh(d.mesh.begin(), d.mesh.end());
  const dim3 bd(32, 2, 4), gd((g.nx + 31) / 32, (g.ny + 1) / 2, (g.nz + 3) / 4);
  auto data = [&](std::vector<std::vector<T>>& a, int i) { return i < 0 ? nullptr : a[i].data(); };
  auto pmean = [&](const T* a, T* o, bool add) {
    for (int k = 0; k < g.nz; ++k) {
      T sm[256] = {};   // 256 strided sums, then a tree, as on the device
      for (long long q = 0; q < g.sz; ++q) sm[q % 256] += a[k * g.sz + q];
      for (int s = 128; s > 0; s /= 2)
        for (int t = 0; t < s; ++t) sm[t] += sm[t + s];
      const T m = sm[0] / (T)g.sz;
      for (long long q = 0; q < g.sz; ++q) o[k * g.sz + q] = add ? o[k * g.sz + q] + m : m;
    }
  };
  for (int i = 0; i < nn; ++i) {
    const GNode& nd = d.nodes[i];
    v[i].assign(g.n, 0);
    if (nd.op == G_INPUT) v[i] = in[nd.sk];
    else if (nd.op == G_PMEAN) pmean(v[nd.a].data(), v[i].data(), false);
    else
      for_op(nd.op, [&](auto op) {
        launch(g_forward<T, decltype(op)::value>, gd, bd, nullptr, nd, data(v, nd.a), data(v, nd.b),
               data(v, nd.c), v[i].data(), mesh.data(), g);
      });
  }
  ReversePlan rp;
  plan_reverse(d, rp);
  gr.assign(rp.nslots, std::vector<T>(g.n, (T)NAN));
  for (int k = 0; k < 8; ++k) gr[rp.gslot[d.out[k]]] = seed[k];
  std::vector<T> S(15 * g.n);
  for (int i = nn - 1; i >= 0; --i) {
    const GNode& nd = d.nodes[i];
    if (!rp.hasg[i] || !has_transpose(nd.op)) continue;
    auto gp = [&](int x) { return x < 0 ? nullptr : gr[rp.gslot[x]].data(); };
    if (nd.op == G_PMEAN) {
      pmean(gp(i), gp(nd.a), !rp.wa[i]);
    } else if (nd.op == G_QUENCH) {
      launch(g_quench_q<T>, gd, bd, nullptr, nd, v[nd.a].data(), S.data() + 7 * g.n, g);
      launch(g_quench_b1<T>, gd, bd, nullptr, nd, v[nd.a].data(), S.data() + 7 * g.n, gp(i), S.data(), g);
      launch(g_quench_b3<T>, gd, bd, nullptr, nd, S.data() + 7 * g.n, S.data(), gp(nd.a), rp.wa[i], g);
    } else {
      for_op(nd.op, [&](auto op) {
        launch(g_backward<T, decltype(op)::value>, gd, bd, nullptr, nd, data(v, nd.a), data(v, nd.b),
               v[i].data(), gp(i), gp(nd.a), gp(nd.b), gp(nd.c), rp.wa[i], rp.wb[i], rp.wc[i], g);
      });
    }
  }
  for (int k = 0; k < 8; ++k) {
    out[k] = v[d.out[k]];
    gin[k] = rp.gslot[d.in[k]] >= 0 ? gr[rp.gslot[d.in[k]]] : std::vector<T>(g.n, (T)0);
  }
}

// The executor's sweeps on host arrays; shift moves the caller's arrays off 16-byte
// alignment.  Returns init's status.
template <typename T>
static int sweeps(GraphExec<T>& G, const GraphDef& d, const Geo& g, const Fields<T>& in,
                  const Fields<T>& seed, const Fields<T>& gin0, Fields<T>& out, Fields<T>& gin,
                  int set = 0, int shift = 0) {
  const int rc = G.init(d, g, true);
  if (rc) return rc;
  std::vector<T*> own;
  auto caller = [&](const Fields<T>& f, T* p[8]) {
    for (int k = 0; k < 8; ++k) {
      T* a = nullptr;
      cudaMalloc(&a, sizeof(T) * (g.n + 4));
      own.push_back(a);
      p[k] = a + shift;
      std::copy(f[k].begin(), f[k].end(), p[k]);
    }
  };
  T *pin[8], *ps[8], *pg[8];
  caller(in, pin);
  caller(seed, ps);
  caller(gin0, pg);
  G.forward(pin, nullptr, set);
  for (int k = 0; k < 8; ++k) out[k].assign(G.output(k), G.output(k) + g.n);
  if (set) {   // another set in between
    T* other[8];
    for (int k = 0; k < 8; ++k) other[k] = ps[k];
    G.forward(other, nullptr, 0);
    G.use(set, pin);
  }
  G.backward(ps, pg, nullptr);
  for (int k = 0; k < 8; ++k) gin[k].assign(pg[k], pg[k] + g.n);
  for (T* a : own) cudaFree(a);
  return rc;
}

static stagger_params base_params() {   // the library's defaults, for the fields the graph reads
  stagger_params p;
  memset(&p, 0, sizeof(p));
  p.gamma = 5.0 / 3.0;
  p.nuE = p.nuB = 1.0;
  p.qmax = 8.0;
  p.qlim = 2.0;
  p.quench_eps = 1e-4;
  p.log_interp = 1;
  p.rho_cool = 1.0;
  p.d2lnr_lim = 0.3;
  p.rho_bot = 1.0;
  p.cor_Tunit = 1.0;
  p.nu1 = 0.04;
  p.nu2 = 1.0;
  p.nu3 = 0.04;
  p.do_quench = 1;
  p.ref[0] = 1.0;
  p.ref[4] = 1.5;
  p.ref[7] = 0.5;
  return p;
}

template <typename T>
static bool same(const Fields<T>& a, const Fields<T>& b) {
  for (int k = 0; k < 8; ++k)
    if (std::memcmp(a[k].data(), b[k].data(), sizeof(T) * a[k].size())) return false;
  return true;
}

template <typename T>
static int compare(const char* name, const stagger_grid& gg, const stagger_params& p, int shift = 0) {
  const Geo g = make_geo(gg.nx, gg.ny, gg.nz);
  const double tol = sizeof(T) == 8 ? 1e-12 : 1e-5;
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  Fields<T> in(8, std::vector<T>(g.n)), seed = in, gin0 = in, ro(8), rg(8), out(8), gin(8);
  for (int k = 0; k < 8; ++k)
    for (long long q = 0; q < g.n; ++q) {
      in[k][q] = (T)((k == 0 || k == 4 ? 0.1 : 0.3) * U(rng));
      seed[k][q] = (T)U(rng);
      gin0[k][q] = (T)U(rng);
    }
  GraphDef d, d1;
  build_rhs_graph(d1, gg, p, false);
  build_rhs_graph(d, gg, p, true);
  reference(d1, g, in, seed, ro, rg);
  int fails = 0;
  size_t took = 0;
  // FP64 with a second set of values, FP32 with one and with three planes a thread.
  for (int set = 0; set < 2; ++set) {
    GraphExec<T> G;
    G.planes3_from = set ? 0 : 1LL << 40;
    fails += sweeps(G, d, g, in, seed, gin0, out, gin, sizeof(T) == 8 ? set : 0, shift) != 0;
    took = g_used;
    int deep = 0;
    for (const auto& t : G.lp.terms) deep = std::max(deep, (int)t.size());
    double worst = 0;
    for (int k = 0; k < 8; ++k) {
      double e = 0, s = 0;
      for (long long q = 0; q < g.n; ++q) {
        const double d = std::fabs((double)gin[k][q] - ((double)gin0[k][q] + (double)rg[k][q]));
        e = d <= e ? e : d;   // (keeps a NaN)
        s = std::max(s, std::fabs((double)rg[k][q]));
      }
      worst = e / std::max(s, 1.0) <= worst ? worst : e / std::max(s, 1.0);
    }
    const bool ok = same(ro, out) && worst <= tol && G.ready(true);
    printf("%s %s %dx%dx%d run %d: %d levels, longest sum %d of %d a batch, forward %s, reverse max rel err "
           "%.2e%s\n", name, sizeof(T) == 8 ? "FP64" : "FP32", g.nx, g.ny, g.nz, set, G.lp.nrlev, deep,
           RevBatch<T>::MAX, same(ro, out) ? "equal" : "DIFFERS", worst, ok ? "" : "  FAIL");
    fails += !ok;
    G.release();
    fails += G.ready(false);
  }
  // With less memory: the lean layout (the same bits), then none.
  if (p.do_quench) {
    Fields<T> o2(8), g2(8);
    GraphExec<T> G;
    g_limit = took - sizeof(T) * g.n;
    // (the caller's arrays come after init: give them room again)
    const int rc = G.init(d, g, true);
    const bool lean = G.lean;
    G.release();
    g_limit = ~(size_t)0;
    fails += rc != 0 || !lean;
    GraphExec<T> L;
    L.init(d, g, true, true);
    T *pin[8], *ps[8], *pg[8];
    for (int k = 0; k < 8; ++k) {
      for (T** a : {&pin[k], &ps[k], &pg[k]}) cudaMalloc(a, sizeof(T) * g.n);
      std::copy(in[k].begin(), in[k].end(), pin[k]);
      std::copy(seed[k].begin(), seed[k].end(), ps[k]);
      std::copy(gin0[k].begin(), gin0[k].end(), pg[k]);
    }
    L.forward(pin, nullptr);
    for (int k = 0; k < 8; ++k) o2[k].assign(L.output(k), L.output(k) + g.n);
    L.backward(ps, pg, nullptr);
    for (int k = 0; k < 8; ++k) g2[k].assign(pg[k], pg[k] + g.n);
    if (!shift && !(same(out, o2) && same(gin, g2))) {
      printf("%s lean layout differs  FAIL\n", name);
      ++fails;
    }
    for (int k = 0; k < 8; ++k)
      for (T* a : {pin[k], ps[k], pg[k]}) cudaFree(a);
    L.release();
    for (double part : {0.3, 0.6}) {
      g_limit = (size_t)(part * took);
      if (sizeof(T) == 8 && part > 0.4) continue;   // (the lean layout fits)
      const bool none = G.init(d, g, true) == STAGGER_EOOM && !G.ready(false) && g_used == 0;
      if (!none) printf("%s without room  FAIL\n", name);
      fails += !none;
    }
    g_limit = ~(size_t)0;
  }
  fails += g_used != 0 || g_badgrid;
  return fails;
}

int main() {
  int fails = 0;
  auto grid = [](int nx, int ny, int nz) { return stagger_grid{nx, ny, nz, 1.0 / nx, 1.0 / ny, 1.0 / nz}; };
  stagger_params visc = base_params(), cool = base_params(), opts = base_params();
  cool.t_chromo = 0.05;
  cool.rho_bot = 0.9;
  cool.cor_L0 = 0.3;
  cool.cor_Tunit = 8e3;
  cool.t_cool = 0.2;
  cool.e_cool = 1.2;
  const stagger_grid gs = grid(12, 10, 11);   // stretched
  std::vector<double> zc(gs.nz), zf(gs.nz);
  for (int k = 0; k < gs.nz; ++k) {
    zc[k] = (1.0 + 0.3 * std::sin(2 * M_PI * (k + 0.5) / gs.nz)) / gs.nz;
    zf[k] = (1.0 + 0.3 * std::sin(2 * M_PI * k / (double)gs.nz)) / gs.nz;
  }
  opts.csmag = 0.2;
  opts.c1 = -1.0 / 3.0;
  opts.g[0] = 0.1;
  opts.g[2] = -1.0;
  opts.ediffav = 1;
  opts.lnp_aver = 1;
  opts.do_2nddiv = 1;
  opts.log_interp = 0;
  opts.zc = zc.data();
  opts.zf = zf.data();
  for (const stagger_grid& g : {grid(16, 11, 9), grid(13, 7, 17)}) {
    fails += compare<double>("viscosity+quench", g, visc);
    fails += compare<float>("viscosity+quench", g, visc);
  }
  for (int nz : {3, 4, 5, 13, 26}) fails += compare<float>("planes", grid(9, 6, nz), visc);
  fails += compare<float>("unaligned caller", grid(16, 6, 5), visc, 1);
  fails += compare<float>("one plane", grid(12, 9, 1), visc);
  fails += compare<double>("cooling", grid(13, 11, 9), cool);
  fails += compare<float>("cooling", grid(13, 11, 9), cool);
  fails += compare<double>("options+stretched", gs, opts);
  fails += compare<float>("options+stretched", gs, opts);
  return fails;
}
