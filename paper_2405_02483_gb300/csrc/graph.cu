// Op-graph executor (see graph.cuh): the sweeps as batches of independent
// nodes, one launch per dependency level (kernels in graph_kernels.cuh).
#include <math.h>

#include <stdint.h>

#include <algorithm>

#include "graph_kernels.cuh"

namespace stg {

// ---------------------------------------------------------------------------
// Schedule.  A sweep is a sequence of batches of at most cap nodes that do not
// depend on one another, each the next ready nodes in the graph's order.
// Reverse: the cotangent of a node is the sum of what its consumers pass to it;
// a node whose only term is the consumer's cotangent itself shares that array.
// A cotangent's array is free again after the last batch that reads it.
// ---------------------------------------------------------------------------
static bool special_op(int op) { return op == G_QUENCH || op == G_PMEAN; }

// Whether the term (consumer nd, role) passes nd's cotangent on unchanged.
static bool identity_term(const GNode& nd, int role) {
  if (role == R_COPY) return true;
  if (nd.ep) return false;
  if (role == R_C) return nd.pop != 2;
  if (nd.pop == 3) return false;
  return nd.op == G_ADD || (nd.op == G_SUB && role == R_A);
}

static void plan_sweeps(const GraphDef& G, int cap, LevelPlan& P) {
  const int nn = (int)G.nodes.size();
  P = LevelPlan();
  P.flev.assign(nn, 0);   // 0: an input, or not scheduled yet
  for (int left = nn, lo = 0; lo < nn; ++P.nflev) {
    const int now = P.nflev + 1;
    int took = 0;
    for (int i = lo; i < nn && took < cap; ++i) {
      const GNode& nd = G.nodes[i];
      bool ready = nd.op != G_INPUT && !P.flev[i];
      for (int o : {nd.a, nd.b, nd.c})
        if (o >= 0 && G.nodes[o].op != G_INPUT && (!P.flev[o] || P.flev[o] == now)) ready = false;
      if (ready) {
        P.flev[i] = now;
        ++took;
      }
    }
    while (lo < nn && (G.nodes[lo].op == G_INPUT || P.flev[lo])) ++lo;
    if (!took && --left < 0) break;   // (every pass takes a node: operands come first)
  }
  // Nodes a gradient is worth forming for: those an input reaches.
  std::vector<char> useful(nn, 0);
  for (int i = 0; i < nn; ++i) {
    const GNode& nd = G.nodes[i];
    useful[i] = nd.op == G_INPUT;
    if (has_transpose(nd.op))
      for (int o : {nd.a, nd.b, nd.c})
        if (o >= 0 && useful[o]) useful[i] = 1;
  }
  P.terms.assign(nn, {});
  P.rlev.assign(nn, -1);
  P.alias.assign(nn, P.OWN);
  P.gslot.assign(nn, -1);
  std::vector<int> seeds(nn, 0);
  for (int k = 0; k < 8; ++k)
    if (useful[G.out[k]]) {
      // (the seed of output k as a term with consumer -1 - k)
      P.terms[G.out[k]].push_back({-1 - k, R_COPY});
      ++seeds[G.out[k]];
    }
  for (int i = nn - 1; i >= 0; --i) {
    const GNode& nd = G.nodes[i];
    if (P.terms[i].empty() || !has_transpose(nd.op)) continue;
    if (special_op(nd.op)) {   // its own array holds the operand's contribution
      if (useful[nd.a]) P.terms[nd.a].push_back({i, R_COPY});
      continue;
    }
    if (nd.a >= 0 && useful[nd.a]) P.terms[nd.a].push_back({i, R_A});
    if (nd.b >= 0 && useful[nd.b]) P.terms[nd.b].push_back({i, R_B});
    if (nd.c >= 0 && useful[nd.c]) P.terms[nd.c].push_back({i, R_C});
  }
  for (int i = nn - 1; i >= 0; --i) {
    const GNode& nd = G.nodes[i];
    if (P.terms[i].size() != 1 || nd.op == G_INPUT || special_op(nd.op)) continue;
    const auto& t = P.terms[i][0];
    if (t.consumer < 0 || identity_term(G.nodes[t.consumer], t.role))
      P.alias[i] = t.consumer >= 0 && P.alias[t.consumer] != P.OWN ? P.alias[t.consumer] : t.consumer;
  }
  // A node with no array of its own is ready with the one it shares (a
  // special's after its own passes, which end its batch).
  for (int hi = nn - 1; hi >= 0;) {
    const int now = P.nrlev;
    int took = 0;
    for (int i = hi; i >= 0; --i) {
      if (P.rlev[i] >= 0 || P.terms[i].empty()) continue;
      if (P.alias[i] != P.OWN) {
        if (P.alias[i] < 0) P.rlev[i] = 0;
        else if (P.rlev[P.alias[i]] >= 0) P.rlev[i] = P.rlev[P.alias[i]];
        continue;
      }
      if (took == cap) continue;
      bool ready = true;
      for (const auto& t : P.terms[i])
        if (t.consumer >= 0) {
          const int r = P.alias[t.consumer] == P.OWN ? t.consumer : P.alias[t.consumer];
          if (r >= 0 && (P.rlev[r] < 0 || P.rlev[r] == now)) ready = false;
        }
      if (ready) {
        P.rlev[i] = now;
        ++took;
      }
    }
    while (hi >= 0 && (P.terms[hi].empty() || P.rlev[hi] >= 0)) --hi;
    if (!took) break;   // (every pass takes a node: consumers come last)
    ++P.nrlev;
  }
  // Arrays by liveness: root r's is read up to level last[r].
  auto root = [&](int i) { return P.alias[i] == P.OWN ? i : P.alias[i]; };
  std::vector<int> last(nn, -1);
  for (int i = 0; i < nn; ++i) {
    if (P.rlev[i] < 0 || P.alias[i] != P.OWN) continue;
    for (const auto& t : P.terms[i])
      if (t.consumer >= 0 && root(t.consumer) >= 0)
        last[root(t.consumer)] = std::max(last[root(t.consumer)], P.rlev[i]);
  }
  std::vector<int> freel;
  std::vector<std::pair<int, int>> live;   // (last level, slot)
  for (int L = 0; L < P.nrlev; ++L) {
    for (size_t q = 0; q < live.size();)
      if (live[q].first < L) {
        freel.push_back(live[q].second);
        live[q] = live.back();
        live.pop_back();
      } else {
        ++q;
      }
    for (int i = 0; i < nn; ++i) {
      if (P.rlev[i] != L || P.alias[i] != P.OWN || G.nodes[i].op == G_INPUT) continue;
      if (freel.empty()) freel.push_back(P.nslots++);
      P.gslot[i] = freel.back();
      freel.pop_back();
      live.push_back({std::max(last[i], L), P.gslot[i]});
    }
  }
}

// ---------------------------------------------------------------------------
// Executor
// ---------------------------------------------------------------------------
template <typename T>
int GraphExec<T>::init(const GraphDef& d, const Geo& g, bool with_grads, bool lean_only) {
  release();
  lean = lean_only;
  // Out of memory: what is held goes, and the lean layout is tried.
  auto no_room = [&] {
    release();
    const int rc = no_memory();
    return lean || !with_grads ? rc : init(d, g, with_grads, true);
  };
  def = d;
  geo = g;
  size_t nn = def.nodes.size();
  size_t nval = 0;
  for (auto& nd : def.nodes)
    if (nd.op != G_INPUT) ++nval;
  // FP64: values of all three stages where they take no more than 8 GiB (the
  // quenched physics to 128^3), so that the adjoint evaluates each stage once.
  // FP32 takes its stage states from the fused kernels, whose results differ from
  // the graph's by rounding, and keeps one set.
  nsets = sizeof(T) == sizeof(double) && with_grads && !lean &&
                  3.0 * sizeof(T) * nval * g.n <= 8.0 * (1ull << 30) ? 3 : 1;
  if (cudaMalloc(&vals, sizeof(T) * nsets * nval * g.n) != cudaSuccess) {
    vals = nullptr;
    return no_room();
  }
  bool has_pmean = false;
  int nquench = 0;
  near = true;
  for (auto& nd : def.nodes) {
    has_pmean |= nd.op == G_PMEAN;
    nquench += nd.op == G_QUENCH;
    if ((nd.op == G_SHIFT || nd.op == G_NB3) && nd.sk != 1 && nd.sk != -1) near = false;
  }
  if (nquench && with_grads) {
    // Scratch for several quench nodes at a time, within 8 GiB (at 512^3 one
    // node's launches fill the GPU by themselves).
    const size_t one = sizeof(T) * 15 * (size_t)g.n;
    const size_t fit = std::max<size_t>(1, ((size_t)8 << 30) / one);
    nscr = lean ? 1 : (int)std::min({(size_t)nquench, (size_t)QuenchBatch<T>::MAX, fit});
    if (cudaMalloc(&qscr, one * nscr) != cudaSuccess) {
      qscr = nullptr;
      return no_room();
    }
  }
  if (has_pmean && cudaMalloc(&psum, sizeof(T) * g.nz) != cudaSuccess) {
    psum = nullptr;
    return no_room();
  }
  if (!def.mesh.empty()) {
    std::vector<T> m(def.mesh.begin(), def.mesh.end());
    if (cudaMalloc(&mesh, sizeof(T) * m.size()) != cudaSuccess) {
      mesh = nullptr;
      return no_room();
    }
    if (cudaMemcpy(mesh, m.data(), sizeof(T) * m.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
      release();
      return STAGGER_ECUDA;
    }
  }
  plan_sweeps(def, FwdBatch<T>::MAX, lp);
  if (with_grads) {
    if (cudaMalloc(&grads, sizeof(T) * (size_t)std::max(1, lp.nslots) * g.n) != cudaSuccess) {
      grads = nullptr;
      return no_room();
    }
  }
  nvals = nval;
  ptr.assign(nn, nullptr);
  T* none[8] = {};
  use(0, none);
  return STAGGER_OK;
}

template <typename T>
void GraphExec<T>::use(int set, T* const in[8]) {
  size_t v = (size_t)set * nvals;
  for (size_t i = 0; i < def.nodes.size(); ++i)
    ptr[i] = def.nodes[i].op == G_INPUT ? in[def.nodes[i].sk] : vals + (v++) * geo.n;
}

template <typename T>
void GraphExec<T>::release() {
  if (vals) cudaFree(vals);
  if (grads) cudaFree(grads);
  if (mesh) cudaFree(mesh);
  if (psum) cudaFree(psum);
  if (qscr) cudaFree(qscr);
  vals = grads = mesh = psum = qscr = nullptr;
  ptr.clear();
}

static inline bool al16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// Block shape of a sweep with w cells a thread along x and wz along z: the widest
// along x among those that cover the box with the fewest threads (256 threads; at nx
// = 64 half the lanes of a 32-lane row of four-cell threads have no cell).
static dim3 level_block(const Geo& g, int w, int wz) {
  static const int sh[6][3] = {{32, 2, 4}, {16, 4, 4}, {8, 8, 4}, {32, 8, 1}, {16, 16, 1}, {8, 32, 1}};
  const long long lanes = (g.nx + w - 1) / w;
  const int* best = sh[0];
  long long least = -1;
  for (const auto& s : sh) {
    const long long t = (lanes + s[0] - 1) / s[0] * s[0] * ((g.ny + s[1] - 1) / s[1] * s[1]) *
                        ((g.nz + wz * s[2] - 1) / (wz * s[2]) * s[2]);
    if (least < 0 || t < least) {
      least = t;
      best = s;
    }
  }
  return dim3((unsigned)best[0], (unsigned)best[1], (unsigned)best[2]);
}
struct LevelGrid {
  dim3 b;
  unsigned gx, gy;
  int nzb;
  LevelGrid(const Geo& g, int W) {   // W as in GCell
    const int w = W == 4 ? 4 : 1, wz = W / w;
    b = level_block(g, w, wz);
    gx = (unsigned)((g.nx + b.x * w - 1) / (b.x * w));
    gy = (unsigned)((g.ny + b.y - 1) / b.y);
    nzb = (int)((g.nz + b.z * wz - 1) / (b.z * wz));
  }
  int most(int cap) const { return std::max(1, std::min(cap, 65535 / nzb)); }   // gridDim.z
  dim3 grid(int n) const { return dim3(gx, gy, (unsigned)(nzb * n)); }
};

// Four cells a thread: rows of whole 16-byte chunks, aligned arrays, shifts of
// one cell.
template <typename T>
static bool cells4(const GraphExec<T>& G, T* const* a, int n) {
  bool ok = G.geo.nx % 4 == 0 && G.near;
  for (int i = 0; i < n; ++i) ok = ok && al16(a[i]);
  return ok;
}

// FP32 rows of other lengths: three planes a thread (GCell), from the size where
// fewer threads still fill the GPU (viscous adjoint step, us, one plane / three: 30^3
// 848 / 980, 43^3 1371 / 1449, 53^3 2029 / 1858, 65^3 3612 / 2993).
template <typename T>
static bool planes3(const GraphExec<T>& G) {
  return G.geo.nz >= 3 && G.geo.n >= G.planes3_from;
}

template <typename T, int W>
static int forward_w(GraphExec<T>& G, cudaStream_t s) {
  const Geo& g = G.geo;
  const int nn = (int)G.def.nodes.size();
  const LevelGrid lg(g, W);
  FwdBatch<T> b;
  const int most = lg.most(FwdBatch<T>::MAX);
  for (int L = 1; L <= G.lp.nflev; ++L) {
    b.n = 0;
    auto flush = [&] {
      if (!b.n) return;
      b.rn = recip32(b.n);
      launch_dep(g_level_fwd<T, W>, lg.grid(b.n), lg.b, 0, s, b, G.mesh, g);
      ++G.launches;
      b.n = 0;
    };
    for (int i = 0; i < nn; ++i) {
      const GNode& nd = G.def.nodes[i];
      if (nd.op == G_INPUT || G.lp.flev[i] != L) continue;
      const T* A = nd.a >= 0 ? G.ptr[nd.a] : nullptr;
      if (nd.op == G_PMEAN) {
        const LevelGrid l1(g, 1);
        launch(g_plane_sum<T>, dim3(g.nz), dim3(256), s, A, G.psum, g);
        launch(g_plane_bcast<T>, l1.grid(1), l1.b, s, G.psum, G.ptr[i], g);
        G.launches += 2;
        continue;
      }
      b.t[b.n++] = {nd, A, nd.b >= 0 ? G.ptr[nd.b] : nullptr, nd.c >= 0 ? G.ptr[nd.c] : nullptr,
                    G.ptr[i]};
      if (b.n == most) flush();
    }
    flush();
  }
  STG_CUDA_OK(cudaGetLastError());
  return STAGGER_OK;
}

template <typename T>
int GraphExec<T>::forward(T* const in[8], cudaStream_t s, int set) {
  use(set, in);
  // FP64 takes one cell a thread: its pipe, not the loads, is the bound (32^3
  // adjoint step 2.8 ms against 3.8 with four).
  if constexpr (sizeof(T) == sizeof(float))
    return cells4(*this, in, 8) ? forward_w<T, 4>(*this, s)
           : planes3(*this)      ? forward_w<T, 3>(*this, s)
                                 : forward_w<T, 1>(*this, s);
  return forward_w<T, 1>(*this, s);
}

// The quench nodes q[0 .. n) of a level, nscr at a time.
template <typename T, int W>
static void quench_rev(GraphExec<T>& G, const std::vector<int>& q, const LevelGrid& lg,
                       cudaStream_t s) {
  const int most = lg.most(G.nscr);
  for (size_t q0 = 0; q0 < q.size(); q0 += most) {
    QuenchBatch<T> b;
    b.n = (int)std::min<size_t>(most, q.size() - q0);
    b.rn = recip32(b.n);
    for (int j = 0; j < b.n; ++j) {
      const int i = q[q0 + j];
      b.nd[j] = G.def.nodes[i];
      b.A[j] = G.ptr[G.def.nodes[i].a];
      b.G[j] = G.grads + (size_t)G.lp.gslot[i] * G.geo.n;
      b.scr[j] = G.qscr + (size_t)15 * j * G.geo.n;
    }
    launch_dep(g_level_quench<T, W, 0>, lg.grid(b.n), lg.b, 0, s, b, G.geo);
    launch_dep(g_level_quench<T, W, 1>, lg.grid(b.n), lg.b, 0, s, b, G.geo);
    launch_dep(g_level_quench<T, W, 2>, lg.grid(b.n), lg.b, 0, s, b, G.geo);
    G.launches += 3;
  }
}

template <typename T, int W>
static int backward_w(GraphExec<T>& G, T* const seed[8], T* gin[8], cudaStream_t s) {
  const Geo& g = G.geo;
  const LevelPlan& P = G.lp;
  const int nn = (int)G.def.nodes.size();
  const LevelGrid lg(g, W);
  const int most = lg.most(RevBatch<T>::MAX);
  // The cotangent array of node i (-1 - k: the seed of output k).
  auto garr = [&](int i) -> T* {
    if (i >= 0 && P.alias[i] != P.OWN) i = P.alias[i];
    return i < 0 ? seed[-1 - i] : G.grads + (size_t)P.gslot[i] * g.n;
  };
  RevBatch<T> b;
  b.n = b.nterm = 0;
  auto flush = [&] {
    if (!b.n) return;
    b.rn = recip32(b.n);
    launch_dep(g_level_rev<T, W>, lg.grid(b.n), lg.b, 0, s, b, g);
    ++G.launches;
    b.n = b.nterm = 0;
  };
  for (int L = 0; L < P.nrlev; ++L) {
    // The nodes with most terms first: their blocks run longest.
    std::vector<int> lev;
    for (int i = 0; i < nn; ++i)
      if (P.rlev[i] == L && P.alias[i] == P.OWN) lev.push_back(i);
    std::stable_sort(lev.begin(), lev.end(),
                     [&](int x, int y) { return P.terms[x].size() > P.terms[y].size(); });
    std::vector<int> quench, pmean;
    for (int i : lev) {
      const GNode& nd = G.def.nodes[i];
      if (nd.op == G_QUENCH) quench.push_back(i);
      if (nd.op == G_PMEAN) pmean.push_back(i);
      const auto& tm = P.terms[i];
      T* dst = nd.op == G_INPUT ? gin[nd.sk] : garr(i);
      // An input's sum goes onto what gin holds; a sum of more than MAX terms
      // runs in parts.
      for (size_t t0 = 0; t0 < tm.size(); t0 += RevBatch<T>::MAX) {
        const int n = (int)std::min<size_t>(RevBatch<T>::MAX, tm.size() - t0);
        if (b.n == most || b.nterm + n > RevBatch<T>::MAX) flush();
        const int add = t0 > 0 ? ADD_FIRST
                      : nd.op != G_INPUT ? ADD_NO
                      : (int)tm.size() <= RevBatch<T>::MAX ? ADD_LAST : ADD_FIRST;
        b.t[b.n++] = {dst, b.nterm, n, add};
        for (int q = 0; q < n; ++q) {
          const auto& t = tm[t0 + q];
          RevTerm<T>& r = b.c[b.nterm++];
          r = RevTerm<T>();
          r.role = t.role;
          r.G = garr(t.consumer);
          if (t.consumer < 0 || t.role == R_COPY) continue;
          r.nd = G.def.nodes[t.consumer];
          r.A = r.nd.a >= 0 ? G.ptr[r.nd.a] : nullptr;
          r.B = r.nd.b >= 0 ? G.ptr[r.nd.b] : nullptr;
          r.Y = G.ptr[t.consumer];
        }
        if (t0 + n < tm.size()) flush();   // the next part adds to this one's result
      }
    }
    flush();
    // Their own arrays become the operand's contribution.
    quench_rev<T, W>(G, quench, lg, s);
    for (int i : pmean) {
      const LevelGrid l1(g, 1);
      launch(g_plane_sum<T>, dim3(g.nz), dim3(256), s, garr(i), G.psum, g);
      launch(g_plane_bcast<T>, l1.grid(1), l1.b, s, G.psum, garr(i), g);
      G.launches += 2;
    }
  }
  STG_CUDA_OK(cudaGetLastError());
  return STAGGER_OK;
}

template <typename T>
int GraphExec<T>::backward(T* const seed[8], T* gin[8], cudaStream_t s) {
  if (!grads) return STAGGER_EINVAL;
  T* in[8];
  int ni = 0;
  for (size_t i = 0; i < def.nodes.size() && ni < 8; ++i)
    if (def.nodes[i].op == G_INPUT) in[ni++] = ptr[i];
  if constexpr (sizeof(T) == sizeof(float))
    return cells4(*this, seed, 8) && cells4(*this, gin, 8) && cells4(*this, in, ni)
               ? backward_w<T, 4>(*this, seed, gin, s)
           : planes3(*this) ? backward_w<T, 3>(*this, seed, gin, s)
                            : backward_w<T, 1>(*this, seed, gin, s);
  return backward_w<T, 1>(*this, seed, gin, s);
}

template struct GraphExec<float>;
template struct GraphExec<double>;

}  // namespace stg
