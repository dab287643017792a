// lattice.cu -- an acyclic input lattice composed with the FST.
//
// The paper decodes input strings and names input lattices as the general
// case its approach extends to (Sec. 6.1).  A lattice here is a DAG whose
// nodes are numbered in a topological order: node 0 is the start, node N-1
// the end, and edge e goes from from[e] to to[e] > from[e], reads symbol
// label[e] and carries the log-weight weight[e].  Its paths replace the one
// path of a string; the FST reads the symbols along them.  The recursions
// run node by node, and each edge relaxes every arc of its symbol's slice
// (the paper's slice-wide relaxation, Sec. 5) into dense per-node tables:
//   Viterbi  V[v][q'] = max over edges e = (u -> v) and arcs k = (q -> q') of
//            fl(fl(V[u][q] + theta_k) + w_e), packed 64-bit keys
//            (score << 32 | ~arc id) so that ties go to the lowest arc id;
//            the backtrace takes the lowest edge id among the edges that
//            reach the same score with that arc;
//   forward  alpha[v][q'] = log-sum-exp of alpha[u][q] + w_e + theta_k in
//            float64: an exact maximum (64-bit order keys), then exp(value -
//            maximum) summed in 2^-40 fixed point, as in the step kernels;
//   backward beta[u][q] likewise from the end node; log Z, and the
//            posterior of each arc (summed over the edges reading its
//            symbol) and of each edge (summed over its arcs).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "fst_internal.cuh"
#include "frontier.cuh"

using namespace fstgpu;

namespace {

constexpr int TB = 256;
inline unsigned nb(int64_t n) { return (unsigned)std::max<int64_t>(1, (n + TB - 1) / TB); }

// The lattice's edges on the device, grouped by the node they go into (or
// come out of), each group in increasing edge id.  pre[j] counts the padded
// arcs of the edges before position j, so that one launch covers all edges
// of a node: flat arc pre[lo] + i belongs to the last edge with pre <= it.
// The slices are whole 128-arc windows, so a warp's 32 arcs are one edge's.
struct EdgeRec {
  int64_t i0;     // first arc record of the edge's symbol
  int32_t id;     // caller's edge id
  int32_t from, to;
  float w;
};
struct EdgeView {
  const EdgeRec* e;
  const int64_t* pre;
};
__device__ __forceinline__ int32_t edge_of(const EdgeView& G, int32_t lo, int32_t hi, int64_t x) {
  while (hi - lo > 1) {
    const int32_t mid = (lo + hi) >> 1;
    if (__ldg(G.pre + mid) <= x) lo = mid; else hi = mid;
  }
  return lo;
}

// One flat arc of a node's edges: its edge, record and weight.  None of it
// changes during a call, so a chained launch reads its first ones before it
// waits for the launch before it.
struct FlatArc {
  EdgeRec e;
  int4 a;
  float th;
};
__device__ __forceinline__ FlatArc flat_arc(const EdgeView& G, int32_t lo, int32_t hi, const int4* __restrict__ arcs,
                                            const float* __restrict__ theta, int64_t x) {
  FlatArc f;
  const int32_t j = edge_of(G, lo, hi, x);
  f.e = G.e[j];
  const int64_t i = f.e.i0 + (x - __ldg(G.pre + j));
  f.a = __ldg(arcs + i);
  f.th = __ldg(theta + i);
  return f;
}
// The launch after this one may begin (it waits for this one's end, and so
// for all before), and this one's inputs are there.
__device__ __forceinline__ void chain_through() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Start node: the start weights as keys (no incoming arc: low word 0).
__global__ void k_lat_vit_init(const float* __restrict__ theta_s, int32_t Q, unsigned long long* __restrict__ keys0) {
  const int32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= Q) return;
  const float v = theta_s[q];
  keys0[q] = v == neg_inf() ? 0ull : ((unsigned long long)fkey(v) << 32);
}

// The edges [lo, hi) into a node: every arc of their slices with a live
// source.
__global__ void __launch_bounds__(TB) k_lat_vit_node(EdgeView G, int32_t lo, int32_t hi,
                                                     const int4* __restrict__ arcs, const float* __restrict__ theta,
                                                     int32_t Q, unsigned long long* __restrict__ keys) {
  const int64_t p1 = __ldg(G.pre + hi), step = (int64_t)gridDim.x * TB;
  int64_t x = __ldg(G.pre + lo) + (int64_t)blockIdx.x * TB + threadIdx.x;
  FlatArc f{};
  if (x < p1) f = flat_arc(G, lo, hi, arcs, theta, x);
  chain_through();
  while (x < p1) {
    if (f.a.z >= 0) {
      const unsigned long long kp = __ldcg(keys + (int64_t)f.e.from * Q + f.a.x);
      if (kp) {
        const float c = __fadd_rn(__fadd_rn(fkey_inv((uint32_t)(kp >> 32)), f.th), f.e.w);
        if (c != neg_inf())
          atomicMax(keys + (int64_t)f.e.to * Q + f.a.y,
                    ((unsigned long long)fkey(c) << 32) | (unsigned long long)(~(uint32_t)f.a.z));
      }
    }
    if ((x += step) < p1) f = flat_arc(G, lo, hi, arcs, theta, x);
  }
}

__device__ __forceinline__ float key_score(unsigned long long k) {
  return k ? fkey_inv((uint32_t)(k >> 32)) : neg_inf();
}

// Best end state (lowest id on ties), over all blocks, then the backtrace by
// a warp of the last of them: at node v in state q the key names the best arc
// k; the edge is the lowest id into v that reads k's symbol (k is among its
// source's arcs on the edge's symbol) and reaches the same score through it
// -- a lane per edge.  At most N-1 steps (each moves to a lower node).
// out: score, path length, the edges, the arcs (both from the end back).
// end: {best key, blocks done}, both 0 before.  (One block over 50,000 states
// and 30 nodes took 108 us, most of it the states.)
__global__ void __launch_bounds__(TB) k_lat_vit_final(LayoutView L, EdgeView G, const int32_t* __restrict__ in_off,
                                                      const int32_t* __restrict__ elabel,
                                                      const unsigned long long* __restrict__ keys, int32_t N,
                                                      int32_t Q, const float* __restrict__ theta_f,
                                                      const int32_t* __restrict__ src_by_id,
                                                      unsigned long long* __restrict__ end, int32_t* __restrict__ out) {
  __shared__ unsigned long long red[TB / 32];
  const int lane = threadIdx.x & 31;
  const unsigned long long* last = keys + (int64_t)(N - 1) * Q;
  unsigned long long best = 0ull;
  for (int32_t q = (int32_t)(blockIdx.x * TB + threadIdx.x); q < Q; q += (int32_t)(gridDim.x * TB)) {
    const float c = __fadd_rn(key_score(last[q]), theta_f[q]);
    if (c == neg_inf()) continue;
    const unsigned long long k = ((unsigned long long)fkey(c) << 32) | (unsigned long long)(~(uint32_t)q);
    best = k > best ? k : best;
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    const unsigned long long o = __shfl_xor_sync(FULL, best, d);
    best = o > best ? o : best;
  }
  if (lane == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  if (lane == 0) {
    for (int w = 1; w < TB / 32; ++w) best = red[w] > best ? red[w] : best;
    if (best) atomicMax(end, best);
    __threadfence();
    const bool done = atomicAdd(end + 1, 1ull) + 1ull == gridDim.x;
    __threadfence();
    red[0] = done ? 1ull : 0ull;
    red[1] = __ldcg(end);
  }
  __syncwarp();
  if (!red[0]) return;
  best = red[1];
  int32_t* edge_path = out + 2;
  int32_t* arc_path = edge_path + (N > 1 ? N - 1 : 1);
  int32_t len = 0;
  if (best) {
    int32_t v = N - 1, q = (int32_t)(~(uint32_t)best);
    for (int32_t step = 0; step < N - 1 && v != 0; ++step) {
      const unsigned long long kv = keys[(int64_t)v * Q + q];
      const int32_t k = (int32_t)(~(uint32_t)kv);
      const int32_t lo = __ldg(in_off + v), hi = __ldg(in_off + v + 1);
      if (!kv || k < 0) { len = -1; break; }
      const float s = key_score(kv);
      const int32_t src = __ldg(src_by_id + k);
      int32_t e_best = -1, from = 0;
      for (int32_t j0 = lo; j0 < hi && e_best < 0; j0 += 32) {  // edges into v, by increasing id
        const int32_t j = j0 + lane;
        bool hit = false;
        EdgeRec e{0, 0, 0, 0, 0.f};
        if (j < hi) {
          e = G.e[j];
          SegProbe<true> pr;
          seg_load(L, __ldg(elabel + e.id), src, pr);
          const float vu = key_score(keys[(int64_t)e.from * Q + src]);
          int4 a = make_int4(0, 0, -1, 0);
          const Arcs r = seg_find(L, pr, &a);
          if (vu != neg_inf())
            for (int32_t i = 0; i < r.len; ++i) {
              if (i > 0) a = __ldg(L.arcs + r.pos + i);
              if (a.z == k) {
                hit = __fadd_rn(__fadd_rn(vu, __int_as_float(a.y)), e.w) == s;
                break;
              }
            }
        }
        const uint32_t hits = __ballot_sync(FULL, hit);
        if (hits) {
          e_best = __shfl_sync(FULL, e.id, __ffs(hits) - 1);
          from = __shfl_sync(FULL, e.from, __ffs(hits) - 1);
        }
      }
      if (e_best < 0) { len = -1; break; }
      if (lane == 0) {
        edge_path[len] = e_best;
        arc_path[len] = k;
      }
      ++len;
      v = from;
      q = src;
    }
  }
  if (lane == 0) {
    out[0] = __float_as_int(best ? fkey_inv((uint32_t)(best >> 32)) : neg_inf());
    out[1] = len;
  }
}

// A node's values in the forward and backward passes: {fixed-point sum,
// order key of the maximum} per state, the value formed where it is read (a
// sum that is one term takes no logarithm), so that no pass over the states
// stands between the nodes.
__device__ __forceinline__ double lse_value(const ulonglong2* __restrict__ tab, int64_t i) {
  const ulonglong2 x = __ldcg(tab + i);
  return x.y ? fix_log_sum64(dkey_inv(x.y), x.x) : -INFINITY;
}
__global__ void k_lat_lse_init(const float* __restrict__ in, int32_t Q, ulonglong2* __restrict__ tab) {
  const int32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= Q) return;
  const float v = in[q];
  tab[q] = v == neg_inf() ? make_ulonglong2(0ull, 0ull) : make_ulonglong2(1099511627776ull, dkey((double)v));  // 2^40
}

// Step by step both passes at once: the forward relaxation of all edges into
// a node (F.lo .. F.hi of its edges) and the backward one of all edges out of
// another (B), which need nothing of each other.  Two phases a step: the
// exact maximum of each target, then the fixed-point sums.
// Forward: target = destination, value = tab[from][src] + w + theta;
// backward: target = source, value = tab[to][dst] + w + theta.
// A launch is bound by its own latency (a lookup, a value, an atomic); with
// the passes one after the other a call on 30 nodes took 116 of them, now 58.
struct StepSide {
  EdgeView G;
  int32_t lo, hi;
  int64_t n;  // flat arcs
  ulonglong2* tab;
};
template <bool SUM>
__device__ __forceinline__ void lse_arc(const FlatArc& f, bool fwd, ulonglong2* tab, int32_t Q) {
  if (f.a.z < 0 || dead32(f.th)) return;
  const double u = lse_value(tab, (int64_t)(fwd ? f.e.from : f.e.to) * Q + (fwd ? f.a.x : f.a.y));
  if (dead64(u)) return;
  const double v = u + (double)f.e.w + (double)f.th;
  if (dead64(v)) return;
  unsigned long long* t = (unsigned long long*)(tab + (int64_t)(fwd ? f.e.to : f.e.from) * Q + (fwd ? f.a.y : f.a.x));
  if (!SUM) atomicMax(t + 1, dkey(v));
  else atomicAdd(t, fix_exp64(v, dkey_inv(__ldcg(t + 1))));
}
template <bool SUM>
__global__ void __launch_bounds__(TB) k_lat_lse_step(const __grid_constant__ StepSide F,
                                                     const __grid_constant__ StepSide B,
                                                     const int4* __restrict__ arcs, const float* __restrict__ theta,
                                                     int32_t Q) {
  // (the sides have whole 128-arc windows: a warp's arcs are one side's)
  const int64_t n = F.n + B.n, step = (int64_t)gridDim.x * TB;
  int64_t x = (int64_t)blockIdx.x * TB + threadIdx.x;
  auto get = [&]() {
    return x < F.n ? flat_arc(F.G, F.lo, F.hi, arcs, theta, __ldg(F.G.pre + F.lo) + x)
                   : flat_arc(B.G, B.lo, B.hi, arcs, theta, __ldg(B.G.pre + B.lo) + x - F.n);
  };
  FlatArc f{};
  if (x < n) f = get();
  chain_through();
  while (x < n) {
    const bool fwd = x < F.n;
    lse_arc<SUM>(f, fwd, fwd ? F.tab : B.tab, Q);
    if ((x += step) < n) f = get();
  }
}

// log Z = LSE_q(alpha_end[q] + theta_f[q]) in float64: every block a part
// (its largest value and the sum of the exponentials below it), the last of
// them the parts in their order.  (One block over 50,000 states took 113 us.)
struct LogzPart {
  double m, s;
};
constexpr int LOGZ_BLOCKS = 128;
__global__ void __launch_bounds__(TB) k_lat_logz(const ulonglong2* __restrict__ end, const float* __restrict__ theta_f,
                                                 int32_t Q, LogzPart* __restrict__ part, uint32_t* __restrict__ done,
                                                 double* __restrict__ logz) {
  chain_enter();
  __shared__ double red[TB / 32];
  auto over = [&](double x, bool sum) {  // the block's largest value, or its sum
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
      const double y = __shfl_xor_sync(FULL, x, d);
      x = sum ? x + y : fmax(x, y);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    x = red[0];
    for (int w = 1; w < TB / 32; ++w) x = sum ? x + red[w] : fmax(x, red[w]);
    return x;
  };
  auto value = [&](int32_t q) { return dead32(theta_f[q]) ? -INFINITY : lse_value(end, q) + (double)theta_f[q]; };
  const int32_t q0 = (int32_t)(blockIdx.x * TB + threadIdx.x), step = (int32_t)(gridDim.x * TB);
  double m = -INFINITY, s = 0.0;
  for (int32_t q = q0; q < Q; q += step) m = fmax(m, value(q));
  m = over(m, false);
  if (m != -INFINITY)
    for (int32_t q = q0; q < Q; q += step) {
      const double v = value(q);
      if (!dead64(v)) s += exp(v - m);
    }
  s = over(s, true);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = LogzPart{m, s};
    __threadfence();
    last = atomicAdd(done, 1u) + 1u == gridDim.x;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  const bool mine = threadIdx.x < gridDim.x;  // (a thread a part)
  const double pm = mine ? __ldcg(&part[threadIdx.x].m) : -INFINITY, ps = mine ? __ldcg(&part[threadIdx.x].s) : 0.0;
  m = over(pm, false);
  s = over(m == -INFINITY || pm == -INFINITY ? 0.0 : pm == m ? ps : ps * exp(pm - m), true);
  if (threadIdx.x == 0) *logz = m == -INFINITY ? -INFINITY : m + log(s);
}

// Posteriors through every edge: exp(alpha[u][src] + w + theta + beta[v][dst]
// - log Z) to each arc's count and to the edge's posterior.
__global__ void __launch_bounds__(TB) k_lat_post(EdgeView G, int32_t E, const int4* __restrict__ arcs,
                                                 const float* __restrict__ theta, int32_t Q,
                                                 const ulonglong2* __restrict__ alpha,
                                                 const ulonglong2* __restrict__ beta, const double* logz,
                                                 double* __restrict__ cnt, double* __restrict__ epost) {
  chain_enter();
  const double lz = __ldcg(logz);
  if (lz == -INFINITY) return;
  const int64_t p1 = __ldg(G.pre + E);
  // (whole warps: p1 is a multiple of 128)
  for (int64_t x = (int64_t)blockIdx.x * TB + threadIdx.x; x < p1; x += (int64_t)gridDim.x * TB) {
    const FlatArc f = flat_arc(G, 0, E, arcs, theta, x);
    const EdgeRec& e = f.e;
    const int4 a = f.a;
    const float th = f.th;
    double g = 0.0;
    if (a.z >= 0 && !dead32(th)) {
      const double al = lse_value(alpha, (int64_t)e.from * Q + a.x);
      if (!dead64(al)) {
        const double be = lse_value(beta, (int64_t)e.to * Q + a.y);
        if (!dead64(be)) {
          g = exp(al + (double)e.w + (double)th + be - lz);
          atomicAdd(cnt + a.z, g);
        }
      }
    }
    if (!__any_sync(FULL, g != 0.0)) continue;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) g += __shfl_xor_sync(FULL, g, d);
    if ((threadIdx.x & 31) == 0) atomicAdd(epost + e.id, g);
  }
}

// Counts of the arcs, then posteriors of the edges, to float32.
__global__ void k_lat_to_f32(const double* __restrict__ in, int64_t n, float* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

struct DevGuard {
  int old = -1;
  explicit DevGuard(int dev) {
    if (cudaGetDevice(&old) != cudaSuccess) old = -1;
    if (old != dev) cudaSetDevice(dev);
  }
  ~DevGuard() {
    int cur = -1;
    if (old >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != old) cudaSetDevice(old);
  }
};

// A validated lattice on the host: edges grouped by destination and by
// source node, each group in increasing edge id.
struct HostLattice {
  int32_t N = 0, E = 0;
  std::vector<int32_t> in_off, in_edge, out_off, out_edge;
};

int check_lattice(const fst_s* f, int32_t N, int32_t E, const int32_t* from, const int32_t* to, const int32_t* label,
                  const float* weight, HostLattice* L) {
  if (N < 1 || E < 0 || (E > 0 && (!from || !to || !label || !weight))) {
    set_error("lattice: bad sizes or NULL arrays");
    return FST_ERR_INVALID_ARG;
  }
  for (int32_t e = 0; e < E; ++e) {
    if (from[e] < 0 || to[e] <= from[e] || to[e] >= N) {
      set_error("lattice edge %d goes from node %d to node %d: edges must go to a higher node id below %d", e,
                from[e], to[e], N);
      return FST_ERR_INVALID_ARG;
    }
    if (label[e] < 0 || label[e] >= f->m) {
      set_error("lattice edge %d reads symbol %d outside [0, %d)", e, label[e], f->m);
      return FST_ERR_INVALID_ARG;
    }
    if (isnan(weight[e]) || weight[e] == INFINITY) {
      set_error("lattice edge %d has weight NaN or +inf", e);
      return FST_ERR_INVALID_ARG;
    }
  }
  L->N = N;
  L->E = E;
  L->in_off.assign(N + 1, 0);
  L->out_off.assign(N + 1, 0);
  for (int32_t e = 0; e < E; ++e) {
    ++L->in_off[to[e] + 1];
    ++L->out_off[from[e] + 1];
  }
  for (int32_t v = 0; v < N; ++v) {
    L->in_off[v + 1] += L->in_off[v];
    L->out_off[v + 1] += L->out_off[v];
  }
  L->in_edge.assign(std::max(E, 1), 0);
  L->out_edge.assign(std::max(E, 1), 0);
  std::vector<int32_t> fi(L->in_off.begin(), L->in_off.end() - 1), fo(L->out_off.begin(), L->out_off.end() - 1);
  for (int32_t e = 0; e < E; ++e) {
    L->in_edge[fi[to[e]]++] = e;
    L->out_edge[fo[from[e]]++] = e;
  }
  return FST_OK;
}

// One host image of the device's edge tables: the edges grouped by
// destination node, and (both) by source node too, their arcs counted.
struct EdgeTables {
  std::vector<EdgeRec> e;
  std::vector<int64_t> pre;
  void add(const SliceView& sv, const std::vector<int32_t>& order, int32_t E, const int32_t* from, const int32_t* to,
           const int32_t* label, const float* weight) {
    int64_t x = 0;
    for (int32_t j = 0; j < E; ++j) {
      const int32_t k = order[j], a = label[k];
      e.push_back(EdgeRec{sv.h_sym_win[a] * (int64_t)WIN, k, from[k], to[k], weight[k]});
      pre.push_back(x);
      x += (sv.h_sym_win[a + 1] - sv.h_sym_win[a]) * (int64_t)WIN;
    }
    pre.push_back(x);
  }
};

// A launch over n flat arcs, chained to the one before it; half the blocks
// an SM holds, so that the next launch's fit beside them.
constexpr int LAT_BLOCKS = 4;
template <class... KArgs, class... Args>
int launch_arcs(void (*kernel)(KArgs...), int64_t n, int num_sms, cudaStream_t s, Args... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>((n + TB - 1) / TB, LAT_BLOCKS * (int64_t)num_sms)));
  cfg.blockDim = dim3(TB);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  FST_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
  return FST_OK;
}

}  // namespace

extern "C" int fst_lattice_viterbi(fst_t* f, int32_t num_nodes, int32_t num_edges, const int32_t* from,
                                   const int32_t* to, const int32_t* label, const float* weight, float* best_score,
                                   int32_t* edge_path, int32_t* arc_path, int32_t* path_len) {
  if (!f || !best_score || !path_len || (num_nodes > 1 && (!edge_path || !arc_path))) {
    set_error("fst_lattice_viterbi: bad arguments");
    return FST_ERR_INVALID_ARG;
  }
  HostLattice H;
  int rc = check_lattice(f, num_nodes, num_edges, from, to, label, weight, &H);
  if (rc) return rc;
  DevGuard g(f->device);
  cudaStream_t s = 0;
  SliceView sv;
  if ((rc = slice_view(f, s, &sv))) return rc;
  const int64_t Q = f->Q, N = num_nodes, E = num_edges, np = std::max<int64_t>(N - 1, 1);
  EdgeTables T;
  T.add(sv, H.in_edge, num_edges, from, to, label, weight);
  Scratch mem;
  if ((rc = mem.take(f, Scratch::piece((N * Q + 2) * 8) + Scratch::piece(E * (int64_t)sizeof(EdgeRec)) +
                            Scratch::piece((E + 1) * 8) + Scratch::piece((N + 1) * 4) + Scratch::piece(E * 4) +
                            Scratch::piece((2 + 2 * np) * 4))))
    return rc;
  unsigned long long* keys = mem.get<unsigned long long>(N * Q + 2);
  EdgeRec* d_e = mem.get<EdgeRec>(E);
  int64_t* d_pre = mem.get<int64_t>(E + 1);
  int32_t* d_in = mem.get<int32_t>(N + 1);
  int32_t* d_label = mem.get<int32_t>(E);
  int32_t* d_out = mem.get<int32_t>(2 + 2 * np);
  if (E > 0) {
    FST_CUDA(cudaMemcpyAsync(d_e, T.e.data(), (size_t)E * sizeof(EdgeRec), cudaMemcpyHostToDevice, s));
    FST_CUDA(cudaMemcpyAsync(d_label, label, (size_t)E * 4, cudaMemcpyHostToDevice, s));
  }
  FST_CUDA(cudaMemcpyAsync(d_pre, T.pre.data(), (size_t)(E + 1) * 8, cudaMemcpyHostToDevice, s));
  FST_CUDA(cudaMemcpyAsync(d_in, H.in_off.data(), (size_t)(N + 1) * 4, cudaMemcpyHostToDevice, s));
  FST_CUDA(cudaMemsetAsync(keys, 0, (size_t)(N * Q + 2) * 8, s));
  const EdgeView G{d_e, d_pre};
  k_lat_vit_init<<<nb(Q), TB, 0, s>>>(f->theta_s, f->Q, keys);
  // node by node: every edge into v
  for (int32_t v = 1; v < N; ++v) {
    const int32_t lo = H.in_off[v], hi = H.in_off[v + 1];
    const int64_t n = T.pre[hi] - T.pre[lo];
    if (n && (rc = launch_arcs(k_lat_vit_node, n, f->num_sms, s, G, lo, hi, sv.arcs, sv.theta, f->Q, keys))) return rc;
  }
  k_lat_vit_final<<<std::min(nb(Q), (unsigned)f->num_sms), TB, 0, s>>>(view_of(f->bwd), G, d_in, d_label, keys, num_nodes,
                                                                       f->Q, f->theta_f, f->src_by_id, keys + N * Q, d_out);
  FST_CUDA(cudaGetLastError());
  std::vector<int32_t> h((size_t)(2 + 2 * np));
  FST_CUDA(cudaMemcpy(h.data(), d_out, h.size() * 4, cudaMemcpyDeviceToHost));
  memcpy(best_score, &h[0], 4);
  const int32_t len = h[1];
  if (len < 0) {
    set_error("fst_lattice_viterbi: the backtrace found no edge reaching the recorded score");
    return FST_ERR_STATE;
  }
  // the path was recorded from the end node back: reverse it
  for (int32_t i = 0; i < len; ++i) {
    edge_path[i] = h[(size_t)(2 + len - 1 - i)];
    arc_path[i] = h[(size_t)(2 + np + len - 1 - i)];
  }
  *path_len = len;
  if (*best_score == -INFINITY) {
    set_error("no accepting path");
    return FST_ERR_NO_PATH;
  }
  return FST_OK;
}

extern "C" int fst_lattice_forward_backward(fst_t* f, int32_t num_nodes, int32_t num_edges, const int32_t* from,
                                            const int32_t* to, const int32_t* label, const float* weight,
                                            double* log_z, float* arc_posteriors, float* edge_posteriors) {
  if (!f || !log_z) {
    set_error("fst_lattice_forward_backward: bad arguments");
    return FST_ERR_INVALID_ARG;
  }
  HostLattice H;
  int rc = check_lattice(f, num_nodes, num_edges, from, to, label, weight, &H);
  if (rc) return rc;
  DevGuard g(f->device);
  cudaStream_t s = 0;
  SliceView sv;
  if ((rc = slice_view(f, s, &sv))) return rc;
  const int64_t Q = f->Q, N = num_nodes, E = num_edges, A = f->A;
  EdgeTables T;  // by destination node, then by source node
  T.add(sv, H.in_edge, num_edges, from, to, label, weight);
  T.add(sv, H.out_edge, num_edges, from, to, label, weight);
  // the values of both passes, log Z (with its count of finished blocks and
  // their parts), and the counts of the arcs and the posteriors of the edges
  // side by side, as float64 and as float32
  Scratch mem;
  if ((rc = mem.take(f, Scratch::piece((2 * N * Q + (A + E + 3) / 2) * 16) + Scratch::piece((A + E) * 4 + 8) +
                            Scratch::piece(LOGZ_BLOCKS * (int64_t)sizeof(LogzPart)) +
                            Scratch::piece(2 * E * (int64_t)sizeof(EdgeRec)) + Scratch::piece(2 * (E + 1) * 8))))
    return rc;
  ulonglong2* alpha = mem.get<ulonglong2>(2 * N * Q + (A + E + 3) / 2);
  ulonglong2* beta = alpha + N * Q;
  double* d_logz = (double*)(beta + N * Q);
  uint32_t* d_done = (uint32_t*)(d_logz + 1);
  double* cnt = d_logz + 2;
  double* epost = cnt + A;
  float* out = mem.get<float>(A + E + 2);
  LogzPart* d_part = mem.get<LogzPart>(LOGZ_BLOCKS);
  EdgeRec* d_e = mem.get<EdgeRec>(2 * E);
  int64_t* d_pre = mem.get<int64_t>(2 * (E + 1));
  FST_CUDA(cudaMemsetAsync(alpha, 0, (size_t)(2 * N * Q) * 16 + 16 + (size_t)(A + E) * 8, s));
  if (E > 0) FST_CUDA(cudaMemcpyAsync(d_e, T.e.data(), (size_t)(2 * E) * sizeof(EdgeRec), cudaMemcpyHostToDevice, s));
  FST_CUDA(cudaMemcpyAsync(d_pre, T.pre.data(), (size_t)(2 * (E + 1)) * 8, cudaMemcpyHostToDevice, s));
  const EdgeView Gi{d_e, d_pre}, Go{d_e + E, d_pre + E + 1};
  const int64_t* pi = T.pre.data();
  const int64_t* po = T.pre.data() + E + 1;
  // node by node, forward and (for the posteriors) backward from the end
  const bool post = arc_posteriors || edge_posteriors;
  k_lat_lse_init<<<nb(Q), TB, 0, s>>>(f->theta_s, f->Q, alpha);
  if (post) k_lat_lse_init<<<nb(Q), TB, 0, s>>>(f->theta_f, f->Q, beta + (N - 1) * Q);
  for (int32_t v = 1; v < N; ++v) {
    const int32_t u = num_nodes - 1 - v;
    const StepSide F{Gi, H.in_off[v], H.in_off[v + 1], pi[H.in_off[v + 1]] - pi[H.in_off[v]], alpha};
    const StepSide B{Go, H.out_off[u], H.out_off[u + 1], post ? po[H.out_off[u + 1]] - po[H.out_off[u]] : 0, beta};
    if (F.n + B.n == 0) continue;
    if ((rc = launch_arcs(k_lat_lse_step<false>, F.n + B.n, f->num_sms, s, F, B, sv.arcs, sv.theta, f->Q)) ||
        (rc = launch_arcs(k_lat_lse_step<true>, F.n + B.n, f->num_sms, s, F, B, sv.arcs, sv.theta, f->Q)))
      return rc;
  }
  k_lat_logz<<<std::min(nb(Q), (unsigned)LOGZ_BLOCKS), TB, 0, s>>>(alpha + (N - 1) * Q, f->theta_f, f->Q, d_part, d_done,
                                                                    d_logz);
  if (post) {
    if (pi[E] && (rc = launch_arcs(k_lat_post, pi[E], f->num_sms, s, Gi, num_edges, sv.arcs, sv.theta, f->Q, alpha, beta,
                                   d_logz, cnt, epost)))
      return rc;
    if (A + E > 0)
      k_lat_to_f32<<<(unsigned)std::min<int64_t>(nb(A + E), 8 * (int64_t)f->num_sms), TB, 0, s>>>(cnt, A + E, out);
  }
  FST_CUDA(cudaGetLastError());
  FST_CUDA(cudaMemcpyAsync(log_z, d_logz, 8, cudaMemcpyDeviceToHost, s));
  if (arc_posteriors && A > 0)
    FST_CUDA(cudaMemcpyAsync(arc_posteriors, out, (size_t)A * 4, cudaMemcpyDeviceToHost, s));
  if (edge_posteriors && E > 0)
    FST_CUDA(cudaMemcpyAsync(edge_posteriors, out + A, (size_t)E * 4, cudaMemcpyDeviceToHost, s));
  FST_CUDA(cudaStreamSynchronize(s));
  if (*log_z == -INFINITY) {
    set_error("no accepting path");
    return FST_ERR_NO_PATH;
  }
  return FST_OK;
}
