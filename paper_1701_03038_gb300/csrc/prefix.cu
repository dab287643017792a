// prefix.cu -- the weight of a string by a parallel product over time.
//
// Eq. 1 is a product of the matrices delta[w_1] ... delta[w_n] between the
// start and final vectors.  Instead of a sweep over the positions, the
// matrices can be multiplied pairwise in parallel, and the products again,
// until one matrix is left (the parallel prefix approach of Sec. 6.1, which
// the paper leaves for future work).  Each product costs Q^3 instead of the
// Q^2 of a matrix-vector step, so this pays only for small dense FSTs and
// long strings: it takes log2(n) dependent rounds instead of n.
//
// Matrices are dense Q x Q log-weights (-inf = no arc), one per symbol of
// the string (parallel arcs combined: log-sum for the weight, max for the
// best path).  A product entry is log sum_k exp(A[i][k] + B[k][j]) or max_k
// A[i][k] + B[k][j].  The sums are taken in the linear domain: with r_i the
// largest entry of row i and c_j that of column j, exp(A - r) and exp(B - c)
// are multiplied as matrices and r_i + c_j + log of the sum is the entry --
// Q^2 exponentials a product where adding the logs one by one takes Q^3.
// (logprod.cuh keeps the errors down: over 40 HMMs each of 16, 40 and 64
// states, their weights plain or scaled by up to e^8, and 64 to 1,000 symbols,
// the mean error of log Z against float64 is 0.20 to 0.86 of what log-sums
// taken term by term give; with expf and rounded sums it is up to 2.1 of it,
// and a call takes 134 us in place of 138.)  A sum so small that terms may
// have underflowed (the largest A + B far below r + c) is taken again in the
// log domain.  The Viterbi score is the best path's weight with its float32
// additions associated in tree order rather
// than left to right.
//
// A level of the tree is one launch over its products, both semirings side by
// side.  What bounds a call on 64 states and 1,000 symbols is the chain of
// its ten levels; all products together are 0.5 GFLOP.
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "frontier.cuh"
#include "fst_internal.cuh"
#include "logprod.cuh"

using namespace fstgpu;

namespace {

constexpr int TB = 256;
constexpr int KC = 64;     // k chunk staged in shared memory
constexpr int PREFIX_MAX_STATES = 512;
// sums below this may have lost terms to underflow (a lost term is below
// 2^-126, and the at most 512 of them below half a rounding of this)
constexpr float TINY = 1e-28f;

__global__ void k_fill(float* __restrict__ p, int64_t n, float v, uint32_t* __restrict__ zero) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *zero = 0u;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

// log(e^a + e^b) with -inf handled.
__device__ __forceinline__ float log_add(float a, float b) {
  if (a == neg_inf()) return b;
  if (b == neg_inf()) return a;
  const float hi = fmaxf(a, b), lo = fminf(a, b);
  return hi + log1pf(expf(lo - hi));
}

// The dense matrices of the symbols syms[blockIdx.y] (both filled with
// -inf): every arc of the slice adds into M[src][dst] (log-sum: a
// compare-and-swap loop; max: atomics on the float's bits, ordered as
// integers for v >= 0 and reversed as unsigned ones below).
__global__ void k_dense(const int4* __restrict__ arcs, const float* __restrict__ theta,
                        const int64_t* __restrict__ sym_win, const int32_t* __restrict__ syms, int32_t Q,
                        float* __restrict__ msum, float* __restrict__ mmax) {
  const int32_t a = syms[blockIdx.y];
  const int64_t i1 = sym_win[a + 1] * WIN;
  for (int64_t i = sym_win[a] * WIN + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < i1;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int4 r = __ldg(arcs + i);
    if (r.z < 0) continue;
    const float th = __ldg(theta + i);
    if (th == neg_inf()) continue;
    const int64_t e = (int64_t)blockIdx.y * Q * Q + (int64_t)r.x * Q + r.y;
    if (th >= 0.f) atomicMax((int*)(mmax + e), __float_as_int(th));
    else atomicMin((unsigned int*)(mmax + e), __float_as_uint(th));
    unsigned int* u = (unsigned int*)(msum + e);
    unsigned int old = *u, seen;
    do {
      seen = old;
      const float v = log_add(__uint_as_float(seen), th);
      if (__float_as_uint(v) == seen) break;
      old = atomicCAS(u, seen, __float_as_uint(v));
    } while (old != seen);
  }
}

// One level of the tree: matrix 2p times matrix 2p + 1 of the level below,
// for every p (blockIdx.y), one T x T tile of the result per block
// (blockIdx.x), the log-sum and the max-plus products side by side
// (blockIdx.z).  The matrices below are in[slot[k]] (slot null: in[k]); a
// last matrix without a partner is carried up as it is.
//
// A thread holds T / 16 x T / 16 entries and reads both operands from shared
// memory as vectors, four k at a time.  T = 64 needs the fewest reads and
// exponentials a product; T = 32 spreads a product over four times the
// blocks, for the levels that have too few to fill the GPU (the last eight
// of ten on 64 states and 1,000 symbols).
struct MulArgs {
  const float *in_sum, *in_max;
  const int32_t* slot;
  float *out_sum, *out_max;
  int32_t count, Q;
};
template <int N>
struct alignas(4 * N) Vec {
  float v[N];
};
template <int T>
struct alignas(16) MulShared {
  static constexpr int PARTS = TB / T;
  float A[T][KC + 4], B[KC][T + 4];
  float rmax[T], cmax[T], part[PARTS][T];
};
// The rows that a thread reads as vectors: four of A at once, T / 16 of B.
template <class S>
constexpr bool vector_rows(int r) {
  return alignof(S) % alignof(Vec<4>) == 0 && offsetof(S, A) % alignof(Vec<4>) == 0 &&
         sizeof(S::A[0]) % alignof(Vec<4>) == 0 && offsetof(S, B) % (4 * r) == 0 && sizeof(S::B[0]) % (4 * r) == 0;
}
static_assert(vector_rows<MulShared<32>>(2) && vector_rows<MulShared<64>>(4), "vector reads need aligned rows");

template <int T, bool MAX>
__device__ __forceinline__ void mul_tile(MulShared<T>& sh, const float* A, const float* B, float* out, int32_t i0, int32_t j0, int32_t Q) {
  constexpr int R = T / 16, PARTS = MulShared<T>::PARTS, LOADS = T * KC / TB;
  const int32_t t = threadIdx.x, tx = t % 16, ty = t / 16;
  auto load = [&](int32_t k0) {
    float a[LOADS], b[LOADS];
#pragma unroll
    for (int u = 0; u < LOADS; ++u) {
      const int32_t e = t + u * TB, i = i0 + e / KC, k = k0 + e % KC, kk = k0 + e / T, j = j0 + e % T;
      a[u] = i < Q && k < Q ? __ldcg(A + (int64_t)i * Q + k) : neg_inf();
      b[u] = kk < Q && j < Q ? __ldcg(B + (int64_t)kk * Q + j) : neg_inf();
    }
#pragma unroll
    for (int u = 0; u < LOADS; ++u) {
      const int32_t e = t + u * TB;
      sh.A[e / KC][e % KC] = a[u];
      sh.B[e / T][e % T] = b[u];
    }
  };
  const bool once = Q <= KC;
  load(0);
  __syncthreads();
  if (!MAX) {
    // row and column maxima: PARTS threads a row (neighbours) and a column
    const int32_t row = t / PARTS, rp = t % PARTS, col = t % T, cp = t / T;
    float m = neg_inf(), c = neg_inf();
    for (int32_t k0 = 0;;) {
#pragma unroll 8
      for (int k = 0; k < KC; k += PARTS) {
        m = fmaxf(m, sh.A[row][k + rp]);
        c = fmaxf(c, sh.B[k + cp][col]);
      }
      if ((k0 += KC) >= Q) break;
      __syncthreads();
      load(k0);
      __syncthreads();
    }
#pragma unroll
    for (int d = PARTS / 2; d >= 1; d >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, d));
    if (rp == 0) sh.rmax[row] = scale_of(m);
    sh.part[cp][col] = c;
    __syncthreads();
    if (t < T) {
      c = sh.part[0][t];
#pragma unroll
      for (int p = 1; p < PARTS; ++p) c = fmaxf(c, sh.part[p][t]);
      sh.cmax[t] = scale_of(c);
    }
    __syncthreads();
  }
  float acc[R][R];
#pragma unroll
  for (int u = 0; u < R; ++u)
#pragma unroll
    for (int v = 0; v < R; ++v) acc[u][v] = MAX ? neg_inf() : 0.f;
  for (int32_t k0 = 0; k0 < Q; k0 += KC) {
    if (!once && (k0 > 0 || !MAX)) {
      __syncthreads();
      load(k0);
      __syncthreads();
    }
    if (!MAX) {
#pragma unroll
      for (int u = 0; u < LOADS; ++u) {
        const int32_t e = t + u * TB;
        float& a = sh.A[e / KC][e % KC];
        float& b = sh.B[e / T][e % T];
        a = exp_below(a, sh.rmax[e / KC]);
        b = exp_below(b, sh.cmax[e % T]);
      }
      __syncthreads();
    }
    // (past Q the operands are 0, or -inf: they change nothing)
    const int32_t kn = min(KC, (Q - k0 + 3) & ~3);
    for (int32_t k = 0; k < kn; k += 4) {
      Vec<4> a[R];
      Vec<R> b[4];
#pragma unroll
      for (int u = 0; u < R; ++u) a[u] = *(const Vec<4>*)&sh.A[R * ty + u][k];
#pragma unroll
      for (int x = 0; x < 4; ++x) b[x] = *(const Vec<R>*)&sh.B[k + x][R * tx];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int u = 0; u < R; ++u)
#pragma unroll
          for (int v = 0; v < R; ++v)
            acc[u][v] = MAX ? fmaxf(acc[u][v], a[u].v[x] + b[x].v[v]) : fmaf(a[u].v[x], b[x].v[v], acc[u][v]);
    }
  }
#pragma unroll
  for (int u = 0; u < R; ++u) {
#pragma unroll
    for (int v = 0; v < R; ++v) {
      const int32_t i = i0 + R * ty + u, j = j0 + R * tx + v;
      if (i >= Q || j >= Q) continue;
      float r = acc[u][v];
      if (!MAX) {
        const float rm = sh.rmax[R * ty + u], cm = sh.cmax[R * tx + v];
        if (rm == neg_inf() || cm == neg_inf()) {
          r = neg_inf();
        } else if (r >= TINY) {
          r = add_log(rm, cm, r);
        } else {
          // terms may have underflowed: the log-sum one by one
          float m = neg_inf(), s = 0.f;
          for (int32_t k = 0; k < Q; ++k) {
            const float x = __ldcg(A + (int64_t)i * Q + k), y = __ldcg(B + (int64_t)k * Q + j);
            if (x == neg_inf() || y == neg_inf()) continue;
            const float w = x + y;
            if (w > m) {
              s = s * expf(m - w) + 1.f;  // m == -inf gives s * 0 + 1
              m = w;
            } else {
              s += expf(w - m);
            }
          }
          r = m == neg_inf() ? m : m + logf(s);
        }
      }
      out[(int64_t)i * Q + j] = r;
    }
  }
}

template <int T>
__global__ void __launch_bounds__(TB, 3) k_mul(const MulArgs M) {
  __shared__ MulShared<T> sh;
  // (what the level below wrote is read with __ldcg: read-only loads may be
  // moved up, over the wait)
  chain_enter();
  const bool maxplus = blockIdx.z != 0;
  const int32_t Q = M.Q;
  const int64_t QQ = (int64_t)Q * Q;
  const float* in = maxplus ? M.in_max : M.in_sum;
  float* out = (maxplus ? M.out_max : M.out_sum) + (int64_t)blockIdx.y * QQ;
  const int32_t ka = 2 * blockIdx.y, kb = ka + 1;
  const float* A = in + (M.slot ? M.slot[ka] : ka) * QQ;
  const int32_t tiles = (Q + T - 1) / T;
  const int32_t i0 = ((int32_t)blockIdx.x / tiles) * T, j0 = ((int32_t)blockIdx.x % tiles) * T;
  if (kb >= M.count) {
    for (int32_t e = threadIdx.x; e < T * T; e += TB) {
      const int32_t i = i0 + e / T, j = j0 + e % T;
      if (i < Q && j < Q) out[(int64_t)i * Q + j] = __ldcg(A + (int64_t)i * Q + j);
    }
    return;
  }
  const float* B = in + (M.slot ? M.slot[kb] : kb) * QQ;
  if (maxplus) mul_tile<T, true>(sh, A, B, out, i0, j0, Q);
  else mul_tile<T, false>(sh, A, B, out, i0, j0, Q);
}

// What a call returns, and the blocks' parts of it.
struct Part {
  double m, sum;  // largest term, sum of exp(term - m)
  float best, pad;
};
constexpr int CLOSE_BLOCKS = 64;
struct Out {
  double logz;
  float best;
  uint32_t done;
  Part part[CLOSE_BLOCKS];
};

// log Z = LSE_{i,j}(theta_s[i] + P[i][j] + theta_f[j]) (float64) and the
// best score max_{i,j} fl(fl(theta_s[i] + V[i][j]) + theta_f[j]).  A warp
// takes a row at a time (rows of no start state cost one read), a block its
// warps' rows, the last block to finish the blocks' parts in their order.
// P == nullptr: the empty string (P and V the identity of their semiring).
__device__ __forceinline__ void add_terms(double& m, double& s, double m2, double s2) {
  if (m2 == -INFINITY) return;
  if (m == -INFINITY) {
    m = m2;
    s = s2;
    return;
  }
  const double x = fmax(m, m2);
  s = (m == x ? s : s * exp(m - x)) + (m2 == x ? s2 : s2 * exp(m2 - x));
  m = x;
}
__global__ void __launch_bounds__(TB) k_close(const float* P, const float* V, int32_t Q,
                                              const float* __restrict__ ts, const float* __restrict__ tf,
                                              Out* __restrict__ o) {
  constexpr int WARPS = TB / 32;
  __shared__ Part part[WARPS];
  __shared__ bool last;
  chain_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double m = -INFINITY, s = 0.0;
  float best = neg_inf();
  for (int32_t i = (int32_t)blockIdx.x * WARPS + warp; i < Q; i += (int32_t)gridDim.x * WARPS) {
    const float si = __ldg(ts + i);
    if (si == neg_inf()) continue;
    auto term = [&](int32_t j) -> double {
      const float f = __ldg(tf + j), p = P ? __ldcg(P + (int64_t)i * Q + j) : (i == j ? 0.f : neg_inf());
      return p == neg_inf() || f == neg_inf() ? -INFINITY : (double)si + (double)p + (double)f;
    };
    double rm = -INFINITY, rs = 0.0;
    for (int32_t j = lane; j < Q; j += 32) {
      rm = fmax(rm, term(j));
      const float f = __ldg(tf + j), v = P ? __ldcg(V + (int64_t)i * Q + j) : (i == j ? 0.f : neg_inf());
      if (v != neg_inf() && f != neg_inf()) best = fmaxf(best, __fadd_rn(__fadd_rn(si, v), f));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) rm = fmax(rm, __shfl_xor_sync(FULL, rm, d));
    if (rm == -INFINITY) continue;
    for (int32_t j = lane; j < Q; j += 32) {
      const double x = term(j);
      if (x != -INFINITY) rs += exp(x - rm);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) rs += __shfl_xor_sync(FULL, rs, d);
    add_terms(m, s, rm, rs);
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) best = fmaxf(best, __shfl_xor_sync(FULL, best, d));
  if (lane == 0) part[warp] = Part{m, s, best, 0.f};
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < WARPS; ++w) {
      add_terms(m, s, part[w].m, part[w].sum);
      best = fmaxf(best, part[w].best);
    }
    if (gridDim.x > 1) {
      o->part[blockIdx.x] = Part{m, s, best, 0.f};
      __threadfence();
      last = atomicAdd(&o->done, 1u) + 1u == gridDim.x;
    }
  }
  // (the last block, or the only one)
  if (threadIdx.x >= 32) return;
  if (gridDim.x > 1) {
    __syncwarp();
    if (!last) return;
    __threadfence();
    // its first warp adds the parts up, two a lane at most, in a fixed order
    m = -INFINITY;
    s = 0.0;
    best = neg_inf();
    for (unsigned b = lane; b < gridDim.x; b += 32) {
      const Part* q = o->part + b;
      add_terms(m, s, __ldcg(&q->m), __ldcg(&q->sum));
      best = fmaxf(best, __ldcg(&q->best));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
      const double m2 = __shfl_xor_sync(FULL, m, d), s2 = __shfl_xor_sync(FULL, s, d);
      add_terms(m, s, m2, s2);
      best = fmaxf(best, __shfl_xor_sync(FULL, best, d));
    }
  }
  if (lane == 0) {
    o->logz = m == -INFINITY ? -INFINITY : m + log(s);
    o->best = best;
  }
}

// A launch that begins while the one before it drains (chain_enter waits for it).
template <class... KArgs, class... Args>
int launch_after(void (*kernel)(KArgs...), dim3 grid, cudaStream_t s, Args... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(TB);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  FST_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
  return FST_OK;
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

// Window offsets of the symbols on the device, in the order slice_view
// chose.
inline const int64_t* slice_sym_win(const fst_s* f) {
  return f->slice_order == FST_SLICE_BY_SOURCE ? f->bwd.sym_win : f->fwd.sym_win;
}

}  // namespace

extern "C" int fst_prefix_log_z(fst_t* f, const int32_t* ids, int32_t n, double* log_z, float* best_score) {
  if (!f || n < 0 || (n > 0 && !ids) || !log_z || !best_score) {
    set_error("fst_prefix_log_z: bad arguments");
    return FST_ERR_INVALID_ARG;
  }
  if (f->Q > PREFIX_MAX_STATES) {
    set_error("fst_prefix_log_z: %d states; the dense product is for at most %d", f->Q, PREFIX_MAX_STATES);
    return FST_ERR_UNSUPPORTED;
  }
  for (int32_t i = 0; i < n; ++i)
    if (ids[i] < 0 || ids[i] >= f->m) {
      set_error("symbol %d at position %d is outside [0, %d)", ids[i], i, f->m);
      return FST_ERR_INVALID_ARG;
    }
  DevGuard g(f->device);
  cudaStream_t s = 0;
  const int64_t Q = f->Q, QQ = Q * Q;
  int rc;
  Scratch mem;
  struct {
    double logz;
    float best, pad;
  } h;
  if (n == 0) {
    if ((rc = mem.take(f, Scratch::piece(sizeof(Out))))) return rc;
    Out* d_out = mem.get<Out>(1);
    FST_CUDA(cudaMemsetAsync(&d_out->done, 0, sizeof(d_out->done), s));
    if ((rc = launch_after(k_close, dim3((unsigned)std::min<int64_t>((Q + 7) / 8, CLOSE_BLOCKS)), s, (const float*)nullptr,
                           (const float*)nullptr, f->Q, (const float*)f->theta_s, (const float*)f->theta_f, d_out)))
      return rc;
    FST_CUDA(cudaMemcpy(&h, d_out, sizeof(h), cudaMemcpyDeviceToHost));
  } else {
    SliceView sv;
    if ((rc = slice_view(f, s, &sv))) return rc;
    // one dense pair (log-sum, max) per distinct symbol: the matrix of each
    // position, then the symbols, in one upload
    std::vector<int32_t> syms(ids, ids + n), up((size_t)n);
    std::sort(syms.begin(), syms.end());
    syms.erase(std::unique(syms.begin(), syms.end()), syms.end());
    int64_t longest = 1;
    for (int32_t i = 0; i < n; ++i)
      up[i] = (int32_t)(std::lower_bound(syms.begin(), syms.end(), ids[i]) - syms.begin());
    for (const int32_t a : syms) longest = std::max(longest, (sv.h_sym_win[a + 1] - sv.h_sym_win[a]) * (int64_t)WIN);
    const int64_t U = (int64_t)syms.size(), l1 = ((int64_t)n + 1) / 2, l2 = (l1 + 1) / 2;
    // The first level's products are those of pairs of symbols: with few
    // symbols (U^2 at most half of the pairs) each pair that occurs is
    // multiplied once, and the second level names its operands.  (500
    // products of 64 states: 42 us, the 36 of 6 symbols: 8.)
    const int64_t pairs = n / 2;
    int64_t uniq = 0;  // distinct pairs (0: every pair by itself)
    std::vector<int32_t> slot2;
    if (pairs >= 2 && U * U <= pairs / 2) {
      std::vector<int32_t> id((size_t)(U * U), -1), first;
      for (int64_t p = 0; p < pairs; ++p) {
        int32_t& k = id[(size_t)(up[2 * p] * U + up[2 * p + 1])];
        if (k < 0) {
          k = (int32_t)uniq++;
          first.push_back(up[2 * p]);
          first.push_back(up[2 * p + 1]);
        }
        slot2.push_back(k);
      }
      if (n & 1) {
        first.push_back(up[n - 1]);
        slot2.push_back((int32_t)uniq);
      }
      up = first;
    }
    const int64_t count0 = (int64_t)up.size();
    up.insert(up.end(), slot2.begin(), slot2.end());
    const int64_t at_syms = (int64_t)up.size();
    up.insert(up.end(), syms.begin(), syms.end());
    if ((rc = mem.take(f, Scratch::piece(sizeof(Out)) + Scratch::piece((int64_t)up.size() * 4) +
                              Scratch::piece(2 * U * QQ * 4) + 2 * Scratch::piece(l1 * QQ * 4) +
                              2 * Scratch::piece(l2 * QQ * 4))))
      return rc;
    Out* d_out = mem.get<Out>(1);
    int32_t* d_slot = mem.get<int32_t>((int64_t)up.size());
    float* dsum = mem.get<float>(2 * U * QQ);
    float* dmax = dsum + U * QQ;
    // the levels' results take turns: the odd levels' in the larger buffers
    float* buf_s[2] = {mem.get<float>(l1 * QQ), mem.get<float>(l2 * QQ)};
    float* buf_m[2] = {mem.get<float>(l1 * QQ), mem.get<float>(l2 * QQ)};
    FST_CUDA(cudaMemcpyAsync(d_slot, up.data(), up.size() * 4, cudaMemcpyHostToDevice, s));
    k_fill<<<(unsigned)std::min<int64_t>((2 * U * QQ + TB - 1) / TB, 8 * (int64_t)f->num_sms), TB, 0, s>>>(
        dsum, 2 * U * QQ, -INFINITY, &d_out->done);
    for (int64_t u0 = 0; u0 < U; u0 += 65535)
      k_dense<<<dim3((unsigned)std::min<int64_t>((longest + TB - 1) / TB, 64), (unsigned)std::min<int64_t>(65535, U - u0)),
                TB, 0, s>>>(sv.arcs, sv.theta, slice_sym_win(f), d_slot + at_syms + u0, f->Q, dsum + u0 * QQ,
                            dmax + u0 * QQ);
    FST_CUDA(cudaGetLastError());
    // the product tree: level by level, adjacent pairs multiplied
    const float *cur_s = dsum, *cur_m = dmax;
    const int32_t* slot = d_slot;
    int64_t count = count0;
    for (int level = 0; count > 1 || slot; ++level) {
      float *out_s = buf_s[level & 1], *out_m = buf_m[level & 1];
      const int64_t pairs = (count + 1) / 2;
      for (int64_t p0 = 0; p0 < pairs; p0 += 65535) {
        const int64_t cnt = std::min<int64_t>(65535, pairs - p0);
        const MulArgs M{slot ? cur_s : cur_s + 2 * p0 * QQ, slot ? cur_m : cur_m + 2 * p0 * QQ,
                        slot ? slot + 2 * p0 : nullptr, out_s + p0 * QQ, out_m + p0 * QQ, (int32_t)(count - 2 * p0), f->Q};
        const int32_t t64 = (f->Q + 63) / 64, t32 = (f->Q + 31) / 32;
        // (the large tiles once they fill every SM twice)
        rc = 2 * cnt * t64 * t64 >= 2 * f->num_sms
                 ? launch_after(k_mul<64>, dim3((unsigned)(t64 * t64), (unsigned)cnt, 2), s, M)
                 : launch_after(k_mul<32>, dim3((unsigned)(t32 * t32), (unsigned)cnt, 2), s, M);
        if (rc) return rc;
      }
      cur_s = out_s;
      cur_m = out_m;
      slot = uniq && level == 0 ? d_slot + count0 : nullptr;
      count = slot ? (int64_t)slot2.size() : pairs;
    }
    if ((rc = launch_after(k_close, dim3((unsigned)std::min<int64_t>((Q + 7) / 8, CLOSE_BLOCKS)), s, cur_s, cur_m, f->Q,
                           (const float*)f->theta_s, (const float*)f->theta_f, d_out)))
      return rc;
    FST_CUDA(cudaMemcpy(&h, d_out, sizeof(h), cudaMemcpyDeviceToHost));
  }
  *log_z = h.logz;
  *best_score = h.best;
  if (*log_z == -INFINITY) {
    set_error("no accepting path");
    return FST_ERR_NO_PATH;
  }
  return FST_OK;
}
