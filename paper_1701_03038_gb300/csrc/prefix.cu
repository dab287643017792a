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
// Q^2 exponentials a product where adding the logs one by one takes Q^3.  A
// sum so small that terms may have underflowed (the largest A + B far below
// r + c) is taken again in the log domain.  The Viterbi score is the best
// path's weight with its float32 additions associated in tree order rather
// than left to right.
//
// A level of the tree is one launch over its products, both semirings side by
// side.  What bounds a call on 64 states and 1,000 symbols is the chain of
// its ten levels; all products together are 0.5 GFLOP.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "fst_internal.cuh"

using namespace fstgpu;

namespace {

constexpr int TB = 256;
constexpr int TILE = 64;   // output tile TILE x TILE, 4 x 4 entries a thread
constexpr int KC = 64;     // k chunk staged in shared memory
constexpr int PREFIX_MAX_STATES = 512;
// sums below this may have lost terms to underflow (a lost term is below
// 2^-126, and there are at most 512 of them)
constexpr float TINY = 1e-30f;

__device__ __forceinline__ float neg_inf() { return __int_as_float(0xff800000); }

__global__ void k_fill(float* __restrict__ p, int64_t n, float v) {
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
// for every p (blockIdx.y), one TILE x TILE tile of the result per block
// (blockIdx.x), the log-sum and the max-plus products side by side
// (blockIdx.z).  The matrices below are in[slot[k]] (slot null: in[k]); a
// last matrix without a partner is carried up as it is.
__global__ void __launch_bounds__(TB) k_mul(const float* __restrict__ in_sum, const float* __restrict__ in_max,
                                            const int32_t* __restrict__ slot, int32_t count,
                                            float* __restrict__ out_sum, float* __restrict__ out_max, int32_t Q) {
  __shared__ float As[KC][TILE + 1];  // A transposed: [k][row]
  __shared__ float Bs[KC][TILE + 1];
  __shared__ float rmax[TILE], cmax[TILE];
  const bool maxplus = blockIdx.z != 0;
  const int64_t QQ = (int64_t)Q * Q;
  const float* in = maxplus ? in_max : in_sum;
  float* out = (maxplus ? out_max : out_sum) + (int64_t)blockIdx.y * QQ;
  const int32_t ka = 2 * blockIdx.y, kb = ka + 1;
  const float* A = in + (slot ? slot[ka] : ka) * QQ;
  const int32_t tiles = (Q + TILE - 1) / TILE;
  const int32_t i0 = ((int32_t)blockIdx.x / tiles) * TILE, j0 = ((int32_t)blockIdx.x % tiles) * TILE;
  if (kb >= count) {
    for (int32_t e = threadIdx.x; e < TILE * TILE; e += TB) {
      const int32_t i = i0 + e / TILE, j = j0 + e % TILE;
      if (i < Q && j < Q) out[(int64_t)i * Q + j] = A[(int64_t)i * Q + j];
    }
    return;
  }
  const float* B = in + (slot ? slot[kb] : kb) * QQ;
  // (the thread's 4 x 4 entries: rows ty + 16 u, columns tx + 16 v)
  const int32_t tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto load = [&](int32_t k0) {
    for (int32_t e = threadIdx.x; e < TILE * KC; e += TB) {
      const int32_t i = i0 + e / KC, k = k0 + e % KC;
      As[e % KC][e / KC] = (i < Q && k < Q) ? __ldg(A + (int64_t)i * Q + k) : neg_inf();
      const int32_t kk = k0 + e / TILE, j = j0 + e % TILE;
      Bs[e / TILE][e % TILE] = (kk < Q && j < Q) ? __ldg(B + (int64_t)kk * Q + j) : neg_inf();
    }
  };
  if (!maxplus) {
    // row and column maxima (0 stands for -inf: nothing to scale)
    for (int32_t r = warp; r < TILE; r += TB / 32) {
      float m = neg_inf(), c = neg_inf();
      for (int32_t k = lane; k < Q; k += 32) {
        if (i0 + r < Q) m = fmaxf(m, __ldg(A + (int64_t)(i0 + r) * Q + k));
        if (j0 + r < Q) c = fmaxf(c, __ldg(B + (int64_t)k * Q + j0 + r));
      }
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(FULL, m, d));
        c = fmaxf(c, __shfl_xor_sync(FULL, c, d));
      }
      if (lane == 0) {
        rmax[r] = m;
        cmax[r] = c;
      }
    }
    __syncthreads();
  }
  float acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = maxplus ? neg_inf() : 0.f;
  for (int32_t k0 = 0; k0 < Q; k0 += KC) {
    if (k0 > 0) __syncthreads();
    load(k0);
    __syncthreads();
    if (!maxplus) {
      for (int32_t e = threadIdx.x; e < TILE * KC; e += TB) {
        const int32_t k = e / TILE, x = e % TILE;
        const float a = As[k][x], b = Bs[k][x];
        As[k][x] = a == neg_inf() ? 0.f : expf(a - rmax[x]);
        Bs[k][x] = b == neg_inf() ? 0.f : expf(b - cmax[x]);
      }
      __syncthreads();
    }
    const int32_t kn = min(KC, Q - k0);
#pragma unroll 4
    for (int32_t k = 0; k < kn; ++k) {
      float a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = As[k][ty + 16 * u];
        b[u] = Bs[k][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = maxplus ? fmaxf(acc[u][v], a[u] + b[v]) : fmaf(a[u], b[v], acc[u][v]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int32_t i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
      if (i >= Q || j >= Q) continue;
      float r = acc[u][v];
      if (!maxplus) {
        const float rm = rmax[ty + 16 * u], cm = cmax[tx + 16 * v];
        if (rm == neg_inf() || cm == neg_inf()) {
          r = neg_inf();
        } else if (r >= TINY) {
          r = rm + cm + logf(r);
        } else {
          // terms may have underflowed: the log-sum one by one
          float m = neg_inf(), s = 0.f;
          for (int32_t k = 0; k < Q; ++k) {
            const float x = __ldg(A + (int64_t)i * Q + k), y = __ldg(B + (int64_t)k * Q + j);
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

// log Z = LSE_{i,j}(theta_s[i] + P[i][j] + theta_f[j]) (float64) and the
// best score max_{i,j} fl(fl(theta_s[i] + V[i][j]) + theta_f[j]); one block.
// P == nullptr: the empty string (P and V the identity of their semiring).
__global__ void k_close(const float* __restrict__ P, const float* __restrict__ V, int32_t Q,
                        const float* __restrict__ ts, const float* __restrict__ tf, double* __restrict__ logz,
                        float* __restrict__ best) {
  __shared__ double red[TB / 32];
  __shared__ float redf[TB / 32];
  const int64_t QQ = (int64_t)Q * Q;
  auto val = [&](int64_t e, bool vit) -> float {
    const int32_t i = (int32_t)(e / Q), j = (int32_t)(e % Q);
    const float m = P ? (vit ? V[e] : P[e]) : (i == j ? 0.f : neg_inf());
    if (ts[i] == neg_inf() || m == neg_inf() || tf[j] == neg_inf()) return neg_inf();
    return __fadd_rn(__fadd_rn(ts[i], m), tf[j]);
  };
  double mx = -INFINITY;
  float bf = neg_inf();
  for (int64_t e = threadIdx.x; e < QQ; e += TB) {
    const int32_t i = (int32_t)(e / Q), j = (int32_t)(e % Q);
    const float m = P ? P[e] : (i == j ? 0.f : neg_inf());
    if (ts[i] != neg_inf() && m != neg_inf() && tf[j] != neg_inf())
      mx = fmax(mx, (double)ts[i] + (double)m + (double)tf[j]);
    bf = fmaxf(bf, val(e, true));
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    mx = fmax(mx, __shfl_xor_sync(FULL, mx, d));
    bf = fmaxf(bf, __shfl_xor_sync(FULL, bf, d));
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = mx;
    redf[threadIdx.x >> 5] = bf;
  }
  __syncthreads();
  mx = red[0];
  bf = redf[0];
  for (int w = 1; w < TB / 32; ++w) {
    mx = fmax(mx, red[w]);
    bf = fmaxf(bf, redf[w]);
  }
  __syncthreads();
  double sum = 0.0;
  if (mx != -INFINITY)
    for (int64_t e = threadIdx.x; e < QQ; e += TB) {
      const int32_t i = (int32_t)(e / Q), j = (int32_t)(e % Q);
      const float m = P ? P[e] : (i == j ? 0.f : neg_inf());
      if (ts[i] != neg_inf() && m != neg_inf() && tf[j] != neg_inf())
        sum += exp((double)ts[i] + (double)m + (double)tf[j] - mx);
    }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) sum += __shfl_xor_sync(FULL, sum, d);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < TB / 32; ++w) t += red[w];
    *logz = mx == -INFINITY ? -INFINITY : mx + log(t);
    *best = bf;
  }
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
  struct Out {
    double logz;
    float best, pad;
  } h;
  if (n == 0) {
    if ((rc = mem.take(f, Scratch::piece(sizeof(Out))))) return rc;
    Out* d_out = mem.get<Out>(1);
    k_close<<<1, TB, 0, s>>>(nullptr, nullptr, f->Q, f->theta_s, f->theta_f, &d_out->logz, &d_out->best);
    FST_CUDA(cudaGetLastError());
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
        dsum, 2 * U * QQ, -INFINITY);
    for (int64_t u0 = 0; u0 < U; u0 += 65535)
      k_dense<<<dim3((unsigned)std::min<int64_t>((longest + TB - 1) / TB, 64), (unsigned)std::min<int64_t>(65535, U - u0)),
                TB, 0, s>>>(sv.arcs, sv.theta, slice_sym_win(f), d_slot + n + u0, f->Q, dsum + u0 * QQ,
                            dmax + u0 * QQ);
    FST_CUDA(cudaGetLastError());
    // the product tree: level by level, adjacent pairs multiplied
    const float *cur_s = dsum, *cur_m = dmax;
    const int32_t* slot = d_slot;
    int64_t count = n;
    const int32_t tiles = (int32_t)((Q + TILE - 1) / TILE);
    for (int level = 0; count > 1 || slot; ++level) {
      float *out_s = buf_s[level & 1], *out_m = buf_m[level & 1];
      const int64_t pairs = (count + 1) / 2;
      for (int64_t p0 = 0; p0 < pairs; p0 += 65535) {
        const int64_t cnt = std::min<int64_t>(65535, pairs - p0);
        k_mul<<<dim3((unsigned)(tiles * tiles), (unsigned)cnt, 2), TB, 0, s>>>(
            slot ? cur_s : cur_s + 2 * p0 * QQ, slot ? cur_m : cur_m + 2 * p0 * QQ, slot ? slot + 2 * p0 : nullptr,
            (int32_t)(count - 2 * p0), out_s + p0 * QQ, out_m + p0 * QQ, f->Q);
      }
      cur_s = out_s;
      cur_m = out_m;
      slot = nullptr;
      count = pairs;
    }
    k_close<<<1, TB, 0, s>>>(cur_s, cur_m, f->Q, f->theta_s, f->theta_f, &d_out->logz, &d_out->best);
    FST_CUDA(cudaGetLastError());
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
