// frontier.cuh -- device helpers shared by the frontier kernels (kernels.cu:
// one launch per position over all strings; strings.cu: one warp or block
// per string over all positions).
#pragma once

#include "debug_record.cuh"
#include "kernels.cuh"

namespace fstgpu {

// Error bits of a run (FrontierState::flags[1]): the live pool overflowed,
// or a grid barrier of a persistent pass gave up waiting.
constexpr uint32_t ERR_POOL = 1u;
constexpr uint32_t ERR_TIMEOUT = 2u;
__device__ __forceinline__ int32_t run_error(uint32_t err) {
  return (err & ERR_TIMEOUT) ? FST_ERR_TIMEOUT : FST_ERR_OOM;
}

__device__ __forceinline__ float neg_inf() { return __int_as_float(0xff800000); }

// Bounds-checked build (FST_DEBUG): in_bounds(code, i, n) checks 0 <= i < n,
// and on a violation counts it, records the first (code, index, bound) and
// returns false so that the caller skips the access.  A normal build
// compiles every check away.
enum : int { CHK_STAGE = 1, CHK_POOL_WRITE = 2, CHK_POOL_READ = 3, CHK_ACC = 4, CHK_ARC = 5, CHK_TOKEN = 6 };
#ifdef FST_DEBUG
static __device__ unsigned long long g_dbg[4];  // violations, code, index, bound (one record per source file)
static __device__ __noinline__ bool in_bounds_slow(int code, long long i, long long n) {
  if (atomicAdd(&g_dbg[0], 1ull) == 0ull) {
    g_dbg[1] = (unsigned long long)code;
    g_dbg[2] = (unsigned long long)i;
    g_dbg[3] = (unsigned long long)n;
  }
  return false;
}
__device__ __forceinline__ bool in_bounds(int code, long long i, long long n) {
  return (i >= 0 && i < n) ? true : in_bounds_slow(code, i, n);
}
// (this file's record, read with the others')
static int debug_read_own(DebugCounts* out) {
  unsigned long long h[4] = {0, 0, 0, 0};
  FST_CUDA(cudaMemcpyFromSymbol(h, g_dbg, sizeof(h)));
  *out = DebugCounts{h[0], h[1], h[2], h[3]};
  for (unsigned long long& x : h) x = 0;
  FST_CUDA(cudaMemcpyToSymbol(g_dbg, h, sizeof(h)));
  return FST_OK;
}
static DebugRecord g_dbg_record(debug_read_own);
#else
__device__ __forceinline__ bool in_bounds(int, long long, long long) { return true; }
#endif

__device__ __forceinline__ float decode_max(uint32_t k) { return k ? fkey_inv(k) : neg_inf(); }

// Order key of a float64 value rounded to float32 (0 = -inf, nothing).
__device__ __forceinline__ uint32_t fkey64(double v) { return dead64(v) ? 0u : fkey(fx_narrow(v)); }

// The arcs out of state q on symbol a: their first position and count (0
// when none), from the (symbol, state) table.  In two steps, so that the
// loads of several lookups, or other work, go between them: seg_load reads
// the key's bucket (with FIRST the first arcs' records too), seg_find looks
// for the key in it, and further on where the bucket spilled.
struct Arcs {
  int32_t pos, len;
};
template <bool FIRST>
struct SegProbe {
  unsigned long long k;
  uint64_t b;
  ulonglong2 e0, e1;
  int4 f0, f1;
};
template <bool FIRST>
__device__ __forceinline__ void seg_load(const LayoutView& L, int32_t a, int32_t q, SegProbe<FIRST>& p) {
  p.k = seg_hash_key(a, q);
  p.b = seg_bucket(p.k, L.buckets);
  const SegSlot* s = L.seg_hash + 2 * p.b;
  p.e0 = __ldg((const ulonglong2*)&s[0].key);
  p.e1 = __ldg((const ulonglong2*)&s[1].key);
  if (FIRST) {
    p.f0 = __ldg(&s[0].arc);
    p.f1 = __ldg(&s[1].arc);
  }
}
template <bool FIRST>
__device__ __forceinline__ Arcs seg_find(const LayoutView& L, SegProbe<FIRST>& p, int4* first) {
  for (int64_t n = 0; n < L.buckets; ++n) {
    const bool h0 = p.e0.x == p.k, h1 = p.e1.x == p.k;
    if (h0 || h1) {
      const unsigned long long y = h0 ? p.e0.y & ~SPILLED : p.e1.y;
      const Arcs r{(int32_t)(uint32_t)y, (int32_t)(y >> 32)};
      if (r.len > 0 && !in_bounds(CHK_ARC, (long long)r.pos + r.len - 1, L.P)) return Arcs{0, 0};
      if (FIRST) *first = h0 ? p.f0 : p.f1;
      return r;
    }
    // (an empty first slot reads ~0, which is no spill)
    if (p.e0.x == ~0ull || !(p.e0.y & SPILLED)) break;
    p.b = p.b + 1 < (uint64_t)L.buckets ? p.b + 1 : 0;
    const SegSlot* s = L.seg_hash + 2 * p.b;
    p.e0 = __ldg((const ulonglong2*)&s[0].key);
    p.e1 = __ldg((const ulonglong2*)&s[1].key);
    if (FIRST) {
      p.f0 = __ldg(&s[0].arc);
      p.f1 = __ldg(&s[1].arc);
    }
  }
  return Arcs{0, 0};
}
__device__ __forceinline__ Arcs find_arcs(const LayoutView& L, int32_t a, int32_t q) {
  SegProbe<false> p;
  seg_load(L, a, q, p);
  return seg_find(L, p, nullptr);
}

// Chained launches of the per-position kernels (programmatic dependent
// launch).  A step kernel launched with programmatic stream serialization
// may be scheduled while the previous kernel of its stream still runs.  Its
// first instruction waits until that kernel has completed and its writes
// are visible (griddepcontrol.wait), so no access of the step precedes it;
// then it lets the next position's kernel be scheduled in turn.  What
// overlaps is the launch and block scheduling of position t+1 with the work
// of position t.  Launched without the attribute, both do nothing.
__device__ __forceinline__ void chain_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void add_count(const CountView& C, int32_t id, float g) {
  if (C.batched) {
    atomicAdd(C.cnt64 + id, fx_widen(g));
  } else {
    // compensated float32 summation (one string: one writer per arc and
    // step; read through L2, as a persistent pass meets the same arc at
    // later positions in other blocks)
    const float s0 = __ldcg(C.cnt + id), cmp = __ldcg(C.comp + id);
    const float y = __fsub_rn(g, cmp);
    const float s1 = __fadd_rn(s0, y);
    C.comp[id] = __fsub_rn(__fsub_rn(s1, s0), y);
    C.cnt[id] = s1;
  }
}

}  // namespace fstgpu
