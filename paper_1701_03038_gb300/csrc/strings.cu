// strings.cu -- a warp or block per string, over all of its positions.
//
// The strings of a batch are independent, and the frontier of most tokens is
// a handful of states (20M-arc workload: median 1 live state, 90% of the
// tokens at most 12).  The per-position launches of kernels.cu then pay a
// launch and a grid-wide chain of dependent accesses for a microsecond of
// work, at every position of every string.  Here a group of threads takes a
// string and runs its position loop: the accumulators of a position are a
// hash table in shared memory, positions are separated by the group's own
// barrier, and no launch or grid-wide step remains but one kernel a pass.
//
// The blocks of that kernel have two roles, and a string changes hands
// between them through two queues as its frontier grows and shrinks:
//   light -- every warp runs a string of its own while its positions have at
//            most 128 arcs out of live states.  In a run of positions with
//            one arc each (65% of them; nearly all of a long string's) it
//            only walks: a run of up to 32 leaves the values in the lanes
//            and is written at once, so a step is one table lookup;
//   heavy -- the block runs one string: in a larger table, or, past that,
//            over dense accumulators of all states in global memory (one
//            array per block, not per string), whose position is cut into
//            chunks that all heavy blocks share: the few positions that
//            reach most states carry most of the arcs (1% of the tokens,
//            90% of the arcs).
// What a position computes is what kernels.cu computes, operation by
// operation (exact maxima, 2^-40 fixed-point sums, float64 values shifted by
// the position's largest), so scores, paths and log Z are the same bits
// whichever kernels run.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "frontier.cuh"
#include "kernels.cuh"

namespace fstgpu {
namespace {

// Arcs per lane in flight: a light warp's (its table serves at most 128
// arcs) and a heavy block's.  More of them spill: with 4 a heavy block's
// backward pass over 4,096 strings of 5 to 200 symbols on 20M arcs takes 18%
// longer (2.7 ms with 2), and the forward passes (2.9 and 4.6 ms) are the same.
constexpr int VU0 = 1, VU1 = 2;

// Threads of a block (a light block runs NT1 / 32 strings), and the slots of
// a light warp's and a heavy block's table.  The kernels are compiled for
// three blocks an SM (80 registers a thread): with two (128) the same
// backward pass takes 40% longer, with four (64) the Viterbi pass 30%.
constexpr int NT1 = 256, WARPS = NT1 / 32;
constexpr int HS0 = 256, HS1 = 2 * STRING_TABLE_ARCS;
// the same of the backward pass, whose light warps hold at most LIGHT_CAP
// states
constexpr int BHS0 = 128, BHS1 = 1024, LIGHT_CAP = 96;
// a heavy block hands a string back at this many arcs and entries
constexpr int LIGHT_ARCS = 64;
// a light warp leaves a string with more start states to a heavy block, and a
// block shares more than SHARE_ARCS of them out uncounted, in chunks of START_CHUNK
constexpr int LIGHT_STARTS = HS0 / 2, START_CHUNK = NT1 * 2;
// a position is shared among the heavy blocks from SHARE_ARCS arcs on, in
// chunks of about CHUNK_ARCS; a block with a string of its own leaves it for
// jobs of BIG_CHUNKS chunks
constexpr int SHARE_ARCS = 4096, CHUNK_ARCS = 2048, BIG_CHUNKS = 24;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }
__device__ __forceinline__ uint32_t lanes_below() { return (1u << lane_id()) - 1u; }

__device__ __forceinline__ uint32_t slot_of(uint32_t key, uint32_t mask) {
  return ((key * 0x9E3779B1u) >> 15) & mask;
}

// Exclusive prefix of len over the warp, and its total.
__device__ __forceinline__ int32_t warp_excl(int32_t len, int32_t* total) {
  int32_t incl = len;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t o = __shfl_up_sync(FULL, incl, d);
    if (lane_id() >= d) incl += o;
  }
  *total = __shfl_sync(FULL, incl, 31);
  return incl - len;
}
// Lane owning flat arc a: the last lane whose first flat arc is <= a.
template <int N = 32>
__device__ __forceinline__ int owner_of(const int32_t* excl, int32_t a) {
  int o = 0;
#pragma unroll
  for (int step = N / 2; step >= 1; step >>= 1)
    if (excl[o + step] <= a) o += step;
  return o;
}

// The lane after s in the group `peers`, round and round.
__device__ __forceinline__ int next_peer(uint32_t peers, int s) {
  const uint32_t above = peers & ~((2u << s) - 1u);
  return __ffs(above ? above : peers) - 1;
}

// The entries a group of N lanes (a warp or a block) walks at a time, E a lane
// and in shared memory: the lanes take their arcs flat, whatever entry they
// belong to.  (A heavy block's warps with 32 entries each left most of them
// waiting for the one with the most arcs: out-degrees are heavy-tailed.  And
// most entries of a dense position have no arc: 256 of them at a time made
// rounds of 420 arcs on average, each with its own chain of latencies.)
template <class Real, int N, int E>
struct GroupStage {
  static constexpr int LANES = N, PER = E;
  Real r[N * E];        // the source's value,
  int32_t excl[N * E];  // first flat arc and
  int32_t e0[N * E];    // first arc record
  int32_t total[E][N / 32];  // arcs of each warp's entries
  // (a block:) states a warp staged and has not yet listed
  static constexpr int OUT = N == 32 ? 1 : 256;
  int32_t out[N / 32][OUT];
  static __device__ __forceinline__ int lane() { return N == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x; }
};

// A table of one position's accumulators (it fits when the position has at
// most HS / 2 arcs out of live states).
template <int HS, class Val>
struct Table {
  unsigned long long acc[HS];  // Viterbi key / forward maximum (order key)
  Val aux[HS];                 // forward: fixed-point sum; Viterbi: predecessor entry
  uint32_t key[HS];            // state + 1 (0 = empty)
  uint16_t list[HS / 2];       // slots in use
  int32_t staged;
};

// What a group (a light warp or a heavy block) keeps between positions: the
// rest of the pool chunk it holds, and the live entries and arcs of its
// string so far.
struct GroupState {
  int32_t pool_at, pool_left;
  unsigned long long live_e, live_a;
};

// What a heavy block shares: the chunk being worked on, its index (-1:
// none), the search for one, this block's number, and a position's range,
// arcs and largest value.
struct HeavyShared {
  StringJob job;
  unsigned long long tag;  // slot and phase number whose parameters job holds (~0: none)
  bool same, last, halt;   // of the last claim
  int32_t chunk, pick, at, self;
  int32_t base;
  uint32_t tot, mk;
};

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr uint64_t BEGIN_NS = 20000ull;

__device__ __forceinline__ uint32_t peek(const uint32_t* p) { return *(const volatile uint32_t*)p; }

// Whether a wait has run out: the run is over, and what others would have
// brought may not come any more.
__device__ __forceinline__ bool gave_up(const StringQueue& K) { return (peek(K.ctl + CTL_FLAGS + 1) & ERR_TIMEOUT) != 0u; }
// This wait has.  (The forward passes' final kernels read the flag; after a
// backward pass the counts' kernel reads `spoiled`.)
__device__ __forceinline__ void give_up(const StringQueue& K) {
  atomicOr(K.ctl + CTL_FLAGS + 1, ERR_TIMEOUT);
  if (K.spoiled) *(volatile double*)K.spoiled = __longlong_as_double(0x7fffffffffffffffll);
}

// The two string queues (QL light, QH heavy): rings whose slots hold string
// + 1 (0 = empty).  A worker that may wait takes a ticket, the number of an
// item that may still have to come, and polls that item's slot, which no
// other worker reads; one that may not wait takes an item only if there is
// one.  One thread of a group calls these; a push publishes what the group
// wrote before (the caller synchronises first).
enum : int { QL = 0, QH = 1 };
__device__ __forceinline__ uint32_t* queue_slot(const StringQueue& K, int q, uint32_t i) {
  return K.ring + (size_t)q * (K.ring_mask + 1u) + (i & K.ring_mask);
}
__device__ __forceinline__ void queue_push(const StringQueue& K, int q, int32_t b) {
  __threadfence();
  uint32_t* slot = queue_slot(K, q, atomicAdd(K.ctl + CTL_TAIL + q * CTL_LINE, 1u));
  // (a slot a whole ring back has its reader, who empties it)
  const uint64_t t0 = now_ns();
  while (atomicCAS(slot, 0u, (uint32_t)b + 1u) != 0u) {
    if (gave_up(K)) return;
    if (now_ns() - t0 > K.limit_ns) {
      give_up(K);
      return;
    }
  }
  atomicAdd(K.ctl + CTL_PROGRESS, 1u);
}
// The item of ticket i, -1 while there is none.
__device__ __forceinline__ int32_t queue_poll(const StringQueue& K, int q, uint32_t i) {
  uint32_t* slot = queue_slot(K, q, i);
  if (peek(slot) == 0u) return -1;
  const uint32_t v = atomicExch(slot, 0u);
  __threadfence();
  return (int32_t)v - 1;
}
__device__ __forceinline__ uint32_t queue_ticket(const StringQueue& K, int q) {
  return atomicAdd(K.ctl + CTL_HEAD + q * CTL_LINE, 1u);
}
// An item that is there already (-1: none, or others were faster).
__device__ __forceinline__ int32_t queue_pop(const StringQueue& K, int q) {
  for (int tries = 0; tries < 4; ++tries) {
    uint32_t* head = K.ctl + CTL_HEAD + q * CTL_LINE;
    const uint32_t h = peek(head);
    if ((int32_t)(peek(K.ctl + CTL_TAIL + q * CTL_LINE) - h) <= 0) return -1;
    if (atomicCAS(head, h, h + 1u) != h) continue;
    const uint64_t t0 = now_ns();
    for (;;) {  // (its writer has the number and is about to write)
      const int32_t b = queue_poll(K, q, h);
      if (b >= 0) return b;
      if (gave_up(K)) return -1;
      if (now_ns() - t0 > K.limit_ns) {
        give_up(K);
        return -1;
      }
    }
  }
  return -1;
}

// A worker's patience: true once nothing has moved for the limit.
struct Patience {
  uint64_t t0;
  uint32_t seen;
  __device__ __forceinline__ void start(const StringQueue& K) {
    t0 = now_ns();
    seen = peek(K.ctl + CTL_PROGRESS);
  }
  __device__ __forceinline__ bool over(const StringQueue& K) {
    const uint32_t p = peek(K.ctl + CTL_PROGRESS);
    if (p != seen) {
      seen = p;
      t0 = now_ns();
    }
    if (now_ns() - t0 <= K.limit_ns) return false;
    give_up(K);
    return true;
  }
};
__device__ __forceinline__ bool all_done(const StringQueue& K) {
  return peek(K.ctl + CTL_FINISHED) >= (uint32_t)K.strings || gave_up(K);
}
// A string went from position t0 to t1 (one thread): every 4,096 positions
// count as progress, whichever way they were done.  (A run of one-arc
// positions steps over most multiples of 4,096: without its report a string
// of 3.5 million of them ran into the limit of those who wait.)
__device__ __forceinline__ void report(const StringQueue& K, int32_t t0, int32_t t1) {
  if ((t0 ^ t1) >> 12) atomicAdd(K.ctl + CTL_PROGRESS, 1u);
}
// A string is done (one thread, after the group's barrier).
__device__ __forceinline__ void string_done(const StringQueue& K) {
  __threadfence();
  atomicAdd(K.ctl + CTL_FINISHED, 1u);
  atomicAdd(K.ctl + CTL_PROGRESS, 1u);
}

// Whether every block of the launch has begun.  Workers only wait for work
// from others once it is so: before, a block that would bring it may not be
// resident (another stream's kernel may hold its place), and a worker with
// nothing to do leaves (light) or takes what it finds (heavy).
__device__ __forceinline__ bool all_begun(const StringQueue& K) { return peek(K.ctl + CTL_BEGUN) >= gridDim.x; }
// A string that has not been started (-1: none).
__device__ __forceinline__ int32_t take_new(const StringQueue& K) {
  if (peek(K.ctl + CTL_TAKE) >= (uint32_t)K.strings) return -1;
  const uint32_t i = atomicAdd(K.ctl + CTL_TAKE, 1u);
  return i < (uint32_t)K.strings ? (int32_t)i : -1;
}

// The next string of a light warp: one that a heavy block handed back, else
// one not started yet, else wait for one; -1: the warp leaves.
__device__ __forceinline__ int32_t next_light(const StringQueue& K) {
  int32_t b = -1;
  if ((threadIdx.x & 31) == 0) {
    if ((b = queue_pop(K, QL)) < 0 && (b = take_new(K)) < 0 && !all_done(K) && all_begun(K)) {
      const uint32_t ticket = queue_ticket(K, QL);
      Patience w;
      w.start(K);
      for (uint32_t i = 1; (b = queue_poll(K, QL, ticket)) < 0; ++i) {
        if (i % K.polls == 0u && (all_done(K) || w.over(K))) break;
        __nanosleep(1000);
      }
    }
    if (b < 0) atomicSub(K.ctl + CTL_ALIVE, 1u);
  }
  return __shfl_sync(FULL, b, 0);
}

// ----------------------------------------------------------------------
// Shared positions.  A heavy block that meets a position too large for its
// table posts it as a job: a slot {parameters, word} with word = phase
// number, chunks and next chunk in one 64-bit value, so that the atomic add
// that claims a chunk also says of which phase it is.  Any heavy block
// claims chunks, between the positions of its own string or when it has
// none; the owner claims them too, then waits for the chunks that
// others hold.  A claimed chunk is being worked on by a running block, so
// the wait needs no co-residency; it is bounded all the same: past the
// limit the run reports FST_ERR_TIMEOUT, and the owner leaves the kernel.  It
// takes nothing more, because the others go on with the chunks of its slot,
// which a next position's staged states, counts and phases would meet; its
// accumulators are cleared when its block next starts.
// ----------------------------------------------------------------------
constexpr int JOB_BITS = 22;
constexpr unsigned long long JOB_MASK = (1ull << JOB_BITS) - 1ull;
__device__ __forceinline__ int32_t job_left(unsigned long long w) {
  return (int32_t)((w >> JOB_BITS) & JOB_MASK) - (int32_t)(w & JOB_MASK);
}
__device__ __forceinline__ bool job_open(unsigned long long w) { return (w & JOB_MASK) < ((w >> JOB_BITS) & JOB_MASK); }

// Claim a chunk of the job in slot g: its index and (unless they are there)
// the parameters into shared memory.  All threads call it, after the chunk
// claimed before, of slot fin (-1: none), which counts as done now that its
// writes are visible.  False: none left.  It costs one atomic's way to L2 and
// back: the block that holds a job's last chunk does not ask for another, and
// whether its ticket's string has come (*stop) is looked up meanwhile, for
// the next call (sh.halt).  (Done, asked and checked one by one a chunk of 17
// us carried 9 us of this.)
template <class Sh>
__device__ __forceinline__ bool job_claim(Sh& sh, const StringQueue& K, int32_t g, int32_t fin, const uint32_t* stop) {
  StringJob* J = K.jobs + g;
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t come = stop ? peek(stop) : 0u;
    if (fin >= 0) {
      __threadfence();
      atomicAdd(&K.jobs[fin].done, 1u);
    }
    int32_t c = -1;
    if (fin < 0 || !(sh.last || sh.halt)) {
      const unsigned long long w = atomicAdd(&J->word, 1ull);
      if (job_open(w)) {
        c = (int32_t)(w & JOB_MASK);
        sh.last = (w & JOB_MASK) + 1ull == ((w >> JOB_BITS) & JOB_MASK);
        const unsigned long long tag = ((unsigned long long)g << 32) | (w >> (2 * JOB_BITS));
        sh.same = sh.tag == tag;
        sh.tag = tag;
        __threadfence();
      }
    }
    sh.halt = come != 0u;
    sh.chunk = c;
  }
  __syncthreads();
  if (sh.chunk < 0) return false;
  if (sh.same) return true;
  constexpr int W = (int)(sizeof(StringJob) / 4);
  static_assert(sizeof(StringJob) % 4 == 0 && W <= 32, "one word a lane");
  if (threadIdx.x < W) ((uint32_t*)&sh.job)[threadIdx.x] = __ldcg((const uint32_t*)J + threadIdx.x);
  __syncthreads();
  return true;
}
// A slot with at least `least` chunks left, this block's neighbours first
// (-1: none).
template <class Sh>
__device__ __forceinline__ int32_t job_find(Sh& sh, const StringQueue& K, int32_t least) {
  __syncthreads();
  if (threadIdx.x == 0) sh.pick = INT32_MAX;
  __syncthreads();
  for (int32_t i = threadIdx.x; i < K.owners; i += blockDim.x) {
    const int32_t g = (int32_t)((sh.self + i) % (unsigned)K.owners);
    if (job_left(*(volatile unsigned long long*)&K.jobs[g].word) >= least) atomicMin(&sh.pick, i);
  }
  __syncthreads();
  const int32_t i = sh.pick;
  return i == INT32_MAX ? -1 : (int32_t)((sh.self + i) % (unsigned)K.owners);
}
// Post sh.job (filled by thread 0) as the block's next phase of n chunks.
template <class Sh>
__device__ __forceinline__ void job_post(Sh& sh, const StringQueue& K, int32_t n) {
  __syncthreads();
  if (threadIdx.x == 0) {
    StringJob* J = K.jobs + sh.self;
    const unsigned long long w = *(volatile unsigned long long*)&J->word;
    sh.job.done = 0u;
    sh.tag = ~0ull;
    constexpr int W = (int)(sizeof(StringJob) / 4);
    for (int i = 2; i < W; ++i) *((volatile uint32_t*)J + i) = ((const uint32_t*)&sh.job)[i];
    __threadfence();
    atomicExch(&J->word, (((w >> (2 * JOB_BITS)) + 1ull) << (2 * JOB_BITS)) | ((unsigned long long)n << JOB_BITS));
    atomicAdd(K.ctl + CTL_OPEN, 1u);
    if (n >= BIG_CHUNKS) atomicAdd(K.ctl + CTL_BIG, 1u);
  }
  __syncthreads();
}
// Wait for every chunk of the block's own job; false: given up.
template <class Sh>
__device__ __forceinline__ bool job_wait(Sh& sh, const StringQueue& K, int32_t n) {
  __syncthreads();
  if (threadIdx.x == 0) {
    StringJob* J = K.jobs + sh.self;
    const uint64_t t0 = now_ns();
    int32_t ok = 1;
    while (*(volatile uint32_t*)&J->done != (uint32_t)n) {
      if (now_ns() - t0 > K.limit_ns) {
        give_up(K);
        *(volatile uint32_t*)(K.dirty + sh.self) = 1u;
        ok = 0;
        break;
      }
      __nanosleep(100);
    }
    __threadfence();
    atomicSub(K.ctl + CTL_OPEN, 1u);
    if (n >= BIG_CHUNKS) atomicSub(K.ctl + CTL_BIG, 1u);
    atomicAdd(K.ctl + CTL_PROGRESS, 1u);
    sh.pick = ok;
    sh.job.staged = __ldcg(&J->staged);
    sh.job.tot = __ldcg(&J->tot);
    sh.job.mk = __ldcg(&J->mk);
  }
  __syncthreads();
  return sh.pick != 0;
}

// Whether there are jobs that a block with a string of its own leaves it for:
// large ones, while few of the blocks that would do them have no string.
// (With half of the blocks idle a string lost 136 us at one position to them.)
__device__ __forceinline__ bool big_jobs(const StringQueue& K) {
  const uint4 w = __ldcv((const uint4*)(K.ctl + CTL_OPEN));
  return w.y != 0u && w.z * 8u < (uint32_t)K.owners;
}

// What a heavy block does next: a string from the heavy queue (blocks that
// own dense storage), a job of another block, and, while there are no light
// warps, the light ones' strings too; it leaves once every string is done.
// At the start it gives the light blocks, which begin after it, BEGIN_NS: a
// string of 1,000 one-arc positions that a heavy block takes instead, and
// keeps, costs 4 ms against 1.0 ms.
enum : int32_t { PICK_LEAVE = -1, PICK_NONE = -2, PICK_HELP = -3 };
struct HeavyPick {
  Patience wait;
  uint32_t ticket = 0u, polls = 0u;
  bool waiting = false, holds = false, idle = false;
  uint64_t first = 0u;
  // All threads call it; *light: the light warps take light strings.
  __device__ __forceinline__ int32_t next(HeavyShared& hv, const StringQueue& K, bool* light) {
    __syncthreads();  // (every thread has read hv.pick of a search that found no job)
    if (threadIdx.x == 0) {
      int32_t b = PICK_NONE;
      const bool begun = holds || all_begun(K);
      if (first == 0u) first = now_ns();
      const bool lights = peek(K.ctl + CTL_ALIVE) != 0u || (!begun && now_ns() - first < BEGIN_NS);
      if (hv.self < K.owners) {
        if (begun && !holds) {
          ticket = queue_ticket(K, QH);
          holds = true;
          atomicAdd(K.ctl + CTL_IDLE, 1u);
        }
        b = holds ? queue_poll(K, QH, ticket) : queue_pop(K, QH);
        if (b >= 0 && holds) {
          holds = false;
          atomicSub(K.ctl + CTL_IDLE, 1u);
        }
        if (b < 0 && !lights && (b = queue_pop(K, QL)) < 0) b = take_new(K);
        if (b < 0) b = PICK_NONE;
      }
      // else a job to help with, unless there was none to be had the last time
      if (b == PICK_NONE && !idle && peek(K.ctl + CTL_OPEN) != 0u) b = PICK_HELP;
      idle = b == PICK_HELP;
      if (b == PICK_NONE && (!waiting || ++polls % K.polls == 0u)) {
        if (all_done(K)) {
          b = PICK_LEAVE;
        } else if (!waiting) {
          wait.start(K);
          waiting = true;
        } else if (wait.over(K)) {
          b = PICK_LEAVE;
        }
      }
      if (b >= 0) waiting = false;
      hv.pick = b;
      hv.at = lights;
    }
    __syncthreads();
    const int32_t b = hv.pick;
    *light = hv.at != 0;
    __syncthreads();
    return b;
  }
  // Where the string of this block's ticket will appear (null: it has none):
  // its helping stops for it.
  __device__ __forceinline__ const uint32_t* stop(const StringQueue& K) const {
    return holds ? queue_slot(K, QH, ticket) : nullptr;
  }
  // There was a chunk to help with.
  __device__ __forceinline__ void helped() { idle = waiting = false; }
};

// ======================================================================
// Forward recursions (Alg. 1 and Alg. 2 forward loop).
// ======================================================================
template <bool VIT>
struct Forward {
  typedef typename std::conditional<VIT, int32_t, unsigned long long>::type Val;
  typedef typename std::conditional<VIT, float, double>::type Real;
  typedef GroupStage<Real, 32, 1> Stage;
  typedef GroupStage<Real, NT1, 2> BlockStage;
  typedef Table<HS0, Val> LightTable;
  typedef Table<HS1, Val> HeavyTable;
  struct LightShared {
    Stage st;
    LightTable tab;
    GroupState gs;
  };
  struct BlockShared {
    HeavyTable tab;
    BlockStage st;
    HeavyShared hv;
    GroupState gs;
  };

  const LayoutView& L;
  const int32_t* sym;
  const FrontierState& S;
  const StringQueue& K;

  // Dense storage of heavy block g: [Q] keys (Viterbi) or [Q] {sum, maximum}
  // pairs, the staged states, and (Viterbi) the arcs of the entries of the
  // last position; light warp g's share of the last follows the blocks'.
  __device__ __forceinline__ unsigned long long* dacc(int32_t g) const { return K.dense + (int64_t)g * S.Q * (VIT ? 1 : 2); }
  __device__ __forceinline__ int32_t* dstage(int32_t g) const { return K.dstage + (int64_t)g * S.Q; }
  __device__ __forceinline__ int2* fe_heavy(int32_t g) const { return K.fe + (int64_t)g * S.Q; }
  __device__ __forceinline__ int2* fe_light(int32_t g) const { return K.fe + K.fe_light + (int64_t)g * (HS0 / 2); }

  // The arcs of entry i (cap: the entries that fe holds).
  __device__ __forceinline__ void put_arcs(int2* fe, int32_t cap, int32_t i, const Arcs& x) const {
    if (in_bounds(CHK_STAGE, i, cap)) fe[i] = make_int2(x.pos, x.len);
  }

  struct Entry {
    int32_t e0, len, jp;
    Real r;
  };
  static __device__ __forceinline__ Real real(float x) {
    if constexpr (VIT) return x;
    else return fx_widen(x);
  }
  static __device__ __forceinline__ Real none() { return (Real)0; }
  // Entry i of position t-1 (the start states at t = 1).  Read through L2:
  // another SM may have written it.
  __device__ __forceinline__ Entry entry(const int2* fe, int32_t t, int32_t base, int32_t i, int32_t a) const {
    Entry x;
    if (t == 1) {
      const int32_t q = __ldg(S.start_q + i);
      const Arcs s = find_arcs(L, a, q);
      x = Entry{s.pos, s.len, -1, real(__ldg(S.theta_s + q))};
    } else {
      x.jp = base + i;
      if (!in_bounds(CHK_POOL_READ, x.jp, S.pool_cap)) return Entry{0, 0, -1, none()};
      if constexpr (VIT) {
        const int2 s = __ldcg(fe + i);
        x.e0 = s.x;
        x.len = s.y;
        x.r = __ldcg(S.pool_v + x.jp);
      } else {
        x.e0 = __ldcg(S.pool_x + x.jp);
        x.len = __ldcg(S.pool_n + x.jp);
        x.r = __ldcg(S.pool_d + x.jp);
      }
    }
    return x;
  }

  // The value of an arc out of a source of value r (forward, *v) and its
  // key (0: none).
  __device__ __forceinline__ unsigned long long candidate(Real r, const int4& arc, double* v) const {
    if constexpr (VIT) {
      // one rounded float32 addition per candidate
      const float x = __fadd_rn(r, __int_as_float(arc.y));
      return x != neg_inf() ? ((unsigned long long)fkey(x) << 32) | (unsigned long long)(~(uint32_t)arc.z) : 0ull;
    } else {
      // the exact float64 maximum (its term in the sum is then exactly 1)
      if (dead32(__int_as_float(arc.y))) return 0ull;
      *v = r + fx_widen(__int_as_float(arc.y));
      return dkey(*v);
    }
  }

  // The group's next entries staged for load_arcs: those from i0 on, below n,
  // of the position before (fe, t, base, a as for entry).  Returns their
  // arcs.  (A block's walk of the ones before may still be going on: it is
  // waited for.)
  template <class St>
  __device__ __forceinline__ int32_t stage(St& st, const int2* fe, int32_t t, int32_t base, int32_t a, int32_t i0,
                                           int32_t n) const {
    constexpr int N = St::LANES, E = St::PER;
    constexpr bool BLOCK = N > 32;
    Entry x[E];
    int32_t ex[E], total = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int32_t i = i0 + e * N + St::lane();
      x[e] = Entry{0, 0, -1, none()};
      if (i < n) x[e] = entry(fe, t, base, i, a);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      ex[e] = warp_excl(x[e].len, &total);
      if (BLOCK && lane_id() == 0) st.total[e][warp_id()] = total;
    }
    if constexpr (BLOCK) {
      __syncthreads();
      total = 0;
#pragma unroll
      for (int e = 0; e < E; ++e)
#pragma unroll
        for (int w = 0; w < N / 32; ++w) {
          if (w == warp_id()) ex[e] += total;
          total += st.total[e][w];
        }
    } else {
      __syncwarp();
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int k = e * N + St::lane();
      st.excl[k] = ex[e];
      st.e0[k] = x[e].e0;
      st.r[k] = x[e].r;
    }
    if (BLOCK) __syncthreads();
    else __syncwarp();
    return total;
  }
  // This lane's VU flat arcs from a0 on: their owners (-1: none) and records.
  template <int VU, class St>
  __device__ __forceinline__ void load_arcs(const St& st, int32_t a0, int32_t total, int (&oo)[VU], int4 (&arc)[VU]) const {
#pragma unroll
    for (int u = 0; u < VU; ++u) {
      const int32_t a = a0 + u * St::LANES + St::lane();
      oo[u] = a < total ? owner_of<St::LANES * St::PER>(st.excl, a) : -1;
      arc[u] = make_int4(0, 0, 0, 0);
      if (oo[u] >= 0) {
        const int32_t i = st.e0[oo[u]] + (a - st.excl[oo[u]]);
        if (in_bounds(CHK_ARC, i, L.P)) arc[u] = __ldg(L.arcs + i);
        else oo[u] = -1;
      }
    }
  }

  // A list slot for every lane with want set: one atomic on the counter.
  __device__ __forceinline__ int32_t append(int32_t* n, bool want) const {
    const uint32_t w = __ballot_sync(FULL, want);
    if (!w) return 0;
    int32_t at = 0;
    if (lane_id() == __ffs(w) - 1) at = atomicAdd(n, __popc(w));
    return __shfl_sync(FULL, at, __ffs(w) - 1) + __popc(w & lanes_below());
  }

  // The staged chunk's arcs into a table.  PHASE 0: the atomic max of each
  // destination, whose first arc stages it; PHASE 1 (forward), once every
  // maximum is final: the fixed-point terms.  j0: the pool entry of the first
  // staged one (-1: start states).
  template <int PHASE, int HS, class St>
  __device__ __forceinline__ void walk_table(Table<HS, Val>& tab, const St& st, int32_t total, int32_t j0) const {
    constexpr int VU = HS == HS0 ? VU0 : VU1;
    for (int32_t a0 = 0; a0 < total; a0 += St::LANES * VU) {
      int oo[VU];
      int4 arc[VU];
      load_arcs(st, a0, total, oo, arc);
#pragma unroll
      for (int u = 0; u < VU; ++u) {
        if (u > 0 && a0 + u * St::LANES >= total) break;  // (the same in the group)
        double v = 0.0;
        const unsigned long long c = oo[u] >= 0 ? candidate(st.r[oo[u]], arc[u], &v) : 0ull;
        bool fresh = false;
        uint32_t h = 0u;
        if (c != 0ull) {
          const uint32_t k = (uint32_t)arc[u].x + 1u;
          h = slot_of(k, HS - 1);
          // at most HS / 2 keys: an empty slot ends every probe sequence
          for (int n = 0; n < HS; ++n) {
            const uint32_t old = PHASE == 0 ? atomicCAS(tab.key + h, 0u, k) : tab.key[h];
            if (old == k || old == 0u) {
              fresh = PHASE == 0 && old == 0u;
              break;
            }
            h = (h + 1) & (HS - 1);
          }
        }
        if constexpr (PHASE == 0) {
          if (c != 0ull) {
            atomicMax(tab.acc + h, c);
            if constexpr (VIT)
              if (fresh) tab.aux[h] = j0 < 0 ? -1 : j0 + oo[u];
          }
          const int32_t at = append(&tab.staged, fresh);
          if (fresh) tab.list[at] = (uint16_t)h;
        } else if (c != 0ull) {
          atomicAdd(tab.aux + h, fix_exp64(v, dkey_inv(tab.acc[h])));
        }
      }
    }
  }

  // The states the warp staged, to the list: one atomic for up to 256 of them.
  __device__ __forceinline__ void list_staged(int32_t g, int32_t* staged, const BlockStage& st, int32_t& pend) const {
    __syncwarp();
    int32_t at = 0;
    if (lane_id() == 0 && pend) at = atomicAdd(staged, pend);
    at = __shfl_sync(FULL, at, 0);
    for (int32_t i = lane_id(); i < pend; i += 32)
      if (in_bounds(CHK_STAGE, at + i, S.Q)) dstage(g)[at + i] = st.out[warp_id()][i];
    __syncwarp();
    pend = 0;
  }
  // The same into heavy block g's dense accumulators; `staged` counts the
  // staged states (shared memory, or the job's word).
  template <int PHASE>
  __device__ __forceinline__ void walk_dense(int32_t g, int32_t* staged, BlockStage& st, int32_t total, int32_t& pend) const {
    constexpr int VU = VU1;
    unsigned long long* acc = dacc(g);
    int oo[VU];
    int4 arc[VU];
    load_arcs(st, 0, total, oo, arc);
    for (int32_t a0 = 0; a0 < total; a0 += NT1 * VU) {
      double v[VU];
      unsigned long long c[VU];
      int32_t q[VU];
#pragma unroll
      for (int u = 0; u < VU; ++u) {
        v[u] = 0.0;
        q[u] = arc[u].x;
        c[u] = oo[u] >= 0 && in_bounds(CHK_ACC, q[u], S.Q) ? candidate(st.r[oo[u]], arc[u], &v[u]) : 0ull;
      }
      // (the next arcs' records are on their way while these ones' atomics are)
      load_arcs(st, a0 + NT1 * VU, total, oo, arc);
      if constexpr (PHASE == 0) {
        unsigned long long old[VU];
#pragma unroll
        for (int u = 0; u < VU; ++u)
          old[u] = c[u] ? atomicMax(VIT ? acc + q[u] : acc + 2 * (int64_t)q[u] + 1, c[u]) : 1ull;
        // the lanes that met a destination first stage it, with their warp
#pragma unroll
        for (int u = 0; u < VU; ++u) {
          const uint32_t w = __ballot_sync(FULL, old[u] == 0ull);
          if (old[u] == 0ull) st.out[warp_id()][pend + __popc(w & lanes_below())] = q[u];
          pend += __popc(w);
        }
        if (pend > BlockStage::OUT - 32 * VU) list_staged(g, staged, st, pend);
      } else {
        unsigned long long mx[VU];
#pragma unroll
        for (int u = 0; u < VU; ++u) mx[u] = c[u] ? __ldcg(acc + 2 * (int64_t)q[u] + 1) : 0ull;
#pragma unroll
        for (int u = 0; u < VU; ++u)
          if (mx[u]) atomicAdd(acc + 2 * (int64_t)q[u], fix_exp64(v[u], dkey_inv(mx[u])));
      }
    }
  }

  // The pool's next nb entries for a group (its first thread's job; -1: the
  // pool is full).  Short ranges come out of a chunk that the group reserved
  // (at most a quarter of it is left behind), longer ones one by one.
  __device__ __forceinline__ int32_t reserve(GroupState& gs, int32_t nb) const {
    if (nb <= gs.pool_left) {
      const int32_t at = gs.pool_at;
      gs.pool_at = at + nb;
      gs.pool_left -= nb;
      return at;
    }
    const bool small = nb * 4 <= K.chunk;
    const int32_t ask = small ? K.chunk : nb;
    const long long at = (long long)atomicAdd((unsigned long long*)S.pool_top, (unsigned long long)ask);
    if (at + nb > S.pool_cap) {
      atomicOr(S.flags + 1, ERR_POOL);
      return -1;
    }
    if (small) {
      gs.pool_at = (int32_t)at + nb;
      gs.pool_left = (int32_t)min((long long)ask, (long long)S.pool_cap - at) - nb;
    }
    return (int32_t)at;  // (pool entries are numbered in 31 bits)
  }
  __device__ __forceinline__ int32_t warp_reserve(GroupState& gs, int32_t nb) const {
    const int32_t at = lane_id() == 0 ? reserve(gs, nb) : 0;
    return __shfl_sync(FULL, at, 0);
  }

  // State d of value r into the pool at entry j, with its best arc and
  // predecessor (Viterbi) or its arcs on the next symbol (forward).
  __device__ __forceinline__ void put(int32_t j, int32_t d, Real r, int32_t x, int32_t n) const {
    if (!in_bounds(CHK_POOL_WRITE, j, S.pool_cap)) return;
    S.pool_q[j] = d;
    S.pool_x[j] = x;
    S.pool_n[j] = n;
    if constexpr (VIT) S.pool_v[j] = r;
    else S.pool_d[j] = r;
  }

  // Entries [i0, i0 + 32) of a table become pool entries base + i; their
  // slots are emptied.  Returns this lane's entry (len 0 past the end).
  template <int HS>
  __device__ __forceinline__ Entry read_table(Table<HS, Val>& tab, int32_t i0, int32_t nb, int32_t base, float shift,
                                              bool single, int32_t an, int2* fe, int4* first) const {
    const int32_t i = i0 + lane_id();
    Entry x{0, 0, -1, none()};
    if (i >= nb) return x;
    const int32_t h = tab.list[i];
    const int32_t d = (int32_t)tab.key[h] - 1;
    SegProbe<HS == HS0> p;
    if (an >= 0) seg_load(L, an, d, p);
    const unsigned long long acc = tab.acc[h];
    const Val aux = tab.aux[h];
    tab.acc[h] = 0ull;
    tab.key[h] = 0u;
    if (!VIT) tab.aux[h] = 0;
    if constexpr (VIT) x.r = fkey_inv((uint32_t)(acc >> 32));
    else x.r = fix_log_sum64(dkey_inv(acc) - fx_widen(shift), single ? 1099511627776ull : (unsigned long long)aux);  // 2^40
    const Arcs nxt = an >= 0 ? seg_find(L, p, first) : Arcs{0, 0};
    x.e0 = nxt.pos;
    x.len = nxt.len;
    x.jp = base + i;
    if (VIT) {
      put(base + i, d, x.r, (int32_t)(~(uint32_t)acc), single ? (int32_t)aux : -2);
      put_arcs(fe, HS == HS0 ? HS0 / 2 : S.Q, i, nxt);
    } else {
      put(base + i, d, x.r, nxt.pos, nxt.len);
    }
    return x;
  }
  template <int HS>
  __device__ __forceinline__ void empty_table(Table<HS, Val>& tab, int32_t i0, int32_t nb) const {
    const int32_t i = i0 + lane_id();
    if (i >= nb) return;
    const int32_t h = tab.list[i];
    tab.acc[h] = 0ull;
    if (!VIT) tab.aux[h] = 0;
    tab.key[h] = 0u;
  }

  // The same of the states that heavy block g's dense position staged (two a
  // lane in flight): returns their arcs and the largest value's order key.
  __device__ __forceinline__ void read_dense(int32_t g, int32_t i0, int32_t nb, int32_t base, float shift, bool single,
                                             int32_t an, int32_t* tot, uint32_t* mk) const {
    constexpr int RU = 2;
    unsigned long long* acc = dacc(g);
    int32_t d[RU];
    ulonglong2 x[RU];  // {sum, key or maximum}
    SegProbe<false> p[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      const int32_t i = i0 + u * 32 + lane_id();
      d[u] = i < nb ? __ldcg(dstage(g) + i) : -1;
    }
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      x[u] = make_ulonglong2(0ull, 0ull);
      if (d[u] < 0) continue;
      if (!in_bounds(CHK_ACC, d[u], S.Q)) d[u] = -1;
      if (d[u] < 0) continue;
      if (VIT) x[u].y = __ldcg(acc + d[u]);
      else x[u] = __ldcg((const ulonglong2*)acc + d[u]);
      if (an >= 0) seg_load(L, an, d[u], p[u]);
    }
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      if (d[u] < 0) continue;
      const int32_t i = i0 + u * 32 + lane_id();
      const Arcs nxt = an >= 0 ? seg_find(L, p[u], nullptr) : Arcs{0, 0};
      if constexpr (VIT) {
        acc[d[u]] = 0ull;
        put(base + i, d[u], fkey_inv((uint32_t)(x[u].y >> 32)), (int32_t)(~(uint32_t)x[u].y), -2);
        put_arcs(fe_heavy(g), S.Q, i, nxt);
      } else {
        ((ulonglong2*)acc)[d[u]] = make_ulonglong2(0ull, 0ull);
        const double r = fix_log_sum64(dkey_inv(x[u].y) - fx_widen(shift), single ? 1099511627776ull : x[u].x);
        put(base + i, d[u], r, nxt.pos, nxt.len);
        const uint32_t k = fkey64(r);
        *mk = k > *mk ? k : *mk;
      }
      *tot += nxt.len;
    }
  }

  // Where a string stands before position t: its entries of t-1.
  struct Place {
    int32_t n, t, cnt, tot, off, base;
    float shift;  // m_{t-1}, the largest value of position t-1
  };
  __device__ __forceinline__ Place resume(int32_t b) const {
    Place P;
    P.n = __ldg(S.bw_n + b);
    P.off = (int32_t)__ldg(S.bw_off + b);
    P.t = max(1, __ldcg(&K.park[b].t));
    P.cnt = P.n > 0 ? S.nstart : 0;
    P.base = 0;
    P.shift = 0.f;
    if (P.t > 1) {
      P.base = (int32_t)__ldcg(S.pool_base + P.off + P.t - 2);
      P.cnt = __ldcg(S.pool_cnt + P.off + P.t - 2);
      if (!VIT) P.shift = decode_max(__ldcg(S.mkey + P.off + P.t - 2));
    }
    P.tot = 0;
    return P;
  }
  // The arcs of entry i that a string goes on with: the Viterbi entries'
  // are looked up again.
  __device__ __forceinline__ int32_t resume_entry(const Place& P, int2* fe, int32_t cap, int32_t i, int32_t a) const {
    if (VIT && P.t > 1) {
      const Arcs x = find_arcs(L, a, __ldcg(S.pool_q + P.base + i));
      put_arcs(fe, cap, i, x);
      return x.len;
    }
    return entry(fe, P.t, P.base, i, a).len;
  }
  __device__ __forceinline__ void position_done(const Place& P, int32_t p, uint32_t mk) const {
    S.pool_base[p] = P.cnt ? P.base : 0;
    S.pool_cnt[p] = P.cnt;
    if (!VIT) {
      S.mkey[p] = P.cnt ? mk : 0u;
      S.ekey[p] = (uint32_t)P.tot;  // the arcs out of the position, for the backward pass
    }
  }
  // The group leaves the string: at its end or for queue `hand`.
  __device__ __forceinline__ void leave(const Place& P, GroupState& gs, int32_t b, int32_t hand) const {
    if (gs.live_e) atomicAdd((unsigned long long*)(K.ctl + CTL_LIVE), gs.live_e);
    if (gs.live_a) atomicAdd((unsigned long long*)(K.ctl + CTL_LIVE) + 1, gs.live_a);
    gs.live_e = gs.live_a = 0ull;
    if (hand >= 0) {
      K.park[b].t = P.t;
      queue_push(K, hand, b);
    } else {
      string_done(K);
    }
  }
  // No live state from position t on.
  __device__ __forceinline__ void dead_from(const Place& P, int32_t first, int32_t step) const {
    for (int32_t u = P.t + first; u <= P.n; u += step) {
      S.pool_base[P.off + u - 1] = 0;
      S.pool_cnt[P.off + u - 1] = 0;
      if (!VIT) S.mkey[P.off + u - 1] = 0u;
    }
  }

  // Up to 32 positions, from P.t on, that each have one arc: a chain of
  // lookups with nothing to group, the same in every lane.  Step k leaves its
  // entry with lane k, and the entries are written together (their stores,
  // one by one, took longer than the lookup).  Bound by the lookup's DRAM
  // latency: 64 strings of 1,000 symbols on 100M arcs take 0.57 us a position
  // (decoded, scored and counted: 6.9 ms before, 2.9 now).  Afterwards P stands at the
  // last of them, x and first hold its entry.  False: the arc at P.t is dead,
  // nothing was done.
  __device__ __forceinline__ bool chain(Place& P, GroupState& gs, int2* fe, int32_t an, Entry& x, int4& first) const {
    const int lane = lane_id();
    const int src = __ffs(__ballot_sync(FULL, x.len > 0)) - 1;
    Real r = __shfl_sync(FULL, x.r, src);
    const int32_t jp = __shfl_sync(FULL, x.jp, src);
    int4 arc;
    arc.x = __shfl_sync(FULL, first.x, src);
    arc.y = __shfl_sync(FULL, first.y, src);
    arc.z = __shfl_sync(FULL, first.z, src);
    const int32_t p = P.off + P.t - 1;
    // the symbols after each step (after the first: an)
    const int32_t next = P.t + lane < P.n ? __ldg(sym + p + 1 + lane) : -1;
    int32_t my_q = 0, my_x = 0, my_n = 0;
    Real my_r = none();
    float shift = P.shift;
    int4 f = make_int4(0, 0, 0, 0);
    Arcs nxt{0, 0};
    int32_t k = 0;
    while (k < 32) {
      double v = 0.0;
      const unsigned long long c = candidate(r, arc, &v);
      if (c == 0ull) break;
      if (k > 0) an = __shfl_sync(FULL, next, k);
      SegProbe<true> pr;
      if (an >= 0) seg_load(L, an, arc.x, pr);
      if constexpr (VIT) {
        r = fkey_inv((uint32_t)(c >> 32));
      } else {
        r = v - fx_widen(shift);
        shift = fx_narrow(r);  // the largest value: this one
      }
      if (lane == k) {
        my_q = arc.x;
        my_x = arc.z;
        my_r = r;
      }
      nxt = an >= 0 ? seg_find(L, pr, &f) : Arcs{0, 0};
      if (lane == k) {
        my_n = nxt.len;
        if (!VIT) my_x = nxt.pos;
      }
      ++k;
      if (nxt.len != 1) break;
      arc = f;
    }
    if (k == 0) return false;
    const int32_t base = warp_reserve(gs, k);
    const bool full = base < 0;
    if (lane < k) {
      if (!full) put(base + lane, my_q, my_r, my_x, VIT ? (lane == 0 ? jp : base + lane - 1) : my_n);
      S.pool_base[p + lane] = full ? 0 : base + lane;
      S.pool_cnt[p + lane] = full ? 0 : 1;
      if constexpr (!VIT) {
        S.mkey[p + lane] = full ? 0u : fkey64(my_r);
        S.ekey[p + lane] = (uint32_t)my_n;
      }
    }
    P.t += k - 1;
    P.cnt = full ? 0 : 1;
    P.tot = full ? 0 : nxt.len;
    P.base = base + k - 1;
    P.shift = shift;
    if (lane == 0) {
      report(K, P.t - k, P.t);
      if (!full) {
        gs.live_e += (unsigned long long)k;
        gs.live_a += (unsigned long long)(k - 1 + nxt.len);
      }
    }
    if (VIT && lane == 0) fe[0] = make_int2(nxt.pos, nxt.len);
    x = Entry{nxt.pos, lane == 0 ? P.tot : 0, P.base, r};
    first = make_int4(f.x, f.y, f.z, 1);
    return true;
  }

  // ---- a light warp's string --------------------------------------------
  // While a position has at most 32 entries and 32 arcs the frontier lives
  // in registers: a lane per entry, a lane per arc, destinations grouped by
  // a warp match, and the next lookups in flight while the values are formed.
  // The frontiers beyond, up to HS0 / 2 arcs, go through the warp's table.
  __device__ __forceinline__ void light_string(LightTable& tab, Stage& st, GroupState& gs, int32_t g, int32_t b) const {
    const int lane = lane_id();
    Place P = resume(b);
    int2* fe = fe_light(g);
    uint32_t mk = 0u;
    int32_t a = P.n > 0 ? __ldg(sym + P.off + P.t - 1) : 0;
    if (P.t == 1 && P.cnt > LIGHT_STARTS) {
      P.tot = HS0;  // (more than it takes)
    } else {
      for (int32_t i = lane; i < P.cnt; i += 32) P.tot += resume_entry(P, fe, HS0 / 2, i, a);
      P.tot = (int32_t)__reduce_add_sync(FULL, (unsigned)P.tot);
    }
    __syncwarp();
    // this lane's entry (len 0: none), with its first arc when first.w is set
    Entry x{0, 0, -1, none()};
    int4 first = make_int4(0, 0, 0, 0);
    bool have = false;  // the entries are in registers
    int32_t hand = -1;
    for (; P.t <= P.n; ++P.t) {
      const int32_t p = P.off + P.t - 1;
      if (P.cnt == 0 || P.tot == 0) break;
      if (P.tot > HS0 / 2) {
        hand = QH;
        break;
      }
      const int32_t an = P.t < P.n ? __ldg(sym + p + 1) : -1;
      int32_t nb, nbase;
      if (have && P.cnt <= 32 && P.tot == 1 && chain(P, gs, fe, an, x, first)) {
        a = P.t < P.n ? __ldg(sym + P.off + P.t) : -1;
        if (P.cnt == 0) {
          ++P.t;
          break;
        }
        continue;
      } else if (P.cnt <= 32 && P.tot <= 32) {
        if (!have) {
          x = Entry{0, 0, -1, none()};
          if (lane < P.cnt) x = entry(fe, P.t, P.base, lane, a);
          first.w = 0;
        }
        // a lane per arc: its own entry's, or (some entry has several) the
        // flat arc of its number
        Real r = x.r;
        int32_t jp = x.jp, e = x.e0;
        int4 arc = first;
        bool on = x.len > 0;
        if (__any_sync(FULL, x.len > 1)) {
          int32_t total;
          const int32_t ex = warp_excl(x.len, &total);
          int o = 0;
#pragma unroll
          for (int step = 16; step >= 1; step >>= 1) {
            const int32_t v = __shfl_sync(FULL, ex, (o + step) & 31);
            if (v <= lane) o += step;
          }
          on = lane < total;
          r = __shfl_sync(FULL, x.r, o);
          jp = __shfl_sync(FULL, x.jp, o);
          const int32_t k = lane - __shfl_sync(FULL, ex, o);
          e = __shfl_sync(FULL, x.e0, o) + k;
          arc.x = __shfl_sync(FULL, first.x, o);
          arc.y = __shfl_sync(FULL, first.y, o);
          arc.z = __shfl_sync(FULL, first.z, o);
          arc.w = __shfl_sync(FULL, first.w, o);
          if (k != 0) arc.w = 0;
        }
        if (on && !arc.w) {
          if (in_bounds(CHK_ARC, e, L.P)) arc = __ldg(L.arcs + e);
          else on = false;
        }
        double v = 0.0;
        const unsigned long long c = on ? candidate(r, arc, &v) : 0ull;
        on = c != 0ull;
        SegProbe<true> pr;
        if (on && an >= 0) seg_load(L, an, arc.x, pr);
        // the lanes with the same destination
        const uint32_t lanes = __ballot_sync(FULL, on);
        uint32_t peers = 1u << lane;
        int most = 1;
        if (__popc(lanes) > 1) {
          const uint32_t same = __match_any_sync(FULL, on ? arc.x : -1);
          if (on) peers = same;
          most = (int)__reduce_max_sync(FULL, (unsigned)__popc(peers));
        }
        unsigned long long best = c, sum = 1099511627776ull;  // 2^40: one arc alone
        bool lead = on;
        if (most > 1) {
          // the largest of the group, round its lanes
          int s = lane;
          for (int i = 1; i < most; ++i) {
            s = next_peer(peers, s);
            const unsigned long long w = __shfl_sync(FULL, c, s);
            best = w > best ? w : best;
          }
          if (VIT) {
            lead = on && c == best;
          } else {
            const unsigned long long term = on ? fix_exp64(v, dkey_inv(best)) : 0ull;
            sum = term;
            s = lane;
            for (int i = 1; i < most; ++i) {
              s = next_peer(peers, s);
              const unsigned long long w = __shfl_sync(FULL, term, s);
              if (i < __popc(peers)) sum += w;
            }
            lead = on && (peers & lanes_below()) == 0u;
          }
        }
        const uint32_t leads = __ballot_sync(FULL, lead);
        nb = __popc(leads);
        nbase = warp_reserve(gs, nb);
        if (nbase < 0) nb = 0;
        const int32_t i = __popc(leads & lanes_below());
        Arcs nxt{0, 0};
        first = make_int4(0, 0, 0, 0);
        if (lead && nb) {
          if constexpr (VIT) x.r = fkey_inv((uint32_t)(c >> 32));
          else x.r = fix_log_sum64(dkey_inv(best) - fx_widen(P.shift), sum);
          if (an >= 0) nxt = seg_find(L, pr, &first);
          first.w = 1;
          x.jp = nbase + i;
          if (VIT) {
            put(nbase + i, arc.x, x.r, (int32_t)(~(uint32_t)c), jp);
            put_arcs(fe, HS0 / 2, i, nxt);
          } else {
            put(nbase + i, arc.x, x.r, nxt.pos, nxt.len);
          }
        }
        x.e0 = nxt.pos;
        x.len = nxt.len;
        P.tot = (int32_t)__reduce_add_sync(FULL, (unsigned)x.len);
        if (!VIT) mk = __reduce_max_sync(FULL, lead && nb ? fkey64(x.r) : 0u);
        have = true;
      } else {
        for (int32_t c = 0; c < P.cnt; c += 32) {
          const int32_t total = stage(st, fe, P.t, P.base, a, c, P.cnt);
          walk_table<0>(tab, st, total, P.t == 1 ? -1 : P.base + c);
        }
        __syncwarp();
        nb = tab.staged;
        // a position where every destination has one arc needs no second
        // phase: the sum is that arc's term, exactly 1, and the arc the best
        const bool single = nb == P.tot;
        if (!VIT && !single)
          for (int32_t c = 0; c < P.cnt; c += 32) {
            const int32_t total = stage(st, fe, P.t, P.base, a, c, P.cnt);
            walk_table<1>(tab, st, total, P.t == 1 ? -1 : P.base + c);
          }
        nbase = warp_reserve(gs, nb);
        __syncwarp();
        int32_t tot = 0;
        uint32_t k = 0u;
        for (int32_t c = 0; c < nb; c += 32) {
          if (nbase < 0) {
            empty_table(tab, c, nb);
            continue;
          }
          int4 f = make_int4(0, 0, 0, 0);
          const Entry y = read_table(tab, c, nb, nbase, P.shift, single, an, fe, &f);
          tot += y.len;
          if (!VIT && c + lane < nb) k = max(k, fkey64(y.r));
          if (c == 0) {
            x = y;
            first = make_int4(f.x, f.y, f.z, 1);
          }
        }
        if (nbase < 0) nb = 0;
        P.tot = (int32_t)__reduce_add_sync(FULL, (unsigned)tot);
        mk = __reduce_max_sync(FULL, k);
        __syncwarp();
        if (lane == 0) tab.staged = 0;
        __syncwarp();
        have = true;
      }
      P.base = nbase;
      P.cnt = nb;
      if (lane == 0) {
        gs.live_e += (unsigned long long)nb;
        gs.live_a += (unsigned long long)P.tot;
        position_done(P, p, mk);
        report(K, P.t - 1, P.t);
      }
      P.shift = decode_max(mk);
      a = an;
      if (nb == 0) {
        ++P.t;
        break;
      }
    }
    if (hand < 0) dead_from(P, lane, 32);
    __syncwarp();
    if (lane == 0) leave(P, gs, b, hand);
  }

  // ---- heavy blocks ------------------------------------------------------
  // A chunk of a dense position (hv.job).
  __device__ __forceinline__ void chunk(HeavyShared& hv, BlockStage& st, int32_t c, int32_t* staged) const {
    const StringJob& J = hv.job;
    const int32_t lo = c * J.per;
    if (J.phase == 2) {
      int32_t tot = 0;
      uint32_t mk = 0u;
      const int32_t hi = min(lo + J.per, J.nb);
      for (int32_t i = lo + 64 * warp_id(); i < hi; i += 64 * WARPS)
        read_dense(J.owner, i, hi, J.nbase, J.shift, J.single != 0, J.an, &tot, &mk);
      tot = (int32_t)__reduce_add_sync(FULL, (unsigned)tot);
      mk = __reduce_max_sync(FULL, mk);
      if (lane_id() == 0) {
        if (tot) atomicAdd(J.shared ? &K.jobs[J.owner].tot : &hv.tot, (uint32_t)tot);
        if (mk) atomicMax(J.shared ? &K.jobs[J.owner].mk : &hv.mk, mk);
      }
      return;
    }
    const int32_t hi = min(lo + J.per, J.cnt);
    int32_t pend = 0;
    for (int32_t i0 = lo; i0 < hi; i0 += NT1 * BlockStage::PER) {
      const int32_t total = stage(st, fe_heavy(J.owner), J.t, J.base, J.a, i0, hi);
      if (J.phase == 0 && J.t == 1 && J.shared && threadIdx.x == 0) atomicAdd(&K.jobs[J.owner].tot, (uint32_t)total);
      if (J.phase == 0) walk_dense<0>(J.owner, staged, st, total, pend);
      else if constexpr (!VIT) walk_dense<1>(J.owner, nullptr, st, total, pend);
    }
    if (J.phase == 0) list_staged(J.owner, staged, st, pend);
  }

  // A heavy block's life, as one loop with one copy of each part (calls out
  // of line would keep the launch's parameters in local memory): it picks a
  // string, takes it from position to position, and works through chunks --
  // those of its own dense position, phase after phase, or other blocks'.
  __device__ __forceinline__ void heavy_block(BlockShared& sh) const {
    HeavyShared& hv = sh.hv;
    const int lane = lane_id(), tid = threadIdx.x;
    const int32_t self = hv.self;
    int2* fe = fe_heavy(self);
    HeavyPick pick;
    Place P{};
    int32_t b = -1, a = 0, an = -1, nb = 0;
    bool light = false, single = false;
    uint32_t mk = 0u;
    int own = -1;  // the phase of the own dense position (-1: none)
    for (;;) {
      bool help = false;
      if (b < 0) {
        const int32_t got = pick.next(hv, K, &light);
        if (got == PICK_LEAVE) return;
        if (got == PICK_NONE) {
          __nanosleep(1000);
          continue;
        }
        if (got == PICK_HELP) {
          help = true;
        } else {
          b = got;
          P = resume(b);
          a = P.n > 0 ? __ldg(sym + P.off + P.t - 1) : 0;
          if (P.t == 1 && P.cnt >= SHARE_ARCS) {
            // many start states: their arcs are counted as they are walked
            // (200,000 of them, looked up by one warp: a call of 6 symbols
            // took 10.6 ms; shared out it takes 0.1)
            P.tot = P.cnt;
          } else {
            if (tid == 0) hv.tot = 0u;
            __syncthreads();
            for (int32_t i = tid; i < P.cnt; i += NT1) P.tot += resume_entry(P, fe, S.Q, i, a);
            P.tot = (int32_t)__reduce_add_sync(FULL, (unsigned)P.tot);
            if (lane == 0 && P.tot) atomicAdd(&hv.tot, (uint32_t)P.tot);
            __syncthreads();
            P.tot = (int32_t)hv.tot;
          }
        }
      }
      bool done = false;  // position P.t is done
      if (!help && own < 0) {
        const bool over = P.t > P.n || P.cnt == 0 || P.tot == 0;
        if (over || (light && P.tot <= LIGHT_ARCS && P.cnt <= LIGHT_ARCS && P.n - P.t >= 2)) {
          if (over) dead_from(P, tid, NT1);
          __syncthreads();
          if (tid == 0) leave(P, sh.gs, b, over ? -1 : QL);
          __syncthreads();
          b = -1;
          continue;
        }
        an = P.t < P.n ? __ldg(sym + P.off + P.t) : -1;
        if (P.tot > HS1 / 2 || P.cnt >= SHARE_ARCS) {
          __syncthreads();  // (every thread has read hv.tot, hv.mk and hv.at of the position before)
          // (many entries with few arcs are work too: 176,615 of them with
          // 2,627 took a block by itself 860 us)
          const int32_t size = max(P.tot, P.cnt);
          const bool shared = size >= SHARE_ARCS;
          if (tid == 0) {
            StringJob& J = hv.job;
            hv.tag = ~0ull;
            J.phase = 0;
            J.owner = self;
            J.t = P.t;
            J.a = a;
            J.an = an;
            J.cnt = P.cnt;
            // (fewer than 2^31 arcs: the chunks' numbers fit JOB_BITS)
            J.per = shared ? (int32_t)min((long long)P.cnt, max(1ll, (long long)P.cnt * CHUNK_ARCS / size)) : P.cnt;
            if (P.t == 1 && P.cnt >= SHARE_ARCS) J.per = max(START_CHUNK, P.cnt >> (JOB_BITS - 1));
            J.base = P.base;
            J.shift = P.shift;
            J.shared = shared;
            J.staged = J.tot = J.mk = 0u;
            hv.tot = hv.mk = 0u;
          }
          own = 0;
          __syncthreads();
        } else {
          const uint32_t big = tid == 0 ? big_jobs(K) : 0u;  // (used below)
          for (int32_t c = 0; c < P.cnt; c += NT1 * BlockStage::PER) {
            const int32_t total = stage(sh.st, fe, P.t, P.base, a, c, P.cnt);
            walk_table<0>(sh.tab, sh.st, total, P.t == 1 ? -1 : P.base + c);
          }
          __syncthreads();
          nb = sh.tab.staged;
          single = nb == P.tot;
          if (tid == 0) {
            hv.base = reserve(sh.gs, nb);
            hv.tot = hv.mk = 0u;
            if (!light) hv.at = peek(K.ctl + CTL_ALIVE) != 0u;
          }
          if (!VIT && !single)
            for (int32_t c = 0; c < P.cnt; c += NT1 * BlockStage::PER) {
              const int32_t total = stage(sh.st, fe, P.t, P.base, a, c, P.cnt);
              walk_table<1>(sh.tab, sh.st, total, P.t == 1 ? -1 : P.base + c);
            }
          __syncthreads();
          const int32_t nbase = hv.base;
          if (tid == 0) sh.tab.staged = 0;
          int32_t tot = 0;
          uint32_t k = 0u;
          for (int32_t c = 32 * warp_id(); c < nb; c += NT1) {
            if (nbase < 0) {
              empty_table(sh.tab, c, nb);
              continue;
            }
            const Entry y = read_table(sh.tab, c, nb, nbase, P.shift, single, an, fe, nullptr);
            tot += y.len;
            if (!VIT && c + lane < nb) k = max(k, fkey64(y.r));
          }
          tot = (int32_t)__reduce_add_sync(FULL, (unsigned)tot);
          k = __reduce_max_sync(FULL, k);
          if (lane == 0 && tot) atomicAdd(&hv.tot, (uint32_t)tot);
          if (lane == 0 && k) atomicMax(&hv.mk, k);
          help = __syncthreads_or(big != 0u) != 0;
          P.base = nbase;
          P.cnt = nbase < 0 ? 0 : nb;
          P.tot = (int32_t)hv.tot;
          mk = hv.mk;
          light = hv.at != 0;  // (light blocks that began meanwhile)
          done = true;
        }
      }
      if (own >= 0 || help) {
        // the chunks: the own position's, all by itself or shared, or others'
        const bool mine = own >= 0, alone = mine && !hv.job.shared;
        const int32_t n = mine ? ((own == 2 ? hv.job.nb : hv.job.cnt) + hv.job.per - 1) / max(hv.job.per, 1) : 0;
        if (mine && !alone) job_post(hv, K, n);
        const int32_t least = b >= 0 ? BIG_CHUNKS : 1;
        int32_t g = mine ? self : job_find(hv, K, least), fin = -1;
        for (int32_t c = 0; g >= 0; ++c) {
          if (alone) {
            if (c >= n) break;
          } else {
            const bool got = job_claim(hv, K, g, fin, mine ? nullptr : pick.stop(K));
            fin = got ? g : -1;
            if (!got) {
              g = mine || hv.halt ? -1 : job_find(hv, K, least);
              continue;
            }
          }
          if (help) pick.helped();
          chunk(hv, sh.st, alone ? c : hv.chunk, alone ? &sh.tab.staged : (int32_t*)&K.jobs[g].staged);
        }
        if (mine) {
          if (alone) __syncthreads();
          else if (!job_wait(hv, K, n)) return;
          if (own == 0) {
            nb = alone ? sh.tab.staged : (int32_t)hv.job.staged;
            if (!alone && P.t == 1) P.tot = (int32_t)hv.job.tot;  // (start states: counted now)
            single = nb == P.tot;
          }
          __syncthreads();
          if (own == 0 && !VIT && !single) {
            if (tid == 0) {
              hv.job.phase = 1;
              hv.job.tot = 0u;
            }
            own = 1;
          } else if (own < 2) {
            if (tid == 0) {
              hv.job.tot = 0u;
              hv.base = reserve(sh.gs, nb);
              hv.job.phase = 2;
              hv.job.nb = nb;
              hv.job.nbase = hv.base;
              hv.job.single = single;
              hv.job.per = alone ? nb : 2 * 64 * WARPS;
              sh.tab.staged = 0;
            }
            __syncthreads();
            P.base = hv.base;
            own = 2;
            if (P.base < 0) {
              // empty what was staged
              for (int32_t i = tid; i < nb; i += NT1) {
                const int32_t d = __ldcg(dstage(self) + i);
                if (VIT) dacc(self)[d] = 0ull;
                else ((ulonglong2*)dacc(self))[d] = make_ulonglong2(0ull, 0ull);
              }
              P.cnt = P.tot = 0;
              done = true;
            }
          } else {
            P.cnt = nb;
            P.tot = (int32_t)(alone ? hv.tot : hv.job.tot);
            mk = alone ? hv.mk : hv.job.mk;
            done = true;
          }
          __syncthreads();
        }
      }
      if (done) {
        own = -1;
        if (tid == 0) {
          sh.gs.live_e += (unsigned long long)P.cnt;
          sh.gs.live_a += (unsigned long long)P.tot;
          position_done(P, P.off + P.t - 1, mk);
          report(K, P.t - 1, P.t);
        }
        P.shift = decode_max(mk);
        a = an;
        ++P.t;
      }
    }
  }
};

// What every block does first; true: it is a light one.
__device__ __forceinline__ bool block_begins(const StringQueue& K) {
  const bool light = (int32_t)blockIdx.x >= K.heavy_blocks;
  if (threadIdx.x == 0) {
    if (light) atomicAdd(K.ctl + CTL_ALIVE, (uint32_t)K.light_warps);
    __threadfence();
    atomicAdd(K.ctl + CTL_BEGUN, 1u);
  }
  __syncthreads();
  return light;
}

template <bool VIT>
__global__ void __launch_bounds__(NT1, 3)
    k_str_forward(const __grid_constant__ LayoutView L, const int32_t* __restrict__ sym,
                  const __grid_constant__ FrontierState S, const __grid_constant__ StringQueue K) {
  extern __shared__ __align__(16) unsigned char smem[];
  typedef Forward<VIT> F;
  if (block_begins(K)) {
    typename F::LightShared& sh = ((typename F::LightShared*)smem)[warp_id()];
    for (int i = lane_id(); i < HS0; i += 32) {
      sh.tab.acc[i] = 0ull;
      sh.tab.aux[i] = 0;
      sh.tab.key[i] = 0u;
    }
    if (lane_id() == 0) {
      sh.tab.staged = 0;
      sh.gs = GroupState{0, 0, 0ull, 0ull};
    }
    __syncwarp();
    const F f{L, sym, S, K};
    const int32_t g = ((int32_t)blockIdx.x - K.heavy_blocks) * WARPS + warp_id();
    while (warp_id() < K.light_warps) {
      const int32_t b = next_light(K);
      if (b < 0) break;
      f.light_string(sh.tab, sh.st, sh.gs, g, b);
      __syncwarp();
    }
    return;
  }
  typename F::BlockShared& sh = *(typename F::BlockShared*)smem;
  const int32_t self = (int32_t)blockIdx.x;
  for (int i = threadIdx.x; i < HS1; i += NT1) {
    sh.tab.acc[i] = 0ull;
    sh.tab.aux[i] = 0;
    sh.tab.key[i] = 0u;
  }
  if (threadIdx.x == 0) {
    sh.tab.staged = 0;
    sh.gs = GroupState{0, 0, 0ull, 0ull};
    sh.hv.self = self;
    sh.hv.tag = ~0ull;
  }
  __syncthreads();
  const F f{L, sym, S, K};
  if (self < K.owners && peek(K.dirty + self)) {
    // a run that gave up left values behind
    const int64_t w = (int64_t)S.Q * (VIT ? 1 : 2);
    for (int64_t i = threadIdx.x; i < w; i += NT1) f.dacc(self)[i] = 0ull;
    __syncthreads();
    if (threadIdx.x == 0) K.dirty[self] = 0u;
  }
  f.heavy_block(sh);
}

// ======================================================================
// Backward recursion and posteriors (Alg. 2), over the pool entries of the
// forward pass: a table holds the backward values of the states of position
// t while those of t-1 are formed.
// ======================================================================
// A warp's chunk of 32 entries.
struct BwdStage {
  double ra[32], m[32];
  unsigned long long acc[32];
  int32_t excl[32], e0[32];
};
// The values of up to CAP states, one table for each parity of the position.
template <int HS, int CAP>
struct BwdTable {
  double val[2][HS];
  uint32_t key[2][HS];
  uint16_t list[2][CAP];
};
typedef BwdTable<BHS0, LIGHT_CAP> BwdLightTable;
typedef BwdTable<BHS1, BHS1 / 2> BwdHeavyTable;
struct BwdLightShared {
  BwdStage st;
  BwdLightTable tab;
  StringJob job;
};
struct BwdBlockShared {
  BwdHeavyTable tab;
  BwdStage st[WARPS];
  HeavyShared hv;
};

template <int HS, int CAP>
struct Backward {
  typedef BwdTable<HS, CAP> Tab;
  static constexpr bool HEAVY = HS > BHS0;
  static constexpr int VU = HEAVY ? VU1 : VU0;
  const LayoutView& L;
  const int32_t* sym;
  const FrontierState& S;
  const CountView& C;
  const StringQueue& K;
  BwdStage& st;  // of this warp
  Tab& tab;

  __device__ __forceinline__ double* dval(int32_t g, int w) const { return K.dval + ((int64_t)g * 2 + w) * S.Q; }

  // Backward value of state d at position t (w = t & 1), in the dense array
  // or the table: the final weight at the string's last position.
  __device__ __forceinline__ double beta(const StringJob& J, int32_t d) const {
    if (J.last) return fx_widen(__ldg(S.theta_f + d));
    const int w = J.t & 1;
    if (HEAVY && J.cur_big) return __ldcg(dval(J.owner, w) + d);
    const uint32_t k = (uint32_t)d + 1u;
    uint32_t h = slot_of(k, HS - 1);
    for (int i = 0; i < HS; ++i) {
      const uint32_t x = tab.key[w][h];
      if (x == k) return tab.val[w][h];
      if (x == 0u) break;
      h = (h + 1) & (HS - 1);
    }
    return -INFINITY;
  }
  // theta_e + beta_t[q'] - e_t of an arc.
  __device__ __forceinline__ double term(const StringJob& J, const int4& arc) const {
    const float th = __int_as_float(arc.y);
    const double ub = beta(J, arc.x);
    return (dead32(th) || dead64(ub)) ? -INFINITY : fx_widen(th) + (ub - fx_widen(J.shift));
  }
  // The value of state q of position t (w = t & 1) into the table, as entry i.
  __device__ __forceinline__ void insert(int w, int32_t i, int32_t q, double v) const {
    const uint32_t k = (uint32_t)q + 1u;
    uint32_t h = slot_of(k, HS - 1);
    for (int x = 0; x < HS; ++x) {
      if (atomicCAS(tab.key[w] + h, 0u, k) == 0u) break;
      h = (h + 1) & (HS - 1);
    }
    if (!in_bounds(CHK_STAGE, i, CAP)) return;
    tab.val[w][h] = v;
    tab.list[w][i] = (uint16_t)h;
  }

  // Entry i (act: there is one) of position t-1, a warp's 32 together: its
  // backward value from its arcs on w_t, and their posteriors.  Returns the
  // order key of the value.
  __device__ __forceinline__ uint32_t sweep(const StringJob& J, int32_t i, bool act) const {
    const int lane = lane_id();
    int32_t e0 = 0, len = 0, q = -1;
    double ra = 0.0;
    if (act) {
      if (J.t == 1) {
        q = __ldg(S.start_q + i);
        ra = (double)__ldg(S.theta_s + q);
        const Arcs x = find_arcs(L, J.a, q);
        e0 = x.pos;
        len = x.len;
      } else if (in_bounds(CHK_POOL_READ, J.base + i, S.pool_cap)) {
        q = __ldg(S.pool_q + J.base + i);
        ra = __ldg(S.pool_d + J.base + i);
        e0 = __ldg(S.pool_x + J.base + i);
        len = __ldg(S.pool_n + J.base + i);
      }
      if (J.shift == neg_inf()) len = 0;
    }
    int32_t total;
    const int32_t ex = warp_excl(len, &total);
    __syncwarp();
    st.excl[lane] = ex;
    st.ra[lane] = ra;
    st.e0[lane] = e0;
    st.acc[lane] = 0ull;
    __syncwarp();
    // the first 32 * VU arcs stay in registers for the second sweep
    int oo[VU];
    int32_t id[VU];
    double v[VU];
    for (int32_t a0 = 0; a0 < total; a0 += 32 * VU) {
      int oi[VU];
      int4 arc[VU];
#pragma unroll
      for (int u = 0; u < VU; ++u) {
        const int32_t a = a0 + u * 32 + lane;
        oi[u] = a < total ? owner_of(st.excl, a) : -1;
        if (oi[u] >= 0 && !in_bounds(CHK_ARC, (long long)st.e0[oi[u]] + (a - st.excl[oi[u]]), L.P)) oi[u] = -1;
        arc[u] = oi[u] >= 0 ? __ldg(L.arcs + st.e0[oi[u]] + (a - st.excl[oi[u]])) : make_int4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < VU; ++u) {
        const double x = oi[u] >= 0 ? term(J, arc[u]) : -INFINITY;
        if (!dead64(x)) atomicMax(st.acc + oi[u], dkey(x));
        if (a0 == 0) {
          oo[u] = oi[u];
          id[u] = arc[u].z;
          v[u] = x;
        }
      }
    }
    __syncwarp();
    const unsigned long long mkk = st.acc[lane];
    const double m = mkk ? dkey_inv(mkk) : -INFINITY;
    st.m[lane] = m;
    st.acc[lane] = 0ull;
    __syncwarp();
    for (int32_t a0 = 0; a0 < total; a0 += 32 * VU) {
#pragma unroll
      for (int u = 0; u < VU; ++u) {
        if (a0 > 0) {
          const int32_t a = a0 + u * 32 + lane;
          oo[u] = a < total ? owner_of(st.excl, a) : -1;
          v[u] = -INFINITY;
          if (oo[u] >= 0 && in_bounds(CHK_ARC, (long long)st.e0[oo[u]] + (a - st.excl[oo[u]]), L.P)) {
            const int4 arc = __ldg(L.arcs + st.e0[oo[u]] + (a - st.excl[oo[u]]));
            v[u] = term(J, arc);
            id[u] = arc.z;
          }
        }
        if (oo[u] < 0 || dead64(v[u])) continue;
        // the exponent adds terms of either sign and tens in size that
        // cancel to a small number: formed in float64
        const double exn = st.ra[oo[u]] + v[u] + J.K;
        add_count(C, id[u], __expf(fx_narrow(exn)) * J.gw);
        atomicAdd(st.acc + oo[u], fix_exp64(v[u], st.m[oo[u]]));
      }
    }
    __syncwarp();
    uint32_t ek = 0u;
    if (q >= 0) {
      const double uv = fix_log_sum64(m, st.acc[lane]);
      if (J.t > 1) {
        const int w = (J.t & 1) ^ 1;
        if (HEAVY && J.next_big) {
          if (in_bounds(CHK_ACC, q, S.Q)) dval(J.owner, w)[q] = uv;
        } else {
          insert(w, i, q, uv);
        }
        ek = fkey64(uv);
      } else if (C.start64 && uv != -INFINITY) {
        // the item is a start state q, log beta_0[q] = u + E_1
        atomicAdd(C.start64 + q, exp(ra + uv + J.K) * (double)J.gw);
      }
    }
    return ek;
  }

  // A string at position t: E_{t+1}, the order key of e_t (the largest
  // backward value of position t), where the values of position t are and
  // their number.
  struct Place {
    int32_t n, t, cur_n;
    int64_t off;
    double lz, tE;
    uint32_t ek;
    float gw;
    bool cur_big;
  };
  __device__ __forceinline__ Place resume(int32_t b, int32_t first, int32_t step) const {
    Place P;
    P.lz = __ldg(S.logz + b);
    P.n = __ldg(S.bw_n + b);
    P.off = __ldg(S.bw_off + b);
    P.gw = S.gweight ? S.gweight[b] : 1.f;
    const int32_t t = __ldcg(&K.park[b].t);
    P.t = t > 0 ? t : P.n;
    P.tE = __ldcg(&K.park[b].tE);
    P.ek = __ldcg(&K.park[b].ek);
    P.cur_n = 0;
    P.cur_big = false;
    if (P.lz == -INFINITY) P.t = 0;
    if (P.t > 0 && P.t < P.n) {
      // the values of position t, kept in the order of its entries
      const int64_t base = __ldg(S.pool_base + P.off + P.t - 1);
      P.cur_n = __ldg(S.pool_cnt + P.off + P.t - 1);
      const double* kept = K.kept + (int64_t)b * LIGHT_CAP;
      for (int32_t i = first; i < P.cur_n; i += step) insert(P.t & 1, i, __ldg(S.pool_q + base + i), __ldcg(kept + i));
    }
    return P;
  }
  // The values of position t for whoever takes the string over; the table is
  // emptied.
  __device__ __forceinline__ void keep(const Place& P, int32_t g, int32_t b, int32_t first, int32_t step) const {
    const int w = P.t & 1;
    double* kept = K.kept + (int64_t)b * LIGHT_CAP;
    const int64_t base = P.t < P.n ? __ldg(S.pool_base + P.off + P.t - 1) : 0;
    for (int32_t i = first; i < P.cur_n; i += step) {
      if (!in_bounds(CHK_STAGE, i, LIGHT_CAP)) continue;
      if (HEAVY && P.cur_big) {
        kept[i] = __ldcg(dval(g, w) + __ldg(S.pool_q + base + i));
      } else {
        const int32_t h = tab.list[w][i];
        kept[i] = tab.val[w][h];
        tab.key[w][h] = 0u;
      }
    }
  }
  __device__ __forceinline__ void empty(const Place& P, int32_t first, int32_t step) const {
    const int w = P.t & 1;
    if (!P.cur_big)
      for (int32_t i = first; i < P.cur_n; i += step) tab.key[w][tab.list[w][i]] = 0u;
  }
  // Position t's parameters (one thread); the entries of t-1 and their arcs.
  struct Range {
    int64_t base;
    int32_t cnt;
    uint32_t tot;
  };
  __device__ __forceinline__ Range range(const Place& P) const {
    const int64_t p = P.off + P.t - 1;
    if (P.t == 1) return Range{0, S.nstart, 0u};
    return Range{__ldg(S.pool_base + p - 1), __ldg(S.pool_cnt + p - 1), __ldg(S.ekey + p - 1)};
  }
  __device__ __forceinline__ void fill(StringJob& J, const Place& P, const Range& R, int32_t g, float et, bool dense,
                                       bool shared) const {
    const int64_t p = P.off + P.t - 1;
    const float mprev = P.t == 1 ? 0.f : decode_max(__ldg(S.mkey + p - 1));
    J.owner = g;
    J.t = P.t;
    J.a = __ldg(sym + p);
    J.cnt = R.cnt;
    J.base = R.base;
    J.shift = et;
    J.gw = P.gw;
    J.K = ((P.t == 1 ? 0.0 : __ldg(S.csum + p - 1)) + P.tE - P.lz) - (double)mprev;
    J.last = P.t == P.n;
    J.cur_big = P.cur_big;
    J.next_big = dense;
    J.shared = shared;
    J.mk = 0u;
    J.per = (int32_t)min((long long)R.cnt, max(1ll, (long long)R.cnt * CHUNK_ARCS / max((uint32_t)R.cnt, R.tot)));
    report(K, P.t - 1, P.t);
  }
  __device__ __forceinline__ void leave(const Place& P, int32_t b, int32_t hand) const {
    if (hand >= 0) {
      K.park[b] = StringPark{P.t, P.ek, P.tE};
      queue_push(K, hand, b);
    } else {
      string_done(K);
    }
  }

  // Up to 32 positions, from P.t down, whose sources (t-1 >= 1) are one state
  // with one arc: everything but the chain of values itself is done a
  // position a lane.  The value of the first position's destination comes
  // from the table; each further one is the state before it.  Returns the
  // positions done.
  __device__ __forceinline__ int32_t chain(Place& P) const {
    const int lane = lane_id();
    const int32_t t = P.t - lane;  // this lane's position
    const int64_t p = P.off + t - 1;
    int64_t base = 0;
    bool one = false;
    if (t >= 2) {
      base = __ldg(S.pool_base + p - 1);
      one = __ldg(S.pool_cnt + p - 1) == 1 && __ldg(S.ekey + p - 1) == 1u;
    }
    const uint32_t ones = __ballot_sync(FULL, one);
    const int32_t m = ones == FULL ? 32 : __ffs(~ones) - 1;
    if (m < 2) return 0;
    int32_t q = 0;
    double ra = 0.0, th = 0.0, pre = 0.0;
    int4 arc = make_int4(0, 0, 0, 0);
    float mprev = 0.f;
    if (lane < m && in_bounds(CHK_POOL_READ, base, S.pool_cap)) {
      q = __ldg(S.pool_q + base);
      ra = __ldg(S.pool_d + base);
      const int32_t e = __ldg(S.pool_x + base);
      if (in_bounds(CHK_ARC, e, L.P)) arc = __ldg(L.arcs + e);
      mprev = decode_max(__ldg(S.mkey + p - 1));
      pre = __ldg(S.csum + p - 1);
    }
    th = fx_widen(__int_as_float(arc.y));
    // the value of the first position's destination
    StringJob J;
    J.t = P.t;
    J.last = P.t == P.n;
    J.cur_big = 0;
    double u = beta(J, __shfl_sync(FULL, arc.x, 0));
    float et = P.t == P.n ? 0.f : decode_max(P.ek);
    double tE = P.tE, my_x = 0.0, my_tE = 0.0;
    for (int32_t k = 0; k < m; ++k) {
      if (P.t - k < P.n) tE += fx_widen(et);
      const double tk = __shfl_sync(FULL, th, k);
      const double x = (dead64(tk) || dead64(u)) ? -INFINITY : tk + (u - fx_widen(et));
      if (lane == k) {
        my_x = x;
        my_tE = tE;
      }
      u = x;
      et = fx_narrow(x);
    }
    const bool on = lane < m && !dead64(my_x);
    float g = 0.f;
    if (on) {
      const double K0 = (pre + my_tE - P.lz) - (double)mprev;
      g = __expf(fx_narrow(ra + my_x + K0)) * P.gw;
    }
    // A string by itself: positions that use the same arc add to it one after
    // the other, so that its counts are the same bits every time (everywhere
    // else an arc has one writer a position, and barriers between positions).
    if (K.strings == 1) {
      const uint32_t same = __match_any_sync(FULL, on ? arc.z : -1 - lane);
      const int rank = __popc(same & lanes_below());
      const int ranks = (int)__reduce_max_sync(FULL, (unsigned)rank);
      for (int r = 0; r <= ranks; ++r) {
        if (on && rank == r) add_count(C, arc.z, g);
        __syncwarp();
      }
    } else if (on) {
      add_count(C, arc.z, g);
    }
    // the table: the values of position P.t out, the last one in
    empty(P, lane, 32);
    __syncwarp();
    const int32_t last_q = __shfl_sync(FULL, q, m - 1);
    P.t -= m;
    if (lane == 0) report(K, P.t, P.t + m);
    P.tE = tE;
    P.ek = fkey64(u);
    P.cur_n = 1;
    if (lane == 0) insert(P.t & 1, 0, last_q, u);
    __syncwarp();
    return m;
  }

  __device__ __forceinline__ void light_string(StringJob& J, int32_t b) const {
    const int lane = lane_id();
    Place P = resume(b, lane, 32);
    __syncwarp();
    int32_t hand = -1;
    for (; P.t >= 1; --P.t) {
      while (P.t >= 3 && chain(P) > 0) {
      }
      if (P.t < 1) break;
      const Range R = range(P);
      if (R.cnt > CAP || R.tot > 2u * CAP) {
        keep(P, 0, b, lane, 32);
        hand = QH;
        break;
      }
      const float et = P.t == P.n ? 0.f : decode_max(P.ek);
      if (P.t < P.n) P.tE += (double)et;
      if (lane == 0) fill(J, P, R, 0, et, false, false);
      __syncwarp();
      uint32_t ek = 0u;
      for (int32_t c = 0; c < R.cnt; c += 32) {
        const uint32_t k = sweep(J, c + lane, c + lane < R.cnt);
        ek = k > ek ? k : ek;
      }
      P.ek = __reduce_max_sync(FULL, ek);
      empty(P, lane, 32);
      __syncwarp();
      P.cur_n = P.t > 1 ? R.cnt : 0;
    }
    __syncwarp();
    if (lane == 0) leave(P, b, hand);
  }

  // A chunk of a shared position (hv.job), or all of the block's own.
  __device__ __forceinline__ void chunk(HeavyShared& hv, int32_t c) const {
    const StringJob& J = hv.job;
    const int32_t per = J.shared ? J.per : J.cnt, lo = c * per, hi = min(lo + per, J.cnt);
    uint32_t ek = 0u;
    // (few entries of many arcs are spread over the warps: 50 entries of 20 arcs
    // in two of them took 59 us a position, 19 so)
    const int32_t each = min(32, (hi - lo + WARPS - 1) / WARPS);
    for (int32_t i0 = lo + each * warp_id(); i0 < hi; i0 += each * WARPS) {
      const bool act = lane_id() < each && i0 + lane_id() < hi;
      const uint32_t k = sweep(J, i0 + lane_id(), act);
      ek = k > ek ? k : ek;
    }
    ek = __reduce_max_sync(FULL, ek);
    if (lane_id() == 0 && ek) atomicMax(J.shared ? &K.jobs[J.owner].mk : &hv.mk, ek);
  }

  // A heavy block's life, as in the forward pass.
  __device__ __forceinline__ void heavy_block(HeavyShared& hv) const {
    const int tid = threadIdx.x;
    const int32_t self = hv.self;
    HeavyPick pick;
    Place P{};
    Range R{};
    int32_t b = -1;
    bool light = false;
    for (;;) {
      bool help = false, mine = false, dense = false;
      uint32_t big = 0u;
      if (b < 0) {
        const int32_t got = pick.next(hv, K, &light);
        if (got == PICK_LEAVE) return;
        if (got == PICK_NONE) {
          __nanosleep(1000);
          continue;
        }
        if (got == PICK_HELP) {
          help = true;
        } else {
          b = got;
          P = resume(b, tid, NT1);
          __syncthreads();
        }
      }
      if (!help) {
        if (P.t >= 1) R = range(P);
        const bool hand = P.t >= 3 && light && P.t < P.n && R.cnt <= LIGHT_ARCS && R.tot <= (uint32_t)LIGHT_ARCS &&
                          P.cur_n <= LIGHT_CAP;
        if (P.t < 1 || hand) {
          if (hand) keep(P, self, b, tid, NT1);
          __syncthreads();
          if (tid == 0) leave(P, b, hand ? QL : -1);
          __syncthreads();
          b = -1;
          continue;
        }
        const float et = P.t == P.n ? 0.f : decode_max(P.ek);
        if (P.t < P.n) P.tE += (double)et;
        const bool shared = max((uint32_t)R.cnt, R.tot) >= (uint32_t)SHARE_ARCS;
        dense = R.cnt > CAP || shared;  // where the values of t-1 go
        big = tid == 0 ? big_jobs(K) : 0u;  // (used below)
        if (shared && P.t < P.n && !P.cur_big) {
          // the values of position t where every block finds them
          const int w = P.t & 1;
          double* dv = dval(self, w);
          for (int32_t i = tid; i < P.cur_n; i += NT1) {
            const int32_t h = tab.list[w][i];
            dv[tab.key[w][h] - 1u] = tab.val[w][h];
            tab.key[w][h] = 0u;
          }
          P.cur_big = true;
        }
        if (tid == 0) {
          hv.tag = ~0ull;
          fill(hv.job, P, R, self, et, dense, shared);
          hv.mk = 0u;
          if (!light) hv.at = peek(K.ctl + CTL_ALIVE) != 0u;
        }
        mine = true;
        __syncthreads();
        light = hv.at != 0;  // (light blocks that began meanwhile)
      }
      // the chunks: the own position's, all by itself or shared, or, between
      // two positions, others'
      for (int round = 0; round < 2; ++round) {
        const bool alone = mine && !hv.job.shared;
        const int32_t n = mine ? (alone ? 1 : (R.cnt + hv.job.per - 1) / max(hv.job.per, 1)) : 0;
        if (mine && !alone) job_post(hv, K, n);
        const int32_t least = b >= 0 ? BIG_CHUNKS : 1;
        int32_t g = mine ? self : job_find(hv, K, least), fin = -1;
        for (int32_t c = 0; g >= 0; ++c) {
          if (alone) {
            if (c >= n) break;
          } else {
            const bool got = job_claim(hv, K, g, fin, mine ? nullptr : pick.stop(K));
            fin = got ? g : -1;
            if (!got) {
              g = mine || hv.halt ? -1 : job_find(hv, K, least);
              continue;
            }
          }
          if (help) pick.helped();
          chunk(hv, alone ? c : hv.chunk);
        }
        if (!mine) break;
        if (alone) __syncthreads();
        else if (!job_wait(hv, K, n)) return;
        P.ek = alone ? hv.mk : hv.job.mk;
        // the values of position t have been read: empty their table
        empty(P, tid, NT1);
        help = __syncthreads_or(big != 0u) != 0;
        P.cur_big = dense;
        P.cur_n = P.t > 1 ? R.cnt : 0;
        --P.t;
        mine = false;
        if (!help) break;
      }
    }
  }
};

__global__ void __launch_bounds__(NT1, 3)
    k_str_backward(const __grid_constant__ LayoutView L, const int32_t* __restrict__ sym,
                   const __grid_constant__ FrontierState S, const __grid_constant__ CountView C,
                   const __grid_constant__ StringQueue K) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (block_begins(K)) {
    BwdLightShared& sh = ((BwdLightShared*)smem)[warp_id()];
    for (int i = lane_id(); i < BHS0; i += 32) sh.tab.key[0][i] = sh.tab.key[1][i] = 0u;
    __syncwarp();
    const Backward<BHS0, LIGHT_CAP> w{L, sym, S, C, K, sh.st, sh.tab};
    while (warp_id() < K.light_warps) {
      const int32_t b = next_light(K);
      if (b < 0) break;
      w.light_string(sh.job, b);
      __syncwarp();
    }
    return;
  }
  BwdBlockShared& sh = *(BwdBlockShared*)smem;
  for (int i = threadIdx.x; i < BHS1; i += NT1) sh.tab.key[0][i] = sh.tab.key[1][i] = 0u;
  if (threadIdx.x == 0) {
    sh.hv.self = (int32_t)blockIdx.x;
    sh.hv.tag = ~0ull;
  }
  __syncthreads();
  const Backward<BHS1, BHS1 / 2> w{L, sym, S, C, K, sh.st[warp_id()], sh.tab};
  w.heavy_block(sh.hv);
}

// ======================================================================
// Backtrace of the forward pass's entries: a block per string.  An entry
// names its predecessor entry, except (-2) in the positions that took dense
// accumulators, where the block finds the best arc's source among the
// previous token's entries.
// ======================================================================
constexpr int TT = 256;
__global__ void __launch_bounds__(TT) k_str_trace(FrontierState S, const int32_t* __restrict__ olabel_by_id,
                                                  const int32_t* __restrict__ jfinal, int32_t* __restrict__ paths,
                                                  int32_t* __restrict__ olabels) {
  __shared__ int32_t found;
  const int64_t b = blockIdx.x;
  const int32_t n = S.bw_n[b];
  const int64_t off = S.bw_off[b];
  int32_t j = jfinal[b];
  int32_t t = n;
  for (; t >= 1 && j >= 0; --t) {
    const int32_t id = S.pool_x[j], pn = S.pool_n[j];
    if (threadIdx.x == 0) paths[off + t - 1] = id;
    if (pn != -2) {
      j = pn;
      continue;
    }
    if (threadIdx.x == 0) found = -1;
    __syncthreads();
    if (t > 1) {
      const int32_t src = __ldg(S.src_by_id + id);
      const int64_t base = S.pool_base[off + t - 2];
      const int32_t cnt = S.pool_cnt[off + t - 2];
      constexpr int TU = 8;
      for (int32_t i0 = 0; i0 < cnt; i0 += TT * TU) {
        int32_t q[TU];
#pragma unroll
        for (int u = 0; u < TU; ++u) {
          const int32_t i = i0 + u * TT + (int32_t)threadIdx.x;
          q[u] = i < cnt ? __ldg(S.pool_q + base + i) : -1;
        }
        bool hit = false;
#pragma unroll
        for (int u = 0; u < TU; ++u)
          if (q[u] == src) {
            hit = true;
            found = (int32_t)(base + i0 + u * TT + (int32_t)threadIdx.x);
          }
        if (__syncthreads_or(hit)) break;  // the same answer in every thread
      }
    }
    __syncthreads();
    j = found;
    __syncthreads();
  }
  __syncthreads();
  if (olabels)
    for (int32_t u = t + (int32_t)threadIdx.x; u < n; u += TT) olabels[off + u] = __ldg(olabel_by_id + paths[off + u]);
  for (int32_t u = threadIdx.x; u < t; u += TT) {  // no path (or an entry chain cut short): markers
    paths[off + u] = -1;
    if (olabels) olabels[off + u] = -1;
  }
}

inline int check_launch(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, what);
  return FST_OK;
}

// Blocks of a string kernel that are resident at once, looked up once per
// device: its heavy blocks share positions among them.
template <class K>
int resident(K kernel, int which, size_t smem, int num_sms, int* out) {
  static std::atomic<int> cache[3][64];
  int dev = 0;
  FST_CUDA(cudaGetDevice(&dev));
  const bool keep = dev >= 0 && dev < 64;
  if (keep && (*out = cache[which][dev].load()) > 0) return FST_OK;
  FST_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int nb = 0;
  FST_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, NT1, smem));
  if (nb < 1) {
    set_error("a string kernel does not fit the device");
    return FST_ERR_UNSUPPORTED;
  }
  *out = nb * num_sms;
  if (keep) cache[which][dev].store(*out);
  return FST_OK;
}

// The queues and roles of a launch of at most `blocks` blocks: a quarter of
// them light, up to half where that gives every string a warp at once, the
// others heavy.  (The few dense positions are most of the work: with half of
// the blocks light, Viterbi of 4,096 strings on 20M arcs took 3.5 ms instead
// of 3.0, with an eighth 3.3; a training step of 1,024 strings whose last 112
// wait for a warp took 0.92 ms instead of 0.87.)
// Launches of W.share parts on streams of their own divide the blocks among
// them: blocks that wait for a place serve their strings late and by the
// wrong role (sixteen forward-backward parts of 256 strings: 32 ms a step).
StringQueue string_queue(const StringWork& W, int blocks, int32_t* grid) {
  blocks = std::max(blocks / std::max(W.share, 1), 8);
  StringQueue K;
  K.strings = W.Bw;
  K.ctl = W.ctl;
  K.owners = W.groups2;
  uint32_t ring = 1;
  while (ring < (uint32_t)W.Bw) ring <<= 1;
  ring <<= 1;
  K.jobs = (StringJob*)(W.ctl + CTL_WORDS);
  K.ring = W.ctl + CTL_WORDS + (int64_t)W.groups2 * (sizeof(StringJob) / 4);
  K.ring_mask = ring - 1u;
  K.park = (StringPark*)(K.ring + 2 * (size_t)ring);
  K.dirty = W.dirty;
  K.kept = W.kept;
  K.dense = W.dense;
  K.dval = W.dval;
  K.dstage = W.dstage;
  K.fe = W.fe;
  K.fe_light = W.fe_light;
  K.chunk = W.chunk;
  K.limit_ns = W.limit_ns;
  K.spoiled = nullptr;
  // (waiting workers of few strings look at every poll, a microsecond: a kept
  // plan of one string of 3 symbols took 45 us for Viterbi and 85 for forward-
  // backward with a look at every eighth, 33 and 61 so; launches per position
  // 38 and 64)
  K.polls = W.Bw <= 64 ? 1u : 8u;
  // (heavy blocks come first, so that they are resident first)
  const int all = (W.Bw + WARPS - 1) / WARPS;
  const int want = all <= blocks / 2 ? std::max(all, blocks / 4) : blocks / 4;
  K.heavy_blocks = std::max(blocks - want, 1);
  // few strings are spread over the blocks
  const int light = std::max(1, std::min(blocks - K.heavy_blocks, W.Bw));
  K.light_warps = std::max(1, std::min(WARPS, (W.Bw + light - 1) / light));
  *grid = K.heavy_blocks + light;
  return K;
}

template <bool VIT>
int launch_forward(int which, const LayoutView& L, const int32_t* sym, const FrontierState& S, const StringWork& W,
                   int num_sms, cudaStream_t s) {
  const size_t smem = std::max(sizeof(typename Forward<VIT>::LightShared) * WARPS,
                               sizeof(typename Forward<VIT>::BlockShared));
  int blocks = 0;
  int32_t grid = 0;
  const int rc = resident(k_str_forward<VIT>, which, smem, num_sms, &blocks);
  if (rc) return rc;
  const StringQueue K = string_queue(W, blocks, &grid);
  k_str_forward<VIT><<<(unsigned)grid, NT1, smem, s>>>(L, sym, S, K);
  return check_launch("k_str_forward");
}

}  // namespace

int64_t string_ctl_words(int32_t Bw, int32_t groups2) {
  int64_t ring = 1;
  while (ring < Bw) ring <<= 1;
  ring <<= 1;
  return CTL_WORDS + (int64_t)groups2 * (int64_t)(sizeof(StringJob) / 4) + 2 * ring +
         (int64_t)Bw * (int64_t)(sizeof(StringPark) / 4) + 2;
}
int64_t string_light_entries(int num_sms, int64_t Bw) {
  // (at most one light block a string, and half of what is resident)
  return std::min<int64_t>((int64_t)num_sms * 4, std::max<int64_t>(Bw, 1)) * WARPS * (HS0 / 2);
}
int32_t string_kept_values() { return LIGHT_CAP; }

int launch_string_forward(bool viterbi, const LayoutView& L, const int32_t* sym, const FrontierState& S,
                          const StringWork& W, int num_sms, cudaStream_t s) {
  FST_CUDA(cudaMemsetAsync(W.ctl, 0, (size_t)string_ctl_words(W.Bw, W.groups2) * 4, s));
  if (W.Bw <= 0) return FST_OK;
  return viterbi ? launch_forward<true>(0, L, sym, S, W, num_sms, s) : launch_forward<false>(1, L, sym, S, W, num_sms, s);
}

int launch_string_backward(const LayoutView& L, const int32_t* sym, const FrontierState& S, const CountView& C,
                           const StringWork& W, int num_sms, cudaStream_t s) {
  if (W.Bw <= 0) return FST_OK;
  FST_CUDA(cudaMemsetAsync(W.ctl + CTL_TAKE, 0, (size_t)(string_ctl_words(W.Bw, W.groups2) - CTL_TAKE) * 4, s));
  const size_t smem = std::max(sizeof(BwdLightShared) * WARPS, sizeof(BwdBlockShared));
  int blocks = 0;
  int32_t grid = 0;
  const int rc = resident(k_str_backward, 2, smem, num_sms, &blocks);
  if (rc) return rc;
  StringQueue K = string_queue(W, blocks, &grid);
  K.spoiled = C.spoiled;
  k_str_backward<<<(unsigned)grid, NT1, smem, s>>>(L, sym, S, C, K);
  return check_launch("k_str_backward");
}

int launch_string_trace(const FrontierState& S, const int32_t* olabel_by_id, int32_t Bw, const int32_t* jfinal,
                        int32_t* paths, int32_t* olabels, cudaStream_t s) {
  if (Bw <= 0) return FST_OK;
  k_str_trace<<<(unsigned)Bw, TT, 0, s>>>(S, olabel_by_id, jfinal, paths, olabels);
  return check_launch("k_str_trace");
}

}  // namespace fstgpu
