// kernels.cuh -- launch arguments of the frontier kernels (kernels.cu).
#pragma once

#include <stdint.h>

#include "fst_internal.cuh"

namespace fstgpu {

// Device view of the source-segmented arc layout: the arcs out of state q
// on symbol a are consecutive, found through a (symbol, state) hash.
struct LayoutView {
  const int4* arcs;            // [P] {destination, theta bits, caller id, 0}
  const SegSlot* seg_hash;     // (symbol, state) -> arcs
  int64_t buckets;
  int64_t P;                   // arc records (the bounds-checked build checks against it)
};

inline LayoutView view_of(const Layout& L) { return LayoutView{L.arcs, L.seg_hash, L.buckets, L.P}; }

// The tokens of one input position t: slots slot0 .. slot0+n-1 of the
// step list T.step_tok (tokens of a wave in step order).  Token p is
// position t of wave-local string T.b[p]; the tokens of a string are
// consecutive, so the previous position of token p is token p - 1.  The x_*
// fields name a second position the kernel also works on: the next one for
// the forward steps (whose new live states they push there), the previous
// one for the kernels that walk the live states of t-1 (x_n = 0: none).
struct StepView {
  int32_t t;
  int32_t n;
  int32_t slot0;
  int32_t x_t, x_n, x_slot0;
  int32_t blocks;   // grid of the launch (work is a grid-stride loop)
  int32_t y_t;      // backward steps with compact accumulators: the position whose
                    // backward values this step clears (0: none)
};

struct TokenView {
  const int32_t* step_tok;  // [N] token of each step slot
  const int32_t* sym;
  const int32_t* b;
  const int64_t* stf;   // staging offset of the token inside its step
};

// State of one wave (or of one plain-method string).
//
// Accumulators, in one of two layouts, all empty between runs:
//   dense   -- per string, two parity buffers of Q slots each (the plain
//              method's single string, and plans made with
//              FST_PLAN_DENSE_ACC);
//   compact -- open-addressing hash tables keyed by (string, state), one per
//              position parity, sized for the live states of a position
//              rather than for every state of every string: a few MB that
//              stay in L2, where the dense arrays of a large batch take tens
//              of GB.  The staging lists then hold table slots.
// In both, a forward step pushes every arc out of a live state of position
// t into the accumulator of its destination at t+1 with an atomic max (the
// packed Viterbi key, or the forward maximum); the push that finds the
// accumulator empty (or inserts its key) stages the destination.  The next
// step reads each staged accumulator once, turns it into a live-pool entry
// and empties it.
//
// Live pool: for every token, the states with a finite value at its
// position: the state, its value, and the best incoming arc (Viterbi) or
// the segment of its arcs on the next symbol (forward).  The last block of a
// step hands out the pool ranges: the step's tokens get consecutive ranges
// in step order, so one position's entries are one flat range that the next
// kernels split evenly over blocks, whatever the tokens' frontier sizes.
struct FrontierState {
  int32_t Q;
  // dense: [Bw][2][Q] accumulators of acc_stride 64-bit words: Viterbi keys
  // use the first word; the forward passes need stride 2, {fixed-point sum,
  // maximum order key in the low half}, so that both sit on one cache line
  unsigned long long* acc;
  int32_t acc_stride;
  double* beta;                      // [Bw][2][Q] backward values, float64 (null for Viterbi-only state)
  int32_t* vmap;                     // [Bw][2][Q] Viterbi: pool entry of each live state (null for forward-only state)
  // compact (hmask > 0): tables of hmask + 1 slots, key (wave-local string
  // + 1) << 32 | state (0 = empty).  htab0 / htab1 hold the positions of even / odd
  // parity, 2 acc_stride words a slot: {key, Viterbi key} or {key, maximum
  // order key, fixed-point sum, 0}.  btab0..2 hold the backward values of
  // the positions t with t mod 3 = 0, 1, 2, {key, float64 bits}; bslot maps
  // each pool entry to its slot there (-1: none).  Viterbi needs no state
  // map: the backtrace finds each predecessor among its token's entries.
  unsigned long long* htab0;
  unsigned long long* htab1;
  unsigned long long* btab0;
  unsigned long long* btab1;
  unsigned long long* btab2;
  int32_t* bslot;
  uint64_t hmask;
  // Direction switch of the forward pass (dense accumulators, launch
  // driver; dense_min = 0: off).  A token with at least dense_min live
  // states, whose string goes on and whose next symbol's slice has no
  // segment longer than a window (pull_lseg), gets one of DENSE_SLOTS dense
  // value vectors for its position: the forward step scatters its values
  // there instead of pushing its arcs, and the next position pulls over
  // the destination-ordered slice.  dvec [DENSE_SLOTS][2][Q] float64 (-inf
  // between uses), dslot [N] the slot of each token (-1: none), dlist
  // [T+2][DENSE_SLOTS] the dense tokens of each position, dcnt [T+2] their
  // number.
  double* dvec;
  int32_t* dslot;
  int32_t* dlist;
  int32_t* dcnt;
  const int64_t* pull_lseg;  // [m+1] long segments of the destination-ordered slices before each symbol
  int32_t dense_min;
  const int32_t* src_by_id;          // [A] source state of each arc
  int32_t* stage;                    // staged destinations of positions of even parity
  int32_t* stage_b;                  // of odd parity
  int64_t stage_cap;                 // entries of each staging buffer
  int32_t Bw;                        // strings of the wave (dense accumulators: [Bw][2][Q])
  int32_t chain;                     // host only: launch the step kernels chained to their predecessor
  uint32_t* scnt;                    // [N] destinations staged per token
  int32_t* pool_q;                   // [cap] state
  int32_t* pool_x;                   // [cap] Viterbi: best incoming arc id; forward: first arc on the next symbol
  int32_t* pool_n;                   // [cap] Viterbi: pool entry of the best arc's source (-1 at the first
                                     // position); forward: arcs on the next symbol
  float* pool_v;                     // [cap] Viterbi score
  double* pool_d;                    // [cap] forward value r_t, float64 (may share pool_v's storage)
  int64_t* pool_base;                // [N] by token
  int32_t* pool_cnt;                 // [N] by token
  int64_t* slot_base;                // [N] by step slot: first pool entry of the slot's token
  int64_t* step_rng;                 // [2 (T+2)]: pool entries [begin, end) of each position
  int64_t* pool_top;                 // [1] entries handed out in this run
  int64_t pool_cap;
  uint32_t* flags;                   // [2]: last-block counter, error bits (1 = pool full)
  const float* theta_s;
  const float* theta_f;
  const int32_t* start_q;            // states with a finite start weight
  int32_t nstart;
  uint32_t* mkey;                    // [N] forward step maxima (order keys)
  uint32_t* ekey;                    // [N] backward step maxima
  double* csum;                      // [N] C_t = sum_{s<=t} m_s
  double* esum;                      // [N] E_t
  const double* logz;                // [Bw]
  const float* gweight;              // [Bw] or null
  const int32_t* bw_n;               // [Bw] string lengths
  const int64_t* bw_off;             // [Bw] first token of each string
};

constexpr int DENSE_SLOTS = 16;

// The destination-ordered slices the pull reads: records {source,
// destination, caller id (< 0: padding), 0}, weights, and each symbol's
// 128-arc windows [win[a], win[a+1]).
struct PullView {
  const int4* rec;
  const float* theta;
  const int64_t* win;
};

// Step offsets of a wave on the device, for the persistent passes: the
// tokens of position t are step slots step0[t] .. step0[t+1]-1.
struct WaveSteps {
  const int32_t* step0;  // [tmax + 2]
  int32_t tmax;
};

// Grid barrier of a persistent pass: bar[0] counts arrivals, bar[1] is the
// generation; a wait gives up after limit_ns.  `expected` is the number of
// blocks that meet at each barrier beyond the grid (0 in normal use; a
// fault-injection setting raises it so that the wait runs out).
struct GridSync {
  uint32_t* bar;
  uint32_t expected;
  uint64_t limit_ns;
};

// Expected counts by caller arc id.
struct CountView {
  int batched;        // 0: Kahan float pair (one string); 1: double atomics
  float* cnt;
  float* comp;
  double* cnt64;
  double* start64;    // [Q] expected start states, or null
  double* final64;    // [Q] expected final states, or null
  double* spoiled = nullptr;  // [1] NaN once a backward pass gave up waiting, else 0: the counts are partial
};

// First position (Viterbi and forward): the start states push their arcs
// on w_1 into the accumulators of position 1.
int launch_vit_first(const LayoutView& L, const TokenView& T, const StepView& V, const FrontierState& S,
                     cudaStream_t s);
int launch_fwd_first(const LayoutView& L, const TokenView& T, const StepView& V, const FrontierState& S,
                     cudaStream_t s);
// One position of the forward passes: each staged destination of position
// t becomes a pool entry (its accumulator is read and cleared), and each
// new live state at once pushes its arcs on w_{t+1} into the accumulators
// of position t+1.  V.x_* name position t+1 (x_n = 0 at a wave's last
// position).
int launch_vit_step(const LayoutView& L, const TokenView& T, const StepView& V, const FrontierState& S,
                    cudaStream_t s);
int launch_fwd_step(const LayoutView& L, const TokenView& T, const StepView& V, const FrontierState& S,
                    cudaStream_t s);
// Forward sum of position t: the live states of t-1 (V.x_*) add
// exp(value - maximum) of each arc to its destination's accumulator.  With
// the direction switch, the dense tokens of t-1 pull over R (maxima, terms
// and sums of their destinations at once), and the last block hands out
// the pool ranges of t.
int launch_fwd_sum(const LayoutView& L, const TokenView& T, const StepView& V, const FrontierState& S,
                   const PullView& R, cudaStream_t s);

// Backward step of position t: for each live state q of position t-1
// (V.x_*), beta_{t-1}[q] over its arcs on w_t, and the posterior of each of
// those arcs.
int launch_bwd_step(const LayoutView& L, const TokenView& T, const StepView& V, const FrontierState& S,
                    const CountView& C, cudaStream_t s);
// Persistent passes (one cooperative launch of `grid` blocks runs every
// position of the wave, separated by bounded grid barriers).  `grid` must be
// co-resident: at most persist_grid_limit(0: Viterbi, 1: forward,
// 2: backward); FST_ERR_UNSUPPORTED otherwise.  G.bar must be zero.
int persist_grid_limit(int which);
int launch_vit_persist(const LayoutView& L, const TokenView& T, const WaveSteps& D, const FrontierState& S,
                       int32_t grid, const GridSync& G, cudaStream_t s);
int launch_fwd_persist(const LayoutView& L, const TokenView& T, const WaveSteps& D, const FrontierState& S,
                       int32_t grid, const GridSync& G, cudaStream_t s);
int launch_bwd_persist(const LayoutView& L, const TokenView& T, const WaveSteps& D, const FrontierState& S,
                       const CountView& C, int32_t grid, const GridSync& G, cudaStream_t s);
// Best final state of each string; jfinal gets its pool entry (-1: no path).
int launch_vit_final(const FrontierState& S, int32_t Bw, float* scores, int32_t* jfinal, int32_t* status,
                     cudaStream_t s);
// The best path of each string, following the pool entries' predecessors.
int launch_backtrace(const FrontierState& S, const int32_t* olabel_by_id, int32_t Bw, const int32_t* jfinal,
                     int32_t* paths, int32_t* olabels, cudaStream_t s);
int launch_fb_final(const FrontierState& S, int32_t Bw, double* logz, int32_t* status, cudaStream_t s);
// Counts as float32, out[0..A); where a backward pass gave up, NaN, and
// FST_ERR_TIMEOUT in status[0..B) (null: none).
int launch_counts_out(int64_t A, const CountView& C, float* out, int32_t B, int32_t* status, cudaStream_t s);
// Expected final states of every string (and expected start states of the
// empty strings, whose paths start where they end), added to C.final64 and
// C.start64 with the strings' weights.  Needs the forward pass and log Z.
int launch_final_posteriors(const FrontierState& S, int32_t Bw, const CountView& C, cudaStream_t s);
// p[i] = -inf, i < n.
int launch_fill_neg_inf(double* p, int64_t n, cudaStream_t s);
// out[i] = (float)in[i], i < n; NaN where a backward pass gave up.
int launch_to_float(const double* in, int64_t n, float* out, const double* spoiled, cudaStream_t s);
// The string kernels (strings.cu): a warp or block runs one string over all
// of its positions.  Control words of a wave's run: error flags, pool top,
// live entries and arcs; then, cleared before each pass, the strings started
// and finished, a counter of progress, the open jobs, the heads and tails of
// the two queues, the blocks that have begun, the light warps at work and the
// open jobs of many chunks, and the heavy blocks without a string.
// Each on a cache line of its own: they are polled.
enum : int {
  CTL_FLAGS = 0, CTL_TOP = 2, CTL_LIVE = 4, CTL_TAKE = 32, CTL_FINISHED = 64, CTL_PROGRESS = 96, CTL_OPEN = 128,
  CTL_BIG = 129, CTL_IDLE = 130, CTL_HEAD = 160, CTL_TAIL = 224, CTL_BEGUN = 288, CTL_ALIVE = 289, CTL_WORDS = 320,
  CTL_LINE = 32
};
// Where a string was left when it changed hands (t = 0: not started), and
// what its backward pass has so far.
struct StringPark {
  int32_t t;
  uint32_t ek;
  double tE;
};
// A position that a heavy block shares out in chunks (strings.cu).
struct alignas(128) StringJob {
  unsigned long long word;  // phase number, chunks, next chunk
  uint32_t done;            // chunks finished
  uint32_t staged;          // destinations staged (forward, phase 0)
  uint32_t tot, mk;         // arcs of the new entries; order key of the largest value
  int32_t phase, owner;
  int32_t t, a, an;         // position, its symbol, the next symbol (-1: none)
  int32_t cnt, per;         // entries of t-1, entries a chunk
  int32_t nb;               // entries of t
  int32_t base, nbase;      // their pool ranges
  double K;                 // backward: C_{t-1} + E_t - log Z - m_{t-1}
  float shift, gw;          // m_{t-1} (forward) or e_t (backward); the string's weight
  int32_t single, last;     // every destination has one arc; t is the last position
  int32_t cur_big, next_big;  // backward: the values of t and t-1 are in the dense arrays
  int32_t shared;           // its chunks are open to other blocks
};
// Waits of the string kernels give up after this long without progress
// anywhere in the launch, unless a plan sets another limit: the run then
// reports FST_ERR_TIMEOUT.
constexpr uint64_t STRING_WAIT_NS = 2000000000ull;
// Device storage of the string kernels.
struct StringWork {
  int32_t Bw;
  uint32_t* ctl;              // [string_ctl_words] control words, jobs, queues and places of the strings
  uint32_t* dirty;            // [groups2] the block's dense accumulators were left unclean
  double* kept;               // [Bw][string_kept_values()] backward values of a string that changes hands
  unsigned long long* dense;  // [groups2][Q] (Viterbi) or [groups2][Q][2] accumulators, zero between runs
  double* dval;               // [groups2][2][Q] backward values
  int32_t* dstage;            // [groups2][Q] staged states
  int2* fe;                   // arcs of the last position's entries (Viterbi): [groups2][Q], then the light warps'
  int64_t fe_light;           // where the light warps' begin
  int32_t groups2;            // heavy blocks that run strings
  int32_t chunk;              // pool entries a group reserves at a time (0: each range by itself)
  int32_t share = 1;          // launches like this one that run side by side
  uint64_t limit_ns = STRING_WAIT_NS;  // waits give up after this long without progress
};
// What a launch sees of it.
struct StringQueue {
  int32_t strings, heavy_blocks, light_warps, owners;
  uint32_t* ctl;
  StringJob* jobs;
  uint32_t* ring;
  uint32_t ring_mask;
  StringPark* park;
  uint32_t* dirty;
  double* kept;
  unsigned long long* dense;
  double* dval;
  int32_t* dstage;
  int2* fe;
  int64_t fe_light;
  int32_t chunk;
  uint64_t limit_ns;
  double* spoiled;  // backward: CountView::spoiled
  uint32_t polls;   // a waiting worker looks at the end's marks every so many polls
};
// Arcs out of a position's live states up to which a heavy block takes its
// table in shared memory, half of the table's slots.
constexpr int32_t STRING_TABLE_ARCS = 1024;
// Pool entries a group of the string kernels reserves at a time; a capped
// pool is handed out range by range, so that the cap counts live entries.
constexpr int32_t POOL_CHUNK = 64;
int64_t string_ctl_words(int32_t Bw, int32_t groups2);
int64_t string_light_entries(int num_sms, int64_t Bw);
int32_t string_kept_values();
// The forward recursion of every string: S.flags and S.pool_top point into
// W.ctl, which is cleared first.  Fills the pool and the per-token ranges
// (Viterbi: each entry's best arc and predecessor entry, -2 where it has to
// be looked up; forward: the arcs on the next symbol and the step maxima).
int launch_string_forward(bool viterbi, const LayoutView& L, const int32_t* sym, const FrontierState& S,
                          const StringWork& W, int num_sms, cudaStream_t s);
// The backward recursion and the posteriors, after launch_string_forward
// and launch_fb_final.
int launch_string_backward(const LayoutView& L, const int32_t* sym, const FrontierState& S, const CountView& C,
                           const StringWork& W, int num_sms, cudaStream_t s);
// The best path of each string after launch_string_forward and
// launch_vit_final.
int launch_string_trace(const FrontierState& S, const int32_t* olabel_by_id, int32_t Bw, const int32_t* jfinal,
                        int32_t* paths, int32_t* olabels, cudaStream_t s);
// Bounds-checked build (compiled with FST_DEBUG): the kernels check every
// computed index into the staging buffers, the live pool, the dense
// accumulators and the arc records against its buffer's size, count the
// violations, record the first (check code, index, bound) and skip the
// access.  Reads and clears that record; FST_ERR_UNSUPPORTED in a normal
// build.
int debug_read(int64_t* violations, int32_t* code, int64_t* index, int64_t* bound);

// Zero n 64-bit words of accumulators if an error bit is set in *flag: a
// run whose pool overflowed (or that gave up at a barrier) leaves staged
// accumulators behind.
int launch_clear_if_overflow(const uint32_t* flag, unsigned long long* acc, int64_t n, int num_sms, cudaStream_t s);
// Compact accumulators: clear the backward values of position y_t (after
// the pass's last step, which reads those of position 1).
int launch_bwd_clear(const FrontierState& S, int32_t pos, int num_sms, cudaStream_t s);

}  // namespace fstgpu
