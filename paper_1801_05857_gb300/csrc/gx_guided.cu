// Learned guidance for deadlock search (no counterpart in the paper; the
// search it reorders is the exploration of Sec. 3 with on-the-fly deadlock
// detection, and every state still goes through the find-or-put of Sec. 4.1).
//
// Training examples (gx_training_set): after a gx_explore, every state in the
// table gets its distance to the nearest deadlock by level-by-level
// relaxation -- distance 0 for states without successors, distance r for a
// state with a successor at distance r - 1 -- looking successors up in the
// same table.  Then each state becomes one example: the histogram of its
// processes' local states and the capped, normalised distance, and the
// examples are sorted by content so that the set comes out the same way on
// every run.
//
// Guided search (gx_find_deadlocks, GX_DL_GUIDED): open states live in
// priority bins (stacks) by score.  Each iteration:
//   * one CTA pops up to guided_batch states from the best non-empty bin;
//   * a persistent kernel expands them: it logs each (state, parent log
//     index), detects deadlocks, find-or-puts every successor and appends
//     each new one, with its local-state histogram, to a pending buffer;
//   * the scoring kernel runs the MLP on the pending states, 128 per tile, on
//     the tensor cores (tcgen05, BF16 operands, FP32 accumulation in TMEM;
//     gx_tc.cuh) and pushes each state to the bin of its score.
// Every state is pushed once and popped once, so the search ends either at a
// deadlock or after the whole state space.

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "gx_kernels.cuh"
#include "gx_tc.cuh"

namespace gx {

struct GuidedCtl {
  unsigned long long found;      // smallest log index of a deadlock found, ~0 if none
  unsigned long long batch_n;    // states popped for the current iteration
  unsigned long long log_base;   // log index of the first popped state
  unsigned long long log_count;  // states logged (expanded) so far
  unsigned long long inserted;   // states inserted into the table
  unsigned long long transitions;
  unsigned long long probes;
  unsigned int error, done;
  unsigned long long dl_count;
  unsigned long long pending;    // new states appended by the current iteration's expansion
  unsigned long long iters;      // iterations run
  unsigned long long path_len;   // states on the deadlock's path (gx_guided_trace), 0 if none
};

struct GuidedArgs {
  const uint32_t* blob;
  NetBlobLayout lay;
  uint32_t blob_words;
  int stage;
  Muls muls;
  int rounds, log2nb;
  uint32_t* table;
  GuidedCtl* ctl;
  unsigned long long* bin_count;  // [nbins]
  uint32_t* bins;                 // [nbins][bin_cap] entries of E words
  uint64_t bin_cap;
  int nbins;
  float scale;
  uint32_t* batch;                // [batch_cap] entries
  uint32_t batch_cap;
  uint32_t* log;                  // [log_cap] entries
  uint64_t log_cap;
  const float* params;            // MLP, FP32
  gxt::TcWeights* tcw;            // params packed for the scorer, once per search
  uint4* pend_hist;               // [pend_cap] local-state histograms of new states
  uint32_t* pend;                 // [pend_cap] entries of E words (vector, parent)
  uint64_t pend_cap;
  uint32_t init_vec[4];
  cudaGraphConditionalHandle cond;  // device-driven iteration loop
  unsigned long long max_iters;
};

constexpr unsigned int ERR_BINS = 16u, ERR_LOG = 32u, ERR_WIDE = 64u, ERR_PENDING = 128u;

}  // namespace gx

namespace gxd {

using gx::GuidedArgs;
using gx::GuidedCtl;


// Slot index of v in the table, or -1 when v is not stored.  Slots of a
// bucket fill in order and are never freed, so an empty slot ends the search.
template <int W, int B>
__device__ __forceinline__ int64_t find_slot(const uint32_t* __restrict__ table, int log2nb, int rounds,
                                             const uint64_t* __restrict__ muls, const uint32_t (&v)[W]) {
  constexpr int S = B / W;
  const uint64_t h = state_hash<W>(v);
  for (int k = 0; k < rounds; ++k) {
    const uint64_t b = seq_bucket<B>(h, k, muls, log2nb);
    uint32_t s[B];
    load_words<B>(table + b * (uint64_t)B, s);
#pragma unroll
    for (int j = 0; j < S; ++j) {
      bool eq = true, empty = true;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        eq &= s[j * W + w] == v[w];
        empty &= s[j * W + w] == 0u;
      }
      if (eq) return (int64_t)(b * S + j);
      if (empty) return -1;
    }
  }
  return -1;
}

// Histogram of local-state indices (each < 16, else *bad is set), 4 per word.
template <int W>
__device__ __forceinline__ void local_hist(const uint32_t* t, const NetBlobLayout& L, const uint32_t (&v)[W],
                                           uint32_t (&hw)[4], uint32_t& bad) {
  hw[0] = hw[1] = hw[2] = hw[3] = 0;
  for (uint32_t p = 0; p < L.n_procs; ++p) {
    const uint32_t s = local_state<W>(t, L, v, p);
    if (s >= 16) {
      bad = 1;
      continue;
    }
    const uint32_t inc = 1u << ((s & 3) * 8);
    if ((s >> 2) == 0) hw[0] += inc;
    else if ((s >> 2) == 1) hw[1] += inc;
    else if ((s >> 2) == 2) hw[2] += inc;
    else hw[3] += inc;
  }
}

constexpr uint32_t INF = 0xFFFFFFFFu;

// Labelling works on a list of the states found: state i's slot, its distance
// d[i], and where its successors' list indexes start in `adj` (when they are
// kept); `index` gives the list index of a slot.
struct LabelCtl {
  unsigned long long states;   // states found in the table
  unsigned long long edges;    // their successors
  unsigned long long left[4];  // ring: states without a label after round r, at r & 3
  unsigned long long bad;      // a local state index of 16 or more
};

struct LabelArgs {
  const uint32_t* table;
  const uint32_t* blob;
  NetBlobLayout lay;
  uint32_t staged_words;  // network tables the kernels copy to shared memory (0: none)
  gx::Muls muls;
  int rounds, log2nb;
  uint64_t slots;
  uint64_t cap;           // states the last search stored: the lists' size
  uint64_t adj_cap;       // successors there is room for in adj (0: not kept)
  uint32_t* index;        // [slots] (without lists: a slot's distance)
  unsigned long long* slot_of;  // [cap]
  uint32_t* d;            // [cap]
  uint32_t* first;        // [cap] where a state's successors start in adj
  uint32_t* last;         // [cap] and end
  uint32_t* adj;          // [adj_cap]
  uint32_t* todo[2];      // [cap] states without a label, before and after a round
  LabelCtl* ctl;
};

// Lists the states in the table; states without successors are at distance 0,
// the others wait for the first round.  Bound by the table's bytes: a warp reads
// 1 KB at a time, collects the occupied slots in shared memory and lists 32 at a
// time with one atomic per counter (8-process network, 72,000 states in 64 MiB: 42
// us; a lane per slot took 102 us here and another 64 us to gather the examples
// from the whole table again).
template <int W>
__global__ void __launch_bounds__(gx::kBlock) label_collect_kernel(const LabelArgs a) {
  constexpr int kWarps = gx::kBlock / 32, S = 8 / W;
  __shared__ unsigned long long queue_mem[kWarps][64];
  unsigned long long* queue = queue_mem[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  uint32_t n = 0;  // queued (uniform in the warp)
  auto list = [&](uint32_t k) {  // the last k <= 32 queued
    __syncwarp();
    n -= k;
    const bool has = lane < k;
    const unsigned long long slot = has ? queue[n + lane] : 0ull;
    uint32_t v[W];
    load_vec<W>(a.table + slot * W, v);
    const uint32_t cnt = has ? count_succ<W>(a.blob, a.lay, v) : 0u;
    unsigned long long upto = cnt;  // successors of this state and the ones before it
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(FULLMASK, upto, o);
      if ((int)lane >= o) upto += y;
    }
    const uint32_t open = __ballot_sync(FULLMASK, cnt != 0);
    unsigned long long at = 0;  // lane 0: states, 1: todo, 31: edges
    if (lane == 0) at = atomicAdd(&a.ctl->states, (unsigned long long)k);
    if (lane == 1 && open) at = atomicAdd(&a.ctl->left[0], (unsigned long long)__popc(open));
    if (lane == 31 && open) at = atomicAdd(&a.ctl->edges, upto);
    const unsigned long long i = __shfl_sync(FULLMASK, at, 0) + lane;
    const unsigned long long t = __shfl_sync(FULLMASK, at, 1) + __popc(open & below);
    const unsigned long long e = __shfl_sync(FULLMASK, at, 31) + upto - cnt;
    // (more states than the last search stored: the host reports it, no list is used)
    if (has && i < a.cap) {
      a.index[slot] = (uint32_t)i;
      a.slot_of[i] = slot;
      a.d[i] = cnt ? INF : 0u;
      a.first[i] = (uint32_t)e;
      a.last[i] = (uint32_t)(e + cnt);
      if (cnt && t < a.cap) a.todo[0][t] = (uint32_t)i;
    }
    __syncwarp();
  };
  // pieces of 8 words (a table has at least two buckets of four)
  const uint64_t pieces = a.slots * W / 8, stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < pieces; i0 += stride) {
    uint32_t s[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) s[w] = 0;
    if (i0 + lane < pieces) load_words<8>(a.table + (i0 + lane) * 8, s);
#pragma unroll
    for (int i = 0; i < S; ++i) {
      bool tagged = true;
#pragma unroll
      for (int w = 0; w < W; ++w) tagged &= (s[i * W + w] & kTag) != 0;
      const uint32_t m = __ballot_sync(FULLMASK, tagged);
      if (tagged) queue[n + __popc(m & below)] = (i0 + lane) * S + i;
      n += __popc(m);
      if (n >= 32) list(32);
    }
  }
  if (n > 0) list(n);
}

// The lists hold what the last search stored, and (keep) its successors fit.
__device__ __forceinline__ bool label_lists_ok(const LabelArgs& a, bool keep) {
  return a.ctl->states <= a.cap && (!keep || a.ctl->edges <= a.adj_cap);
}

__device__ __forceinline__ const uint32_t* label_tables(const LabelArgs& a, uint64_t* muls, uint32_t* s_tab) {
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  for (uint32_t i = threadIdx.x; i < a.staged_words; i += blockDim.x) s_tab[i] = a.blob[i];
  __syncthreads();
  return a.staged_words ? s_tab : a.blob;
}

// The successors' list indexes of every state, looked up once: a lane per state.
template <int W, int B>
__global__ void __launch_bounds__(gx::kBlock) label_adj_kernel(const LabelArgs a) {
  extern __shared__ __align__(16) uint32_t s_tab[];
  __shared__ uint64_t muls[kMaxRounds];
  if (!label_lists_ok(a, true)) return;
  const uint32_t* t = label_tables(a, muls, s_tab);
  const uint64_t n = a.ctl->states, stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    uint32_t v[W];
    load_vec<W>(a.table + a.slot_of[i] * W, v);
    const uint32_t cnt = count_succ<W>(t, a.lay, v);
    uint32_t* out = a.adj + a.first[i];
    SuccIter it;
    it.init();
    for (uint32_t k = 0; k < cnt; ++k) {
      uint32_t s[W];
      next_succ<W>(it, t, a.lay, v, s);
      const int64_t j = find_slot<W, B>(a.table, a.log2nb, a.rounds, muls, s);
      out[k] = j >= 0 ? a.index[j] : (uint32_t)i;  // (not stored: itself, which never is a label nearer)
    }
  }
}

// The ring of counters of round r; true when the round has nothing to do,
// because nothing is left or the round before labelled nothing.  (This round adds
// to left[r & 3] and reads the two before it.)
__device__ __forceinline__ bool label_round_over(const LabelArgs& a, uint32_t r, unsigned long long n) {
  const bool over = n == 0 || (r >= 2 && n == a.ctl->left[(r - 2) & 3]);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.ctl->left[(r + 1) & 3] = 0;
    if (over) a.ctl->left[r & 3] = n;
  }
  return over;
}

// Round r: the states still without a label that have a successor at distance r -
// 1 get distance r, the others are listed for the next round.  Rounds are
// launched one behind the other.  Here with the successors kept: 8 lanes a state,
// no table lookup (72,000 states, 12.8 successors each: 7-12 us a round; with a
// chain of table lookups per state 34 us; a pass over the whole table 219 us).
constexpr int kLabelLanes = 8;
__global__ void __launch_bounds__(gx::kBlock) label_round_kernel(const LabelArgs a, uint32_t r) {
  constexpr uint32_t kStates = gx::kBlock / kLabelLanes;  // a CTA takes at a time
  __shared__ uint32_t s_open[kStates];
  __shared__ unsigned long long s_base;
  const unsigned long long n = a.ctl->left[(r - 1) & 3];
  if (!label_lists_ok(a, true) || label_round_over(a, r, n)) return;
  const uint32_t lane = threadIdx.x & 31, sub = lane & (kLabelLanes - 1);
  const uint32_t group = ((1u << kLabelLanes) - 1u) << (lane & ~(kLabelLanes - 1u));
  static_assert(kStates == 32, "the first warp lists a CTA's states");
  for (unsigned long long i0 = (unsigned long long)blockIdx.x * kStates; i0 < n;
       i0 += (unsigned long long)gridDim.x * kStates) {
    const unsigned long long i = i0 + threadIdx.x / kLabelLanes;
    bool open = i < n;
    uint32_t idx = 0, e = 0, end = 0;
    if (open) {
      idx = a.todo[(r - 1) & 1][i];
      e = a.first[idx] + sub;
      end = a.last[idx];
    }
    for (; __any_sync(FULLMASK, open && e - sub < end); e += kLabelLanes) {
      const bool hit = open && e < end && a.d[a.adj[e]] == r - 1;
      if (__ballot_sync(FULLMASK, hit) & group) {
        if (open && sub == 0) a.d[idx] = r;
        open = false;
      }
    }
    // one atomic per CTA: one per warp would queue on the counter's address
    if (sub == 0) s_open[threadIdx.x / kLabelLanes] = open ? idx : INF;
    __syncthreads();
    if (threadIdx.x < 32) {
      const uint32_t mine = s_open[lane], m = __ballot_sync(FULLMASK, mine != INF);
      if (lane == 0 && m) s_base = atomicAdd(&a.ctl->left[r & 3], (unsigned long long)__popc(m));
      __syncwarp();
      if (mine != INF) a.todo[r & 1][s_base + __popc(m & ((1u << lane) - 1u))] = mine;
    }
    __syncthreads();
  }
}

// Round r without the successors kept (too many, or a search that was stopped
// early): a lane per state looks them up until one is at distance r - 1.
template <int W, int B>
__global__ void __launch_bounds__(gx::kBlock) label_lookup_round_kernel(const LabelArgs a, uint32_t r) {
  extern __shared__ __align__(16) uint32_t s_tab[];
  __shared__ uint64_t muls[kMaxRounds];
  const unsigned long long n = a.ctl->left[(r - 1) & 3];
  if (!label_lists_ok(a, false) || label_round_over(a, r, n)) return;
  if ((unsigned long long)blockIdx.x * blockDim.x >= n) return;
  const uint32_t* t = label_tables(a, muls, s_tab);
  const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < n;
       i0 += stride) {
    bool open = i0 + lane < n;
    uint32_t idx = 0;
    if (open) {
      idx = a.todo[(r - 1) & 1][i0 + lane];
      uint32_t v[W];
      load_vec<W>(a.table + a.slot_of[idx] * W, v);
      const uint32_t cnt = count_succ<W>(t, a.lay, v);
      SuccIter it;
      it.init();
      for (uint32_t k = 0; k < cnt && open; ++k) {
        uint32_t s[W];
        next_succ<W>(it, t, a.lay, v, s);
        const int64_t j = find_slot<W, B>(a.table, a.log2nb, a.rounds, muls, s);
        if (j >= 0 && a.d[a.index[j]] == r - 1) {
          a.d[idx] = r;
          open = false;
        }
      }
    }
    const uint32_t m = __ballot_sync(FULLMASK, open);
    unsigned long long base = 0;
    if (lane == 0 && m) base = atomicAdd(&a.ctl->left[r & 3], (unsigned long long)__popc(m));
    base = __shfl_sync(FULLMASK, base, 0);
    if (open) a.todo[r & 1][base + __popc(m & below)] = idx;
  }
}

// Histogram i of the caller's array, whose address need not be a multiple of 16.
__device__ __forceinline__ uint4 hist_load(const uint8_t* hist, uint64_t i) {
  if ((reinterpret_cast<uintptr_t>(hist) & 15) == 0) return reinterpret_cast<const uint4*>(hist)[i];
  uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < 16; ++k) w[k >> 2] |= (uint32_t)hist[i * 16 + k] << ((k & 3) * 8);
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ void hist_store(uint8_t* hist, uint64_t i, const uint4& q) {
  if ((reinterpret_cast<uintptr_t>(hist) & 15) == 0) {
    reinterpret_cast<uint4*>(hist)[i] = q;
    return;
  }
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int k = 0; k < 16; ++k) hist[i * 16 + k] = (uint8_t)(w[k >> 2] >> ((k & 3) * 8));
}

// Example i: the histogram and the label of state i of the list.
template <int W>
__global__ void __launch_bounds__(gx::kBlock) label_gather_kernel(const LabelArgs a, uint32_t max_dist,
                                                                  uint8_t* hist_out, float* label_out, uint64_t cap) {
  if (!label_lists_ok(a, false)) return;
  const uint64_t n = a.ctl->states, stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    uint32_t v[W], hw[4], bad = 0;
    load_vec<W>(a.table + a.slot_of[i] * W, v);
    local_hist<W>(a.blob, a.lay, v, hw, bad);
    if (bad) atomicOr(&a.ctl->bad, 1ull);
    if (i >= cap) continue;
    hist_store(hist_out, i, make_uint4(hw[0], hw[1], hw[2], hw[3]));
    const uint32_t d = a.d[i] == INF ? max_dist : min(a.d[i], max_dist);
    label_out[i] = (float)d / (float)max_dist;
  }
}

// ---- labelling without lists, in the caller's scratch alone (dist: a distance per
// slot): for tables of 2^32 or more states, for lack of memory, and for a table that
// is not the one the last search left.  Every round passes over the whole table.

template <int W>
__device__ __forceinline__ bool slot_vec(const uint32_t* table, uint64_t i, uint32_t (&v)[W]) {
  load_vec<W>(table + i * W, v);
  bool tagged = true;
#pragma unroll
  for (int w = 0; w < W; ++w) tagged &= (v[w] & kTag) != 0;
  return tagged;
}

template <int W>
__global__ void __launch_bounds__(gx::kBlock) slot_init_kernel(const LabelArgs a) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.slots; i += stride) {
    uint32_t v[W];
    a.index[i] = slot_vec<W>(a.table, i, v) && count_succ<W>(a.blob, a.lay, v) == 0 ? 0u : INF;
  }
}

// Round r: sets *changed when a slot was labelled.
template <int W, int B>
__global__ void __launch_bounds__(gx::kBlock) slot_round_kernel(const LabelArgs a, uint32_t r,
                                                                unsigned long long* changed) {
  extern __shared__ __align__(16) uint32_t s_tab[];
  __shared__ uint64_t muls[kMaxRounds];
  const uint32_t* t = label_tables(a, muls, s_tab);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  bool any = false;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.slots; i += stride) {
    uint32_t v[W];
    if (a.index[i] != INF || !slot_vec<W>(a.table, i, v)) continue;
    const uint32_t cnt = count_succ<W>(t, a.lay, v);
    SuccIter it;
    it.init();
    for (uint32_t k = 0; k < cnt; ++k) {
      uint32_t s[W];
      next_succ<W>(it, t, a.lay, v, s);
      const int64_t j = find_slot<W, B>(a.table, a.log2nb, a.rounds, muls, s);
      if (j >= 0 && a.index[j] == r - 1) {
        a.index[i] = r;
        any = true;
        break;
      }
    }
  }
  if (any) *changed = 1;
}

// Examples of the occupied slots, at positions counted in out[0]; out[1]: a local state
// index of 16 or more.
template <int W>
__global__ void __launch_bounds__(gx::kBlock) slot_gather_kernel(const LabelArgs a, uint32_t max_dist,
                                                                 uint8_t* hist_out, float* label_out, uint64_t cap,
                                                                 unsigned long long* out) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < a.slots; i0 += stride) {
    uint32_t v[W], hw[4], bad = 0;
    const uint64_t i = i0 + lane;
    const bool has = i < a.slots && slot_vec<W>(a.table, i, v);
    const uint32_t m = __ballot_sync(FULLMASK, has);
    unsigned long long base = 0;
    if (lane == 0 && m) base = atomicAdd(out, (unsigned long long)__popc(m));
    const unsigned long long pos = __shfl_sync(FULLMASK, base, 0) + __popc(m & ((1u << lane) - 1u));
    if (!has) continue;
    local_hist<W>(a.blob, a.lay, v, hw, bad);
    if (bad) out[1] = 1;
    if (pos >= cap) continue;
    hist_store(hist_out, pos, make_uint4(hw[0], hw[1], hw[2], hw[3]));
    const uint32_t d = min(a.index[i], max_dist);  // (INF: max_dist)
    label_out[pos] = (float)d / (float)max_dist;
  }
}

// Content order of the training examples: the states are listed at atomic
// positions, so the examples are sorted by their own content (the 16
// histogram bytes, then the label's bits, compared as unsigned words) to make
// the training set -- and everything trained from it -- the same on every run.
// Equal keys are identical examples, so an unstable sort is enough: a bitonic
// sort over a power-of-two buffer padded with all-ones keys (no histogram byte
// reaches 0xFF).  Passes over distances below a tile of 2^kTileLog2 examples run
// in shared memory, all that follow one another in one launch; the others take
// two distances at a time, four examples per thread.  2^17 examples: 20
// launches instead of 153.
__device__ __forceinline__ bool ex_greater(const uint4& a, uint32_t la, const uint4& b, uint32_t lb) {
  if (a.x != b.x) return a.x > b.x;
  if (a.y != b.y) return a.y > b.y;
  if (a.z != b.z) return a.z > b.z;
  if (a.w != b.w) return a.w > b.w;
  return la > lb;
}

__device__ __forceinline__ void ex_order(uint4& a, uint32_t& la, uint4& b, uint32_t& lb, bool up) {
  if (up != ex_greater(a, la, b, lb)) return;
  const uint4 q = a;
  const uint32_t l = la;
  a = b;
  la = lb;
  b = q;
  lb = l;
}

// Examples at distances 2q and q: four of them a, a + q, a + 2q, a + 3q.
__device__ __forceinline__ void ex_order4(uint4 (&x)[4], uint32_t (&l)[4], bool up) {
  ex_order(x[0], l[0], x[2], l[2], up);
  ex_order(x[1], l[1], x[3], l[3], up);
  ex_order(x[0], l[0], x[1], l[1], up);
  ex_order(x[2], l[2], x[3], l[3], up);
}

constexpr int kTileLog2 = 11;
constexpr int kTile = 1 << kTileLog2;
constexpr int kTileThreads = 512;
constexpr size_t kTileBytes = 20 * kTile;

// The passes of stages k0..k1 (powers of two) at distances below the tile, on one
// tile per CTA.  `load`: the examples come from hist and label (n of them, padded).
__global__ void __launch_bounds__(kTileThreads) ex_tile_kernel(uint4* h, uint32_t* l, uint64_t n2, uint64_t k0,
                                                               uint64_t k1, int load, const uint8_t* hist,
                                                               const float* label, uint64_t n) {
  extern __shared__ __align__(16) unsigned char tile_mem[];
  uint4* sh = reinterpret_cast<uint4*>(tile_mem);
  uint32_t* sl = reinterpret_cast<uint32_t*>(sh + kTile);
  const uint64_t base = (uint64_t)blockIdx.x * kTile;
  const int tile = n2 < (uint64_t)kTile ? (int)n2 : kTile;
  for (int i = threadIdx.x; i < tile; i += kTileThreads) {
    if (!load) {
      sh[i] = h[base + i];
      sl[i] = l[base + i];
    } else if (base + i < n) {
      sh[i] = hist_load(hist, base + i);
      sl[i] = __float_as_uint(label[base + i]);
    } else {
      sh[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
      sl[i] = ~0u;
    }
  }
  __syncthreads();
  // two distances at a time, four examples per thread in registers
  for (uint64_t k = k0; k <= k1; k <<= 1) {
    int j = k / 2 < (uint64_t)tile / 2 ? (int)(k / 2) : tile / 2;
    while (j > 0) {
      if (j >= 2) {
        const int q = j / 2;
        for (int p = threadIdx.x; p < tile / 4; p += kTileThreads) {
          const int a = ((p & ~(q - 1)) << 2) | (p & (q - 1));
          const bool up = ((base + a) & k) == 0;
          uint4 x[4];
          uint32_t lx[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            x[i] = sh[a + i * q];
            lx[i] = sl[a + i * q];
          }
          ex_order4(x, lx, up);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            sh[a + i * q] = x[i];
            sl[a + i * q] = lx[i];
          }
        }
        j >>= 2;
      } else {
        for (int p = threadIdx.x; p < tile / 2; p += kTileThreads) {
          const int a = p << 1;
          ex_order(sh[a], sl[a], sh[a + 1], sl[a + 1], ((base + a) & k) == 0);
        }
        j = 0;
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < tile; i += kTileThreads) {
    h[base + i] = sh[i];
    l[base + i] = sl[i];
  }
}

// Stage k at distances j and, when `two`, j / 2 (both at least a tile).
__global__ void __launch_bounds__(256) ex_wide_kernel(uint4* h, uint32_t* l, uint64_t n2, uint64_t k, uint64_t j,
                                                      int two) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, q = two ? j / 2 : j;
  for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n2 / (two ? 4 : 2); p += stride) {
    const uint64_t a = two ? ((p & ~(q - 1)) << 2) | (p & (q - 1)) : ((p & ~(j - 1)) << 1) | (p & (j - 1));
    const bool up = (a & k) == 0;
    if (!two) {
      uint4 x = h[a], y = h[a + j];
      uint32_t lx = l[a], ly = l[a + j];
      ex_order(x, lx, y, ly, up);
      h[a] = x;
      h[a + j] = y;
      l[a] = lx;
      l[a + j] = ly;
    } else {
      uint4 x[4];
      uint32_t lx[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x[i] = h[a + i * q];
        lx[i] = l[a + i * q];
      }
      ex_order4(x, lx, up);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        h[a + i * q] = x[i];
        l[a + i * q] = lx[i];
      }
    }
  }
}

__global__ void ex_store_kernel(const uint4* h, const uint32_t* l, uint64_t n, uint8_t* hist, float* label) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    hist_store(hist, i, h[i]);
    label[i] = __uint_as_float(l[i]);
  }
}

// ---- guided search

template <int W>
__device__ __forceinline__ void push_bin(const GuidedArgs& a, float score, const uint32_t (&v)[W], uint32_t parent,
                                         uint32_t& err) {
  constexpr int E = W + 1;
  int b0 = (int)(score / a.scale * (float)a.nbins);
  b0 = b0 < 0 ? 0 : (b0 >= a.nbins ? a.nbins - 1 : b0);
  // The calling lanes that share a bin reserve their slots with one atomic
  // (scores cluster, and same-address atomics serialise in L2).
  {
    const uint32_t peers = __match_any_sync(__activemask(), b0);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(&a.bin_count[b0], (unsigned long long)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    const unsigned long long pos = base + __popc(peers & ((1u << lane) - 1u));
    if (pos < a.bin_cap) {
      uint32_t* e = a.bins + ((uint64_t)b0 * a.bin_cap + pos) * E;
#pragma unroll
      for (int w = 0; w < W; ++w) e[w] = v[w];
      e[W] = parent;
      return;
    }
  }
  // a full bin spills into the next one (cyclically): the bins together hold
  // as many entries as the table has slots, so some bin always has room
  for (int i = 1; i < a.nbins; ++i) {
    const int b = (b0 + i) % a.nbins;
    const unsigned long long pos = atomicAdd(&a.bin_count[b], 1ull);
    if (pos < a.bin_cap) {
      uint32_t* e = a.bins + ((uint64_t)b * a.bin_cap + pos) * E;
#pragma unroll
      for (int w = 0; w < W; ++w) e[w] = v[w];
      e[W] = parent;
      return;
    }
  }
  err |= gx::ERR_BINS;
}

// The initial state: into the table and the first bin (as the only open
// state its score does not matter).
template <int W, int B>
__global__ void __launch_bounds__(32) guided_init_kernel(const GuidedArgs a) {
  __shared__ uint64_t muls[kMaxRounds];
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  __syncwarp();
  if (threadIdx.x != 0) return;
  uint32_t v[W];
#pragma unroll
  for (int w = 0; w < W; ++w) v[w] = a.init_vec[w];
  uint32_t hw[4], bad = 0;
  local_hist<W>(a.blob, a.lay, v, hw, bad);
  uint32_t probes = 0, err = bad ? gx::ERR_WIDE : 0u;
  const int r = find_or_put_state<W, B>(a.table, a.log2nb, a.rounds, muls, v, probes);
  if (r != FOP_INSERTED) err |= gx::ERR_TABLE_FULL;
  else {
    a.ctl->inserted = 1;
    push_bin<W>(a, 0.f, v, 0xFFFFFFFFu, err);
  }
  if (err) atomicOr(&a.ctl->error, err);
}

// Pop the next batch from the best non-empty bin (one CTA of up to 1024
// threads, all calling).  The bins are scanned in parallel, one counter per
// thread.  Returns (in every thread) whether a batch was taken; sets done
// when every bin is empty.
template <int W>
__device__ __forceinline__ bool select_batch(const GuidedArgs& a) {
  constexpr int E = W + 1;
  __shared__ int best;
  __shared__ unsigned long long take, top;
  GuidedCtl& c = *a.ctl;
  const bool go = c.found == ~0ull && !c.error;  // uniform: read before anyone writes
  __syncthreads();
  if (threadIdx.x == 0) {
    best = 0x7FFFFFFF;
    c.batch_n = 0;
    c.pending = 0;
  }
  __syncthreads();
  if (!go) return false;
  for (int b = threadIdx.x; b < a.nbins; b += blockDim.x) {
    unsigned long long cnt = a.bin_count[b];
    if (cnt > a.bin_cap) {  // failed pushes left the counter past the end
      cnt = a.bin_cap;
      a.bin_count[b] = cnt;
    }
    if (cnt > 0) atomicMin(&best, b);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (best == 0x7FFFFFFF) {
      c.done = 1;
      best = -1;
    } else {
      const unsigned long long cnt = a.bin_count[best];
      take = cnt < a.batch_cap ? cnt : a.batch_cap;
      top = cnt - take;
      if (c.log_count + take > a.log_cap) {
        c.error |= gx::ERR_LOG;
        best = -1;
      } else {
        a.bin_count[best] = top;
        c.batch_n = take;
        c.log_base = c.log_count;
        c.log_count += take;
      }
    }
  }
  __syncthreads();
  if (best < 0) return false;
  const uint32_t* src = a.bins + ((uint64_t)best * a.bin_cap + top) * E;
  for (uint64_t i = threadIdx.x; i < take * E; i += blockDim.x) a.batch[i] = src[i];
  return true;
}

// One CTA: pop the next batch (the host-driven loop).
template <int W>
__global__ void __launch_bounds__(1024) guided_select_kernel(const GuidedArgs a) {
  select_batch<W>(a);
}

template <int W, int B, bool Share>
__global__ void __launch_bounds__(gx::kBlock) guided_expand_kernel(const GuidedArgs a) {
  constexpr int E = W + 1;
  constexpr int kWarps = gx::kBlock / 32;
  const unsigned long long n = a.ctl->batch_n;
  if ((unsigned long long)blockIdx.x * kWarps >= n) return;  // no state for this CTA
  extern __shared__ __align__(16) uint32_t gsm[];
  __shared__ uint64_t muls[kMaxRounds];
  __shared__ unsigned long long s_sum[3][kWarps];
  __shared__ uint32_t s_err[kWarps];
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  const uint32_t* t = a.blob;
  if (a.stage) {
    uint32_t* s_tab = gsm;
    for (uint32_t i = threadIdx.x; i < a.blob_words; i += blockDim.x) s_tab[i] = a.blob[i];
    t = s_tab;
  }
  __syncthreads();
  const NetBlobLayout& L = a.lay;
  __shared__ uint4 descs[kMaxProcs];
  __shared__ __align__(16) uint32_t queue_mem[kWarps][64 * W];
  __shared__ uint32_t rows_mem[kWarps][64 * E], s_left[kWarps];
  __shared__ unsigned long long s_base;
  const ProcDescs desc = stage_descs(t, L, descs);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned long long log_base = a.ctl->log_base;
  unsigned long long trans = 0, ins = 0;
  uint32_t probes = 0, err = 0;
  // One warp per state: a batch holds a few thousand states, so the time of an
  // iteration is the latency of one state's successors.  The lanes take the
  // state's sources of successors 32 at a time (WarpGen), queue the successors and
  // find-or-put 32 of them at once.  Warp w of the grid takes states w, w + (warps
  // of the grid), ...
  const unsigned long long nwarps = (unsigned long long)gridDim.x * kWarps;
  const uint32_t n_src = L.n_procs + L.n_rules, below = (1u << lane) - 1u;
  uint32_t* queue = queue_mem[threadIdx.x >> 5];
  uint32_t* rows = rows_mem[threadIdx.x >> 5];
  int staged = 0;  // new states (uniform in the warp)
  // the last m <= 32 staged states, with their histograms, to positions base.. of the pending buffer
  auto append = [&](int m, unsigned long long base) {
    staged -= m;
    if (lane < m) {
      ins += 1;
      const uint32_t* r = rows + (staged + lane) * E;
      uint32_t s[W], hw[4], bad = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) s[w] = r[w];
      local_hist<W>(t, L, s, hw, bad);
      if (bad) err |= gx::ERR_WIDE;
      const unsigned long long pos = base + lane;
      if (pos < a.pend_cap) {
        a.pend_hist[pos] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        uint32_t* e = a.pend + pos * E;
#pragma unroll
        for (int w = 0; w < E; ++w) e[w] = r[w];
      } else {
        err |= gx::ERR_PENDING;
      }
    }
    __syncwarp();
  };
  for (unsigned long long idx = (unsigned long long)blockIdx.x * kWarps + (threadIdx.x >> 5); idx < n;
       idx += nwarps) {
    uint32_t v[W];
#pragma unroll
    for (int w = 0; w < W; ++w) v[w] = a.batch[idx * E + w];
    const unsigned long long li = log_base + idx;
    if (lane == 0) {
      uint32_t* le = a.log + li * E;
#pragma unroll
      for (int w = 0; w < W; ++w) le[w] = v[w];
      le[W] = a.batch[idx * E + W];
    }
    WarpGen<W, Share> gen;
    gen.src = gen.e = gen.e_end = gen.word = gen.cur = 0;
    uint32_t total = 0;  // this lane's part of the state's successors
    int queued = 0;
    while (true) {
      uint32_t act = __ballot_sync(FULLMASK, gen.e < gen.e_end);
      if (act != 0) {
        if constexpr (Share) {
          if (__popc(act) <= 16) {
            gen.share(act, 5);
            act = __ballot_sync(FULLMASK, gen.e < gen.e_end);
          }
        }
        if ((act >> lane) & 1u) gen.emit(t, L, desc, v, queue + (queued + __popc(act & below)) * W);
        queued += __popc(act);
        if (queued < 32) continue;
      } else if (gen.src < n_src) {
        gen.open_wide(t, L, desc, true, v, 5);
        total += gen.e_end - gen.e;
        continue;
      }
      if (queued == 0) break;
      __syncwarp();
      const int k = queued < 32 ? queued : 32;
      queued -= k;
      uint32_t s[W];
      bool inserted = false;
      if (lane < k) {
        load_vec<W>(queue + (queued + lane) * W, s);
        const int r = find_or_put_state<W, B>(a.table, a.log2nb, a.rounds, muls, s, probes);
        if (r == FOP_FULL) err |= gx::ERR_TABLE_FULL;
        inserted = r == FOP_INSERTED;
      }
      // stage the new states; 32 of them are appended to the pending buffer at a time
      const uint32_t im = __ballot_sync(FULLMASK, inserted);
      if (inserted) {
        uint32_t* e = rows + (staged + __popc(im & below)) * E;
#pragma unroll
        for (int w = 0; w < W; ++w) e[w] = s[w];
        e[W] = (uint32_t)li;
      }
      staged += __popc(im);
      __syncwarp();
      if (staged >= 32) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&a.ctl->pending, 32ull);
        append(32, __shfl_sync(FULLMASK, base, 0));
      }
    }
    total = __reduce_add_sync(FULLMASK, total);
    if (lane == 0) {
      trans += total;
      if (total == 0) {
        atomicMin(&a.ctl->found, li);
        atomicAdd(&a.ctl->dl_count, 1ull);
      }
    }
  }
  // what the CTA's warps have staged, with one atomic for all of them: most warps
  // expand one or two states, and 8192 atomics on one address would take 8 us
  const int wid = threadIdx.x >> 5;
  if (lane == 0) s_left[wid] = (uint32_t)staged;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t sum = 0;
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t m = s_left[w];
      s_left[w] = sum;
      sum += m;
    }
    s_base = sum ? atomicAdd(&a.ctl->pending, (unsigned long long)sum) : 0ull;
  }
  __syncthreads();
  if (staged > 0) append(staged, s_base + s_left[wid]);
  // the CTA's totals, one atomic per counter (every warp's at once would queue
  // on the same addresses)
  trans = warp_sum(trans);
  ins = warp_sum(ins);
  const unsigned long long pr = warp_sum((unsigned long long)probes);
  err = __reduce_or_sync(FULLMASK, err);
  if (lane == 0) {
    s_sum[0][wid] = trans;
    s_sum[1][wid] = ins;
    s_sum[2][wid] = pr;
    s_err[wid] = err;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    unsigned long long x = 0;
    for (int w = 0; w < kWarps; ++w) x += threadIdx.x < 3 ? s_sum[threadIdx.x][w] : (unsigned long long)s_err[w];
    if (x) {
      if (threadIdx.x == 0) atomicAdd(&a.ctl->transitions, x);
      else if (threadIdx.x == 1) atomicAdd(&a.ctl->inserted, x);
      else if (threadIdx.x == 2) atomicAdd(&a.ctl->probes, x);
      else {
        uint32_t e = 0;
        for (int w = 0; w < kWarps; ++w) e |= s_err[w];
        atomicOr(&a.ctl->error, e);
      }
    }
  }
}

// Score the pending states on the tensor cores and push each to its bin.
// 128 threads; persistent over tiles of 128 states.
template <int W>
__global__ void __launch_bounds__(gxt::kRows) guided_score_kernel(const GuidedArgs a) {
  constexpr int E = W + 1;
  extern __shared__ __align__(16) uint8_t tsm[];
  unsigned long long n = a.ctl->pending;
  if (n > a.pend_cap) n = a.pend_cap;  // the expansion reported the overflow
  const unsigned long long tiles = (n + gxt::kRows - 1) / gxt::kRows;
  if (blockIdx.x >= tiles) return;
  gxt::TcScorer sc = gxt::tc_setup(tsm, a.tcw);
  uint32_t err = 0;
  if (!sc.ok) {
    gxt::tc_teardown(sc);
    if (threadIdx.x == 0) atomicOr(&a.ctl->error, gx::ERR_SPIN);
    return;
  }
  for (unsigned long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const unsigned long long row = tile * gxt::kRows + threadIdx.x;
    const bool valid = row < n;
    uint32_t hw[4] = {0, 0, 0, 0};
    if (valid) {
      const uint4 q = a.pend_hist[row];
      hw[0] = q.x;
      hw[1] = q.y;
      hw[2] = q.z;
      hw[3] = q.w;
    }
    float y = 0.f;
    if (!gxt::tc_score_tile(sc, hw, y)) {
      err |= gx::ERR_SPIN;
      break;
    }
    if (valid) {
      uint32_t v[W];
      const uint32_t* e = a.pend + row * E;
#pragma unroll
      for (int w = 0; w < W; ++w) v[w] = e[w];
      push_bin<W>(a, y, v, e[W], err);
    }
  }
  gxt::tc_teardown(sc);
  if (err) atomicOr(&a.ctl->error, err);
}

// Expansion and scoring in one kernel (gx_explore_opts.guided_fused): the
// same one-warp-per-state expansion as guided_expand_kernel, but a CTA keeps
// the states its warps insert, with their histograms, in shared memory, and
// its warps 0-3 score them 128 at a time on the tensor cores (gx_tc.cuh,
// synchronising among themselves on a named barrier) and push them to their
// bins -- no pending buffer and no scoring kernel.  The warps of a CTA walk
// their states' successors in lock-step chunks of 32 (a CTA barrier after each
// chunk), so at most 127 + 16 x 32 states wait for a tile.
constexpr int kFusedWarps = 16;
constexpr int kFusedThreads = kFusedWarps * 32;
constexpr int kFusedRows = gxt::kRows - 1 + kFusedThreads;

template <int W>
__host__ __device__ constexpr size_t fused_smem_bytes(size_t blob_bytes) {
  return gxt::kTcSmemBytes + 16ull * kFusedRows + 4ull * (W + 1) * kFusedRows + blob_bytes;
}

template <int W, int B>
__global__ void __launch_bounds__(kFusedThreads, 2) guided_fused_kernel(const GuidedArgs a) {
  constexpr int E = W + 1;
  const unsigned long long n = a.ctl->batch_n;
  const unsigned long long nwarps = (unsigned long long)gridDim.x * kFusedWarps;
  if ((unsigned long long)blockIdx.x * kFusedWarps >= n) return;  // no state for this CTA
  extern __shared__ __align__(16) uint8_t fsm[];
  uint8_t* tc_area = fsm;  // the scorer's 1024-aligned part lies within its first kTcSmemBytes
  uint4* rows_h = reinterpret_cast<uint4*>(fsm + gxt::kTcSmemBytes);
  uint32_t* rows_e = reinterpret_cast<uint32_t*>(rows_h + kFusedRows);
  uint32_t* s_tab = rows_e + E * kFusedRows;
  __shared__ uint64_t muls[kMaxRounds];
  __shared__ unsigned int s_rows, s_steps, s_ok;
  __shared__ unsigned long long s_sum[3][kFusedWarps];
  __shared__ uint32_t s_err[kFusedWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int i = tid; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  const uint32_t* t = a.blob;
  if (a.stage) {
    for (uint32_t i = tid; i < a.blob_words; i += blockDim.x) s_tab[i] = a.blob[i];
    t = s_tab;
  }
  uint32_t err = 0;
  gxt::TcScorer sc{};
  if (tid < gxt::kRows) {
    sc = gxt::tc_setup(tc_area, a.tcw);
    if (tid == 0) s_ok = sc.ok ? 1u : 0u;
  }
  if (tid == 0) s_rows = 0;
  __syncthreads();
  if (!s_ok) err |= gx::ERR_SPIN;
  const NetBlobLayout& L = a.lay;
  const unsigned long long log_base = a.ctl->log_base;
  unsigned long long trans = 0, ins = 0;
  uint32_t probes = 0;

  // Score rows [0, m) (m <= 128) with the scoring threads and push them to their bins.
  auto score_rows = [&](unsigned int m) {
    if (tid < gxt::kRows && s_ok) {
      uint32_t hw[4] = {0, 0, 0, 0};
      const bool valid = (unsigned int)tid < m;
      if (valid) {
        const uint4 q = rows_h[tid];
        hw[0] = q.x;
        hw[1] = q.y;
        hw[2] = q.z;
        hw[3] = q.w;
      }
      float y = 0.f;
      if (!gxt::tc_score_tile(sc, hw, y)) {
        err |= gx::ERR_SPIN;
        if (tid == 0) s_ok = 0;
      } else if (valid) {
        uint32_t v[W];
#pragma unroll
        for (int w = 0; w < W; ++w) v[w] = rows_e[tid * E + w];
        push_bin<W>(a, y, v, rows_e[tid * E + W], err);
      }
    }
  };

  const unsigned long long first = (unsigned long long)blockIdx.x * kFusedWarps;
  const unsigned long long rounds = (n - first + nwarps - 1) / nwarps;  // the same for the whole CTA
  for (unsigned long long r = 0; r < rounds; ++r) {
    const unsigned long long idx = first + wid + r * nwarps;
    const bool has = idx < n;
    uint32_t v[W];
#pragma unroll
    for (int w = 0; w < W; ++w) v[w] = has ? a.batch[idx * E + w] : 0u;
    const unsigned long long li = log_base + idx;
    uint32_t total = 0;
    if (has) {
      if (lane == 0) {
        uint32_t* le = a.log + li * E;
#pragma unroll
        for (int w = 0; w < W; ++w) le[w] = v[w];
        le[W] = a.batch[idx * E + W];
      }
      total = count_succ<W>(t, L, v);
      if (lane == 0) {
        trans += total;
        if (total == 0) {
          atomicMin(&a.ctl->found, li);
          atomicAdd(&a.ctl->dl_count, 1ull);
        }
      }
    }
    if (tid == 0) s_steps = 0;
    __syncthreads();
    if (lane == 0 && total) atomicMax(&s_steps, (total + 31u) / 32u);
    __syncthreads();
    const uint32_t steps = s_steps;
    for (uint32_t c = 0; c < steps; ++c) {
      const uint32_t k = c * 32 + lane;
      uint32_t s[W];
      bool inserted = false;
      if (k < total) {
        seek_succ<W>(t, L, v, k, s);
        const int res = find_or_put_state<W, B>(a.table, a.log2nb, a.rounds, muls, s, probes);
        if (res == FOP_FULL) err |= gx::ERR_TABLE_FULL;
        inserted = res == FOP_INSERTED;
      }
      uint32_t hw[4] = {0, 0, 0, 0}, bad = 0;
      if (inserted) local_hist<W>(t, L, s, hw, bad);
      if (bad) err |= gx::ERR_WIDE;
      const uint32_t im = __ballot_sync(FULLMASK, inserted);
      ins += inserted ? 1u : 0u;
      if (im) {  // rows for the warp's new states, one shared-memory atomic per warp
        unsigned int base = 0;
        if (lane == 0) base = atomicAdd(&s_rows, (unsigned int)__popc(im));
        base = __shfl_sync(FULLMASK, base, 0);
        if (inserted) {
          const unsigned int row = base + __popc(im & ((1u << lane) - 1u));
          rows_h[row] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
#pragma unroll
          for (int w = 0; w < W; ++w) rows_e[row * E + w] = s[w];
          rows_e[row * E + W] = (uint32_t)li;
        }
      }
      __syncthreads();
      // full tiles: score rows [0, 128), move the rest to the front
      while (s_rows >= (unsigned int)gxt::kRows) {
        const unsigned int m = s_rows;
        score_rows(gxt::kRows);
        __syncthreads();
        const unsigned int left = m - gxt::kRows;  // < 16 x 32
        uint4 hq = make_uint4(0, 0, 0, 0);
        uint32_t eq[E];
        if ((unsigned int)tid < left) {
          hq = rows_h[gxt::kRows + tid];
#pragma unroll
          for (int w = 0; w < E; ++w) eq[w] = rows_e[(gxt::kRows + tid) * E + w];
        }
        __syncthreads();
        if ((unsigned int)tid < left) {
          rows_h[tid] = hq;
#pragma unroll
          for (int w = 0; w < E; ++w) rows_e[tid * E + w] = eq[w];
        }
        if (tid == 0) s_rows = left;
        __syncthreads();
      }
    }
  }
  if (s_rows > 0) score_rows(s_rows);  // the last, partial tile
  if (tid < gxt::kRows) gxt::tc_teardown(sc);
  // the CTA's totals, one atomic per counter
  trans = warp_sum(trans);
  ins = warp_sum(ins);
  const unsigned long long pr = warp_sum((unsigned long long)probes);
  err = __reduce_or_sync(FULLMASK, err);
  if (lane == 0) {
    s_sum[0][wid] = trans;
    s_sum[1][wid] = ins;
    s_sum[2][wid] = pr;
    s_err[wid] = err;
  }
  __syncthreads();
  if (tid < 4) {
    unsigned long long x = 0;
    for (int w = 0; w < kFusedWarps; ++w) x += tid < 3 ? s_sum[tid][w] : (unsigned long long)s_err[w];
    if (x) {
      if (tid == 0) atomicAdd(&a.ctl->transitions, x);
      else if (tid == 1) atomicAdd(&a.ctl->inserted, x);
      else if (tid == 2) atomicAdd(&a.ctl->probes, x);
      else {
        uint32_t e = 0;
        for (int w = 0; w < kFusedWarps; ++w) e |= s_err[w];
        atomicOr(&a.ctl->error, e);
      }
    }
  }
}

// ---- the device-driven iteration loop and the deadlock's path

// Control block at the start of a search (the rest was cleared).
__global__ void guided_reset_kernel(const GuidedArgs a) { a.ctl->found = ~0ull; }

// Start of the device-driven loop (one CTA of 1024 threads): pop the first
// batch; the loop runs if there is one.
template <int W>
__global__ void __launch_bounds__(1024) guided_loop_start_kernel(const GuidedArgs a) {
  const bool more = select_batch<W>(a);
  if (threadIdx.x == 0) cudaGraphSetConditional(a.cond, more ? 1u : 0u);
}

// After {expand, score}: go on unless a deadlock was found, the open set is
// empty, an error occurred or the iteration bound (every iteration expands at
// least one state, so the log size bounds it) was reached -- and if going on,
// pop the next batch here, so that an iteration takes three kernels.
template <int W>
__global__ void __launch_bounds__(1024) guided_advance_kernel(const GuidedArgs a) {
  GuidedCtl& c = *a.ctl;
  __shared__ int s_more;
  if (threadIdx.x == 0) {
    c.iters += 1;
    s_more = c.found == ~0ull && !c.done && !c.error && c.iters < a.max_iters;
  }
  __syncthreads();
  bool more = s_more != 0;
  if (more) more = select_batch<W>(a);
  if (threadIdx.x == 0) cudaGraphSetConditional(a.cond, more ? 1u : 0u);
}

// One thread: follow the parent log indices from the deadlock back to the
// initial state, writing the path (deadlock first, E words per state) to out;
// c.path_len = its length, or 0 when it does not fit in cap states.
template <int W>
__global__ void guided_path_kernel(const GuidedArgs a, uint32_t* out, uint64_t cap) {
  constexpr int E = W + 1;
  GuidedCtl& c = *a.ctl;
  c.path_len = 0;
  if (c.found == ~0ull) return;
  uint64_t li = c.found, n = 0;
  while (n < cap) {
    const uint32_t* e = a.log + li * E;
#pragma unroll
    for (int w = 0; w < E; ++w) out[n * E + w] = e[w];
    ++n;
    if (e[W] == 0xFFFFFFFFu) {
      c.path_len = n;
      return;
    }
    li = e[W];
  }
}

}  // namespace gxd

namespace gx {
namespace {

#define GG_CUDA(call)                                                                      \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess)                                                                 \
      return gx::fail(GX_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));    \
  } while (0)

inline uint64_t a256(uint64_t x) { return (x + 255) & ~255ull; }

// Temporary device memory of one call, stream-ordered; given back at the end.
struct TempMem {
  cudaStream_t st;
  unsigned char* p = nullptr;
  uint64_t bytes = 0;
  explicit TempMem(cudaStream_t s) : st(s) {}
  TempMem(const TempMem&) = delete;
  TempMem& operator=(const TempMem&) = delete;
  bool alloc(uint64_t n) {
    if (cudaMallocAsync(reinterpret_cast<void**>(&p), n, st) == cudaSuccess) {
      bytes = n;
      return true;
    }
    cudaGetLastError();
    p = nullptr;
    return false;
  }
  void release() {
    if (p) cudaFreeAsync(p, st);
    p = nullptr;
    bytes = 0;
  }
  ~TempMem() { release(); }
};

struct GKernels {
  void (*label_collect)(gxd::LabelArgs);
  void (*label_adj)(gxd::LabelArgs);
  void (*label_lookup_round)(gxd::LabelArgs, uint32_t);
  void (*label_gather)(gxd::LabelArgs, uint32_t, uint8_t*, float*, uint64_t);
  void (*slot_init)(gxd::LabelArgs);
  void (*slot_round)(gxd::LabelArgs, uint32_t, unsigned long long*);
  void (*slot_gather)(gxd::LabelArgs, uint32_t, uint8_t*, float*, uint64_t, unsigned long long*);
  const void* init;
  const void* select;
  const void* expand;
  const void* expand_share;  // for networks with a source of kShareFrom successors or more
  const void* score;
  const void* path;
  const void* start;    // pop the first batch and start the device loop
  const void* advance;  // end an iteration and pop the next batch
  const void* fused;    // expansion with the scoring in the same kernel
};

template <int W, int B>
GKernels gk() {
  return GKernels{&gxd::label_collect_kernel<W>, &gxd::label_adj_kernel<W, B>, &gxd::label_lookup_round_kernel<W, B>,
                  &gxd::label_gather_kernel<W>, &gxd::slot_init_kernel<W>, &gxd::slot_round_kernel<W, B>,
                  &gxd::slot_gather_kernel<W>,
                  reinterpret_cast<const void*>(&gxd::guided_init_kernel<W, B>),
                  reinterpret_cast<const void*>(&gxd::guided_select_kernel<W>),
                  reinterpret_cast<const void*>(&gxd::guided_expand_kernel<W, B, false>),
                  reinterpret_cast<const void*>(&gxd::guided_expand_kernel<W, B, true>),
                  reinterpret_cast<const void*>(&gxd::guided_score_kernel<W>),
                  reinterpret_cast<const void*>(&gxd::guided_path_kernel<W>),
                  reinterpret_cast<const void*>(&gxd::guided_loop_start_kernel<W>),
                  reinterpret_cast<const void*>(&gxd::guided_advance_kernel<W>),
                  reinterpret_cast<const void*>(&gxd::guided_fused_kernel<W, B>)};
}

bool gk_lookup(int W, int B, GKernels& k) {
#define GX_GK(w, b) \
  if (W == w && B == b) { k = gk<w, b>(); return true; }
  GX_GK(1, 4) GX_GK(1, 8) GX_GK(1, 16) GX_GK(1, 32)
  GX_GK(2, 4) GX_GK(2, 8) GX_GK(2, 16) GX_GK(2, 32)
  GX_GK(4, 4) GX_GK(4, 8) GX_GK(4, 16) GX_GK(4, 32)
#undef GX_GK
  return false;
}

int log2_of(uint64_t x) {
  int l = 0;
  while ((1ull << l) < x) ++l;
  return l;
}

struct GPlan {
  int W, B, rounds, nbins;
  float scale;
  uint32_t batch_cap;
  uint64_t nb, slots, bin_cap, log_cap, pend_cap;
  uint64_t off_ctl, off_blob, off_tcw, off_bincnt, off_table, off_bins, off_batch, off_log, off_pend_hist, off_pend,
      total;
  GKernels k;
};

gx_status guided_plan(const Net& net, const gx_explore_opts* o, GPlan& P) {
  gx_explore_opts d;
  gx_default_opts(&d);
  if (!o) o = &d;
  P.W = (int)net.slot_words;
  P.B = o->bucket_words ? (int)o->bucket_words : 8;
  if (P.B < P.W || !gk_lookup(P.W, P.B, P.k)) return fail(GX_ERR_INVALID, "unsupported bucket_words for guided search");
  if (net.lay.max_source >= gxd::kShareFrom) P.k.expand = P.k.expand_share;
  P.rounds = o->hash_rounds ? (int)o->hash_rounds : 8;
  if (P.rounds < 1 || P.rounds > kMaxRounds) return fail(GX_ERR_INVALID, "hash_rounds must be 1..64");
  P.nbins = o->guided_bins ? (int)o->guided_bins : 32;
  if (P.nbins < 1 || P.nbins > 1024) return fail(GX_ERR_INVALID, "guided_bins must be 1..1024");
  P.scale = o->guided_scale > 0.f ? o->guided_scale : 1.0f;
  P.batch_cap = o->guided_batch ? o->guided_batch : 8192;
  const uint64_t table_bytes = o->table_bytes ? o->table_bytes : (1ull << 30);
  uint64_t nb = 1;
  while (nb * 2 * 4ull * P.B <= table_bytes) nb *= 2;
  if (nb < 2) return fail(GX_ERR_INVALID, "table_bytes is smaller than two buckets");
  P.nb = nb;
  P.slots = nb * (uint64_t)(P.B / P.W);
  P.log_cap = P.slots;                                   // every state is expanded at most once
  P.bin_cap = std::max<uint64_t>(P.batch_cap, (P.slots + P.nbins - 1) / P.nbins + 1);
  // one iteration inserts at most batch x (successors of a state) states, and
  // never more than the table holds
  P.pend_cap = std::min<uint64_t>(P.slots, (uint64_t)P.batch_cap * std::max<uint64_t>(net.max_succ, 1));
  const uint64_t E = (uint64_t)P.W + 1;
  uint64_t off = 0;
  P.off_ctl = off;
  off = a256(off + sizeof(GuidedCtl));
  P.off_blob = off;
  off = a256(off + 4ull * net.blob.size());
  P.off_tcw = off;
  off = a256(off + sizeof(gxt::TcWeights));
  P.off_bincnt = off;
  off = a256(off + 8ull * P.nbins);
  P.off_table = off;
  off = a256(off + 4ull * P.B * P.nb);
  P.off_bins = off;
  off = a256(off + 4ull * E * P.bin_cap * P.nbins);
  P.off_batch = off;
  off = a256(off + 4ull * E * P.batch_cap);
  P.off_log = off;
  off = a256(off + 4ull * E * P.log_cap);
  P.off_pend_hist = off;
  off = a256(off + 16ull * P.pend_cap);
  P.off_pend = off;
  off = a256(off + 4ull * E * P.pend_cap);
  P.total = off;
  return GX_OK;
}

}  // namespace

void release_guided(gx_net* h) {
  if (h->guided_exec) cudaGraphExecDestroy(static_cast<cudaGraphExec_t>(h->guided_exec));
  if (h->guided_graph) cudaGraphDestroy(static_cast<cudaGraph_t>(h->guided_graph));
  h->guided_exec = nullptr;
  h->guided_graph = nullptr;
  h->guided_key.clear();
}

namespace {

// One guided search as a graph: clear the control block, bins and table,
// insert the initial state, pop the first batch, then WHILE(cond) {expand,
// score, advance (which pops the next batch)}.
gx_status build_guided_graph(gx_net* h, const GPlan& P, GuidedArgs a, int grid, size_t smem, int score_grid,
                             bool fused, int fused_grid, size_t fused_smem) {
  release_guided(h);
  h->release_guided = &release_guided;
  cudaGraph_t g;
  GG_CUDA(cudaGraphCreate(&g, 0));
  h->guided_graph = g;
  cudaGraphConditionalHandle cond;
  GG_CUDA(cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault));
  a.cond = cond;
  std::vector<cudaGraphNode_t> clears;
  auto add_memset = [&](void* dst, uint64_t words) -> cudaError_t {
    cudaMemsetParams mp{};
    mp.dst = dst;
    mp.value = 0;
    mp.elementSize = 4;
    mp.width = words;
    mp.height = 1;
    cudaGraphNode_t nd;
    cudaError_t e = cudaGraphAddMemsetNode(&nd, g, nullptr, 0, &mp);
    clears.push_back(nd);
    return e;
  };
  GG_CUDA(add_memset(a.ctl, sizeof(GuidedCtl) / 4));
  {  // the scorer's weight image, packed once per search
    const float* pp = a.params;
    gxt::TcWeights* pw = a.tcw;
    void* pargs[] = {&pp, &pw};
    cudaKernelNodeParams kp{};
    kp.func = reinterpret_cast<void*>(&gxt::tc_pack_kernel);
    kp.gridDim = dim3(gxt::kTcPackBlocks);
    kp.blockDim = dim3(256);
    kp.kernelParams = pargs;
    cudaGraphNode_t nd;
    GG_CUDA(cudaGraphAddKernelNode(&nd, g, nullptr, 0, &kp));
    clears.push_back(nd);
  }
  GG_CUDA(add_memset(a.bin_count, 2ull * P.nbins));
  const uint64_t words = (uint64_t)P.B * P.nb;
  constexpr uint64_t kPiece = 1ull << 30;
  for (uint64_t w0 = 0; w0 < words; w0 += kPiece) GG_CUDA(add_memset(a.table + w0, std::min(kPiece, words - w0)));
  auto add_kernel = [&](cudaGraph_t gr, const cudaGraphNode_t* deps, size_t nd, const void* fn, dim3 gd, dim3 bd,
                        size_t sh, cudaGraphNode_t* out) -> cudaError_t {
    void* args[] = {&a};
    cudaKernelNodeParams kp{};
    kp.func = const_cast<void*>(fn);
    kp.gridDim = gd;
    kp.blockDim = bd;
    kp.sharedMemBytes = (unsigned)sh;
    kp.kernelParams = args;
    return cudaGraphAddKernelNode(out, gr, deps, nd, &kp);
  };
  cudaGraphNode_t reset, init, start, ex, sc, adv, cnode;
  GG_CUDA(add_kernel(g, clears.data(), clears.size(), reinterpret_cast<const void*>(&gxd::guided_reset_kernel),
                     dim3(1), dim3(1), 0, &reset));
  GG_CUDA(add_kernel(g, &reset, 1, P.k.init, dim3(1), dim3(32), 0, &init));
  GG_CUDA(add_kernel(g, &init, 1, P.k.start, dim3(1), dim3(1024), 0, &start));
  cudaGraphNodeParams cp{};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = cond;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  GG_CUDA(cudaGraphAddNode(&cnode, g, &start, nullptr, 1, &cp));
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  if (fused) {
    GG_CUDA(add_kernel(body, nullptr, 0, P.k.fused, dim3(fused_grid), dim3(gxd::kFusedThreads), fused_smem, &ex));
    GG_CUDA(add_kernel(body, &ex, 1, P.k.advance, dim3(1), dim3(1024), 0, &adv));
  } else {
    GG_CUDA(add_kernel(body, nullptr, 0, P.k.expand, dim3(grid), dim3(kBlock), smem, &ex));
    GG_CUDA(add_kernel(body, &ex, 1, P.k.score, dim3(score_grid), dim3(gxt::kRows), gxt::kTcSmemBytes, &sc));
    GG_CUDA(add_kernel(body, &sc, 1, P.k.advance, dim3(1), dim3(1024), 0, &adv));
  }
  cudaGraphExec_t exec;
  GG_CUDA(cudaGraphInstantiate(&exec, g, 0));
  h->guided_exec = exec;
  return GX_OK;
}

}  // namespace

gx_status run_guided(gx_net* h, const gx_explore_opts* opts, void* ws, uint64_t ws_bytes, cudaStream_t st) {
  const Net& net = h->net;
  if (!h->guided_params) return fail(GX_ERR_INVALID, "guided mode needs scoring weights (gx_guided_set_weights)");
  for (uint32_t p = 0; p < net.n_procs; ++p)
    if (net.n_states[p] > 16) return fail(GX_ERR_INVALID, "guided mode needs at most 16 local states per process");
  GPlan P;
  gx_status s = guided_plan(net, opts, P);
  if (s != GX_OK) return s;
  if (!ws) return fail(GX_ERR_INVALID, "guided search needs a workspace (gx_guided_workspace_bytes)");
  if (ws_bytes < P.total)
    return fail(GX_ERR_OOM, "workspace holds " + std::to_string(ws_bytes) + " bytes, need " + std::to_string(P.total));
  int dev = 0, sms = 0, optin = 0;
  GG_CUDA(cudaGetDevice(&dev));
  GG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  GG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  char* base = static_cast<char*>(ws);
  GuidedCtl* ctl = reinterpret_cast<GuidedCtl*>(base + P.off_ctl);
  GuidedArgs a{};
  a.blob = reinterpret_cast<const uint32_t*>(base + P.off_blob);
  a.lay = net.lay;
  a.blob_words = (uint32_t)net.blob.size();
  hash_multipliers(a.muls.m, kMaxRounds);
  a.rounds = P.rounds;
  a.log2nb = log2_of(P.nb);
  a.table = reinterpret_cast<uint32_t*>(base + P.off_table);
  a.ctl = ctl;
  a.bin_count = reinterpret_cast<unsigned long long*>(base + P.off_bincnt);
  a.bins = reinterpret_cast<uint32_t*>(base + P.off_bins);
  a.bin_cap = P.bin_cap;
  a.nbins = P.nbins;
  a.scale = P.scale;
  a.batch = reinterpret_cast<uint32_t*>(base + P.off_batch);
  a.batch_cap = P.batch_cap;
  a.log = reinterpret_cast<uint32_t*>(base + P.off_log);
  a.log_cap = P.log_cap;
  a.params = h->guided_params;
  a.tcw = reinterpret_cast<gxt::TcWeights*>(base + P.off_tcw);
  a.pend_hist = reinterpret_cast<uint4*>(base + P.off_pend_hist);
  a.pend = reinterpret_cast<uint32_t*>(base + P.off_pend);
  a.pend_cap = P.pend_cap;
  for (int w = 0; w < 4; ++w) a.init_vec[w] = net.init_vec[w];
  const size_t blob_bytes = 4ull * net.blob.size();
  a.stage = (blob_bytes <= (size_t)optin - 32 * 1024) ? 1 : 0;
  const size_t smem = a.stage ? blob_bytes : 0;
  GG_CUDA(allow_smem(P.k.expand, (size_t)optin));
  GG_CUDA(cudaFuncSetAttribute(P.k.score, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gxt::kTcSmemBytes));
  GG_CUDA(cudaFuncSetAttribute(P.k.score, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  int per_sm = 0;
  GG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, P.k.expand, kBlock, smem));
  const int grid = sms * std::max(per_sm, 1);
  const int score_grid = sms * gxt::tc_ctas_per_sm(dev);
  // the fused kernel: its shared memory holds the scorer, the staged rows and the blob
  const bool fused = opts && opts->guided_fused;
  auto fused_bytes = [&](size_t b) {
    return P.W == 1 ? gxd::fused_smem_bytes<1>(b) : P.W == 2 ? gxd::fused_smem_bytes<2>(b) : gxd::fused_smem_bytes<4>(b);
  };
  size_t fused_smem = 0;
  int fused_grid = 0;
  if (fused) {
    a.stage = fused_bytes(blob_bytes) <= (size_t)optin ? 1 : 0;  // else the tables are read from global memory
    fused_smem = fused_bytes(a.stage ? blob_bytes : 0);
    GG_CUDA(allow_smem(P.k.fused, (size_t)optin));
    int fp = 0;
    GG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fp, P.k.fused, gxd::kFusedThreads, fused_smem));
    fp = std::min(std::max(fp, 1), 4);  // TMEM: 128 columns per CTA, 512 per SM
    fused_grid = sms * fp;
  }

  cudaEvent_t e0, e1;
  GG_CUDA(cudaEventCreate(&e0));
  GG_CUDA(cudaEventCreate(&e1));
  GG_CUDA(cudaEventRecord(e0, st));
  GG_CUDA(cudaMemcpyAsync(base + P.off_blob, net.blob.data(), blob_bytes, cudaMemcpyHostToDevice, st));
  a.max_iters = P.log_cap + 2;  // each iteration expands a state or ends the search
  GuidedCtl hc{};
  uint64_t iters = 0;
  const bool device_loop = !(opts && opts->host_loop);
  if (device_loop) {
    // the graph holds the arguments by value: rebuild it when anything changes
    std::vector<unsigned char> key(sizeof(gx_explore_opts) + 4 * sizeof(uint64_t));
    const uint64_t extra[4] = {reinterpret_cast<uint64_t>(ws), P.total, reinterpret_cast<uint64_t>(a.params),
                               (uint64_t)smem};
    if (opts) std::memcpy(key.data(), opts, sizeof(gx_explore_opts));
    std::memcpy(key.data() + sizeof(gx_explore_opts), extra, sizeof(extra));
    if (!h->guided_exec || h->guided_key != key) {
      s = build_guided_graph(h, P, a, grid, smem, score_grid, fused, fused_grid, fused_smem);
      if (s != GX_OK) return s;
      h->guided_key = key;
    }
    GG_CUDA(cudaGraphLaunch(static_cast<cudaGraphExec_t>(h->guided_exec), st));
  } else {
    GuidedCtl init{};
    init.found = ~0ull;
    GG_CUDA(cudaMemcpyAsync(ctl, &init, sizeof(init), cudaMemcpyHostToDevice, st));
    GG_CUDA(cudaMemsetAsync(a.bin_count, 0, 8ull * P.nbins, st));
    GG_CUDA(cudaMemsetAsync(a.table, 0, 4ull * P.B * P.nb, st));
    gxt::tc_pack_kernel<<<gxt::kTcPackBlocks, 256, 0, st>>>(a.params, a.tcw);
    GG_CUDA(cudaGetLastError());
    void* args[] = {&a};
    GG_CUDA(cudaLaunchKernel(P.k.init, dim3(1), dim3(32), args, 0, st));
    while (true) {
      GG_CUDA(cudaLaunchKernel(P.k.select, dim3(1), dim3(1024), args, 0, st));
      if (fused) {
        GG_CUDA(cudaLaunchKernel(P.k.fused, dim3(fused_grid), dim3(gxd::kFusedThreads), args, fused_smem, st));
      } else {
        GG_CUDA(cudaLaunchKernel(P.k.expand, dim3(grid), dim3(kBlock), args, smem, st));
        GG_CUDA(cudaLaunchKernel(P.k.score, dim3(score_grid), dim3(gxt::kRows), args, gxt::kTcSmemBytes, st));
      }
      GG_CUDA(cudaMemcpyAsync(&hc, ctl, sizeof(hc), cudaMemcpyDeviceToHost, st));
      GG_CUDA(cudaStreamSynchronize(st));
      ++iters;
      if (hc.found != ~0ull || hc.done || hc.error) break;
    }
  }
  // the deadlock's path, walked on the device into the batch buffer (free now)
  {
    uint32_t* out = a.batch;
    uint64_t cap = a.batch_cap;
    void* pargs[] = {&a, &out, &cap};
    GG_CUDA(cudaLaunchKernel(P.k.path, dim3(1), dim3(1), pargs, 0, st));
  }
  GG_CUDA(cudaMemcpyAsync(&hc, ctl, sizeof(hc), cudaMemcpyDeviceToHost, st));
  GG_CUDA(cudaEventRecord(e1, st));
  GG_CUDA(cudaStreamSynchronize(st));
  float ms = 0;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);

  // the path of the deadlock: follow parent log indices back to the initial state
  h->guided_trace.clear();
  h->deadlocks.clear();
  h->violations.clear();
  const int E = P.W + 1;
  if (device_loop) iters = hc.iters;
  if (hc.found != ~0ull && hc.path_len > 0) {
    // deadlock first in the buffer: reverse while unpacking
    std::vector<uint32_t> raw(hc.path_len * (uint64_t)E);
    GG_CUDA(cudaMemcpy(raw.data(), a.batch, 4ull * raw.size(), cudaMemcpyDeviceToHost));
    std::vector<uint32_t> local(net.n_procs);
    for (uint64_t i = hc.path_len; i-- > 0;) {
      uint32_t w4[4] = {0, 0, 0, 0};
      for (int w = 0; w < P.W; ++w) w4[w] = raw[i * E + w];
      unpack_host(net, w4, local.data());
      h->guided_trace.insert(h->guided_trace.end(), local.begin(), local.end());
    }
    h->deadlocks = local;
  } else if (hc.found != ~0ull) {  // a path longer than the batch buffer: one entry at a time
    std::vector<std::vector<uint32_t>> path;
    uint64_t li = hc.found;
    while (true) {
      uint32_t e[5] = {0, 0, 0, 0, 0};
      GG_CUDA(cudaMemcpy(e, a.log + li * E, 4ull * E, cudaMemcpyDeviceToHost));
      uint32_t w4[4] = {0, 0, 0, 0};
      for (int w = 0; w < P.W; ++w) w4[w] = e[w];
      std::vector<uint32_t> local(net.n_procs);
      unpack_host(net, w4, local.data());
      path.push_back(local);
      if (e[P.W] == 0xFFFFFFFFu || path.size() > P.log_cap) break;
      li = e[P.W];
    }
    std::reverse(path.begin(), path.end());
    for (const auto& st2 : path) h->guided_trace.insert(h->guided_trace.end(), st2.begin(), st2.end());
    h->deadlocks = path.back();
  }
  h->launches = 0;
  gx_stats_t& S = h->stats;
  std::memset(&S, 0, sizeof(S));
  S.states = hc.inserted;
  S.explored = hc.log_count;
  S.transitions = hc.transitions;
  S.deadlock_count = hc.found != ~0ull ? 1 : 0;
  S.first_deadlock_level = hc.found != ~0ull ? (int64_t)(h->guided_trace.size() / net.n_procs) - 1 : -1;
  S.table_slots = P.slots;
  S.vector_words = net.vector_words;
  S.slot_words = (uint32_t)P.W;
  S.bucket_words = (uint32_t)P.B;
  S.group_lanes = 1;
  S.hash_rounds = (uint32_t)P.rounds;
  S.complete = hc.done ? 1u : 0u;
  S.fill = (double)hc.inserted / (double)P.slots;
  S.gpu_ms = ms;
  S.expand_launches = iters;
  S.probes = hc.probes;
  h->levels.clear();
  h->have_result = true;
  gx_status rs = GX_OK;
  if (hc.error & ERR_TABLE_FULL) rs = fail(GX_ERR_TABLE_FULL, "hash table full during guided search");
  else if (hc.error & ERR_BINS) rs = fail(GX_ERR_FRONTIER_OVERFLOW, "priority bins full");
  else if (hc.error & ERR_LOG) rs = fail(GX_ERR_OOM, "log of expanded states full");
  else if (hc.error & ERR_WIDE) rs = fail(GX_ERR_INVALID, "a local state index is 16 or more");
  else if (hc.error & ERR_PENDING) rs = fail(GX_ERR_FRONTIER_OVERFLOW, "pending buffer of new states full");
  else if (hc.error & ERR_SPIN) rs = fail(GX_ERR_SPIN_LIMIT, "tensor-core scoring timed out waiting for an MMA");
  S.status = (uint32_t)rs;
  return rs;
}

}  // namespace gx

extern "C" {

gx_status gx_guided_set_weights(gx_net* h, const float* params) {
  gx::clear_error();
  if (!h) return gx::fail(GX_ERR_INVALID, "net is NULL");
  h->guided_params = params;
  return GX_OK;
}

gx_status gx_guided_workspace_bytes(const gx_net* h, const gx_explore_opts* opts, uint64_t* bytes) {
  gx::clear_error();
  if (!h || !bytes) return gx::fail(GX_ERR_INVALID, "net or bytes is NULL");
  gx::GPlan P;
  gx_status s = gx::guided_plan(h->net, opts, P);
  if (s != GX_OK) return s;
  *bytes = P.total;
  return GX_OK;
}

gx_status gx_guided_trace(const gx_net* h, uint32_t* out, uint32_t cap, uint32_t* len) {
  gx::clear_error();
  if (!h) return gx::fail(GX_ERR_INVALID, "net is NULL");
  const uint32_t n = h->net.n_procs;
  const uint32_t states = (uint32_t)(h->guided_trace.size() / n);
  if (cap && !out) return gx::fail(GX_ERR_INVALID, "out is NULL");
  const uint32_t k = std::min(states, cap);
  if (k) std::memcpy(out, h->guided_trace.data(), 4ull * n * k);
  if (len) *len = states;
  return GX_OK;
}

gx_status gx_training_set(gx_net* h, void* ws, uint64_t ws_bytes, void* stream, uint32_t* dist,
                          uint32_t max_dist, uint8_t* hist_out, float* label_out, uint64_t cap, uint64_t* n_out) {
  gx::clear_error();
  if (!h || !ws || !dist) return gx::fail(GX_ERR_INVALID, "net, workspace or dist_scratch is NULL");
  if (!h->have_result || h->levels.empty()) return gx::fail(GX_ERR_STATE, "run gx_explore on this network first");
  if (ws_bytes && ws_bytes < h->ws_total) return gx::fail(GX_ERR_INVALID, "workspace smaller than the last search's");
  if (max_dist == 0) return gx::fail(GX_ERR_INVALID, "max_dist must be positive");
  if (cap && (!hist_out || !label_out)) return gx::fail(GX_ERR_INVALID, "output arrays are NULL");
  const gx_stats_t& S = h->stats;
  gx::GKernels k;
  if (!gx::gk_lookup((int)S.slot_words, (int)S.bucket_words, k))
    return gx::fail(GX_ERR_INVALID, "no labelling kernel for this table layout");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* base = static_cast<char*>(ws);
  const uint64_t slots = S.table_slots, states = S.states;
  gxd::LabelArgs a{};
  a.table = reinterpret_cast<const uint32_t*>(base + h->ws_off_table);
  a.blob = reinterpret_cast<const uint32_t*>(base + h->ws_off_blob);
  a.lay = h->net.lay;
  a.staged_words = h->net.blob.size() <= 11 * 1024 ? (uint32_t)h->net.blob.size() : 0;
  gx::hash_multipliers(a.muls.m, gx::kMaxRounds);
  a.rounds = (int)S.hash_rounds;
  a.log2nb = gx::log2_of(slots * S.slot_words / S.bucket_words);
  a.slots = slots;
  a.cap = states;
  a.index = dist;
  int dev = 0, sms = 0;
  GG_CUDA(cudaGetDevice(&dev));
  GG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int grid = sms * 8;
  const size_t smem = 4ull * a.staged_words;
  gx::TempMem temp{st};
  uint64_t n = 0, bad = 0;  // states found
  // With lists: temporary memory for the control block, the lists (28 bytes a state) and, after
  // a complete search with at most 2^28 transitions, every state's successors (4 bytes each).
  // Less when there is no room, and no lists at all when there is none for them either.
  const uint64_t lists = gx::a256(sizeof(gxd::LabelCtl));
  if (states < (1ull << 32)) {
    a.adj_cap = S.complete && S.transitions <= (1ull << 28) ? S.transitions : 0;
    if (!temp.alloc(lists + 28 * states + 4 * a.adj_cap) && a.adj_cap) {
      a.adj_cap = 0;  // look the successors up in every round
      temp.alloc(lists + 28 * states);
    }
  }
  bool listed = temp.p != nullptr;
  if (listed) {
    a.ctl = reinterpret_cast<gxd::LabelCtl*>(temp.p);
    a.slot_of = reinterpret_cast<unsigned long long*>(temp.p + lists);
    a.d = reinterpret_cast<uint32_t*>(a.slot_of + states);
    a.first = a.d + states;
    a.last = a.first + states;
    a.todo[0] = a.last + states;
    a.todo[1] = a.todo[0] + states;
    a.adj = a.todo[1] + states;
    GG_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(gxd::LabelCtl), st));
    k.label_collect<<<grid, gx::kBlock, 0, st>>>(a);
    if (a.adj_cap) k.label_adj<<<grid, gx::kBlock, smem, st>>>(a);
    GG_CUDA(cudaGetLastError());
    gxd::LabelCtl hc{};
    constexpr uint32_t kAhead = 16;  // rounds launched before the host looks whether any is needed
    for (uint32_t r = 1; r <= max_dist; ++r) {
      if (a.adj_cap) gxd::label_round_kernel<<<grid, gx::kBlock, 0, st>>>(a, r);
      else k.label_lookup_round<<<grid, gx::kBlock, smem, st>>>(a, r);
      GG_CUDA(cudaGetLastError());
      if (r % kAhead == 0 && r < max_dist) {
        GG_CUDA(cudaMemcpyAsync(&hc, a.ctl, sizeof(hc), cudaMemcpyDeviceToHost, st));
        GG_CUDA(cudaStreamSynchronize(st));
        if (hc.states > states || (a.adj_cap && hc.edges > a.adj_cap) || hc.left[r & 3] == 0 ||
            hc.left[r & 3] == hc.left[(r - 1) & 3])
          break;
      }
    }
    k.label_gather<<<grid, gx::kBlock, 0, st>>>(a, max_dist, hist_out, label_out, cap);
    GG_CUDA(cudaGetLastError());
    GG_CUDA(cudaMemcpyAsync(&hc, a.ctl, sizeof(hc), cudaMemcpyDeviceToHost, st));
    GG_CUDA(cudaStreamSynchronize(st));
    n = hc.states;
    bad = hc.bad;
    // (a table that was written to since the search: its states and successors are not held)
    if (hc.states > states || (a.adj_cap && hc.edges > a.adj_cap)) listed = false;
  }
  if (!listed) {
    temp.release();
    unsigned long long* flags = reinterpret_cast<gx::Ctl*>(base + h->ws_off_ctl)->digest;
    k.slot_init<<<grid, gx::kBlock, 0, st>>>(a);
    GG_CUDA(cudaGetLastError());
    for (uint32_t r = 1; r <= max_dist; ++r) {
      unsigned long long changed = 0;
      GG_CUDA(cudaMemsetAsync(flags, 0, sizeof(changed), st));
      k.slot_round<<<grid, gx::kBlock, smem, st>>>(a, r, flags);
      GG_CUDA(cudaGetLastError());
      GG_CUDA(cudaMemcpyAsync(&changed, flags, sizeof(changed), cudaMemcpyDeviceToHost, st));
      GG_CUDA(cudaStreamSynchronize(st));
      if (!changed) break;
    }
    unsigned long long res[2] = {0, 0};
    GG_CUDA(cudaMemsetAsync(flags, 0, sizeof(res), st));
    k.slot_gather<<<grid, gx::kBlock, 0, st>>>(a, max_dist, hist_out, label_out, cap, flags);
    GG_CUDA(cudaGetLastError());
    GG_CUDA(cudaMemcpyAsync(res, flags, sizeof(res), cudaMemcpyDeviceToHost, st));
    GG_CUDA(cudaStreamSynchronize(st));
    n = res[0];
    bad = res[1];
  }
  if (n_out) *n_out = n;
  if (bad) return gx::fail(GX_ERR_INVALID, "a process has a local state index of 16 or more");
  // content order (see ex_greater): buffers of 20 bytes an example, a power of two of them
  const uint64_t m = std::min<uint64_t>(n, cap);
  if (m > 1) {
    uint64_t n2 = 1;
    while (n2 < m) n2 <<= 1;
    if (temp.bytes < 20 * n2) {
      temp.release();
      if (!temp.alloc(20 * n2)) return gx::fail(GX_ERR_CUDA, "no device memory to sort the examples in");
    }
    uint4* sh = reinterpret_cast<uint4*>(temp.p);
    uint32_t* sl = reinterpret_cast<uint32_t*>(sh + n2);
    const int tiles = (int)std::max<uint64_t>(1, n2 / gxd::kTile);
    const uint64_t first = std::min<uint64_t>(n2, gxd::kTile);
    gxd::ex_tile_kernel<<<tiles, gxd::kTileThreads, gxd::kTileBytes, st>>>(sh, sl, n2, 2, first, 1, hist_out, label_out, m);
    for (uint64_t k2 = 2 * first; k2 <= n2; k2 <<= 1) {
      uint64_t j = k2 >> 1;
      while (j >= (uint64_t)gxd::kTile) {
        const int two = j / 2 >= (uint64_t)gxd::kTile;
        gxd::ex_wide_kernel<<<grid, 256, 0, st>>>(sh, sl, n2, k2, j, two);
        j >>= two ? 2 : 1;
      }
      gxd::ex_tile_kernel<<<tiles, gxd::kTileThreads, gxd::kTileBytes, st>>>(sh, sl, n2, k2, k2, 0, nullptr, nullptr, 0);
    }
    gxd::ex_store_kernel<<<grid, 256, 0, st>>>(sh, sl, m, hist_out, label_out);
    GG_CUDA(cudaGetLastError());
    GG_CUDA(cudaStreamSynchronize(st));
  }
  return GX_OK;
}

}  // extern "C"
