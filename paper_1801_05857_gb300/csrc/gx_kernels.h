// Host-visible interface between the level loop and the templated kernels.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "gx_internal.h"

namespace gx {

constexpr int kMaxRounds = 64;
constexpr int kBlock = 256;  // threads per CTA for every exploration kernel

enum : uint32_t { ERR_TABLE_FULL = 1u, ERR_FRONTIER = 2u, ERR_SPIN = 4u };

// Device control block of one search (lives at the start of the workspace).
struct Ctl {
  unsigned long long claim;        // frontier chunks handed out in the current level
  unsigned long long next_end;     // absolute end of the frontier ring's filled part
  unsigned long long transitions;  // successors generated, with multiplicity
  unsigned long long dl_count, dl_sum, dl_xor;
  unsigned long long probes;       // buckets read by find-or-put
  unsigned int error;              // ERR_* bits
  unsigned int pad;
  unsigned long long digest[3];    // gx_set_digest: count, sum, xor
  unsigned long long viol_count, viol_sum, viol_xor;  // safety check
  // device-driven level loop: the level to expand next and the loop's bookkeeping
  unsigned long long cur_begin, cur_end;
  unsigned long long n_levels;      // entries of the level-size list (level 0 included)
  unsigned long long levels_done;   // levels expanded
  unsigned long long explored;
  unsigned long long t_prev;        // %globaltimer (ns) at the end of the previous level
  long long first_dl, first_viol;   // level of the first deadlock / violation, -1 if none
  unsigned int complete, yielded;   // the frontier ran empty / the level arrays filled up
  unsigned int small_launches, large_levels;  // launches of the few-state kernel; levels beside it
};
static_assert(sizeof(Ctl) <= 256, "control block");

// Hash-constant multipliers travel by value in the kernel parameters.
struct Muls {
  uint64_t m[kMaxRounds];
};

// GPU-wide cache of recently seen vectors: 2^n direct-mapped entries in global
// memory, cleared at the start of a search (nullptr = off).  A vector's fields
// packed side by side are a number of at most 64 bits.  Its low bits, plus one,
// are an entry's content (0 = empty); the n bits above them, mixed with a hash of
// the low ones, are the entry's index, which therefore gives them back: an entry
// holds a vector exactly, in 16 or 32 bits where that is enough.
// (cache_layout in gx_explore.cu fills it in.)
struct SeenCache {
  void* base;
  uint64_t tag_mask;  // the low bits: 2^shift - 1
  uint32_t shift;     // bits - n (0 when bits <= n)
  uint32_t mask;      // 2^n - 1
  uint32_t mix_shift; // 32 - n
  uint32_t log2_bytes;  // of an entry: 1, 2 or 3
  uint32_t word_at[3];  // bit offset in the key of the payload of words 1, 2, 3 (64: no fields;
                        // set without a cache too, for the per-warp one)
};

struct ExpandArgs {
  const uint32_t* blob;      // encoded network (global memory)
  uint32_t blob_words;
  int stage;                 // 1: copy the blob into shared memory first
  NetBlobLayout lay;
  Muls muls;                 // hash-constant multipliers
  int rounds;
  int log2nb;                // table has 2^log2nb buckets
  uint32_t* table;
  uint32_t* frontier;        // ring of vectors, W words each
  uint64_t fmask;            // ring capacity - 1 (capacity is a power of two)
  uint64_t cur_begin, cur_end;  // absolute indices of the level being expanded
  Ctl* ctl;
  uint32_t* dl_buf;          // deadlock vectors, W words each
  uint32_t dl_cap;
  int cache_log2;            // per-warp cache of recently seen vectors: 2^cache_log2 entries (0 = off)
  int cache_key64;           // its entries are 64-bit keys (4-word vectors whose fields fit)
  // safety check: a state whose field (word, shift, mask) equals watch_value violates
  int watch;
  uint32_t watch_word, watch_shift, watch_mask, watch_value;
  uint32_t* viol_buf;        // violating vectors, W words each
  uint32_t viol_cap;
  int dev_range;             // 1: read cur_begin / cur_end from the control block
  // Region passes: a level is expanded in several passes, and a pass probes only
  // the successors whose first bucket b has (b & region_mask) == region_bits, so
  // the table accesses of one pass stay inside one region of the table (see
  // gx_explore_opts.region_passes).  region_mask = 0: one pass, no filter.
  uint64_t region_mask, region_bits;
  int count_states;          // 1: this pass counts transitions, deadlocks and violations
  SeenCache gcache;
};

// The device-driven level loop (see run_search).
struct LoopArgs {
  Ctl* ctl;
  unsigned long long* lv_size;    // [cap] level sizes (level 0 = 1)
  unsigned long long* lv_tns;     // [cap] per expanded level: device time in ns (%globaltimer)
  unsigned long long* lv_probes;  // [cap] cumulative bucket reads after the level
  unsigned long long* lv_trans;   // [cap] cumulative transitions after the level
  uint32_t cap;
  int stop_dl, stop_viol;
  uint64_t max_levels;            // 0 = no limit
  cudaGraphConditionalHandle cond, cond_big;  // go on with a level / with a large one
};

// Partitioned expansion of one level (or one batch of it): successors are
// counted per table slice, scattered slice-major into a buffer, then probed
// slice by slice so the probed part of the table stays in L2.
struct PartArgs {
  uint32_t* hist;   // [nb * P]: successors of CTA b that fall in slice q, at b * P + q
  uint32_t* off;    // [nb * P]: exclusive scan over the batch's CTAs, per slice
  uint32_t* ptot;   // [P]: successors of the batch per slice
  uint32_t* tot;    // [nb]: successors per CTA
  uint32_t* succ;   // successor buffer, W words per vector, slice-major
  int nb;           // CTAs of the count and scatter passes (static frontier ranges)
  int logp;         // P = 2^logp slices
  uint64_t range;   // frontier states per CTA
  int b0, b1;       // CTAs of the current batch
};

struct InitArgs {
  Muls muls;
  int rounds, log2nb;
  uint32_t* table;
  uint32_t* frontier;
  Ctl* ctl;
  uint32_t vec[4];
};

struct DigestArgs {
  const uint32_t* table;
  uint64_t slots;
  const uint32_t* blob;
  NetBlobLayout lay;
  unsigned long long* out;   // count, sum, xor
};

struct FopArgs {
  const uint32_t* keys;
  uint64_t n;
  uint32_t* table;
  int log2nb, rounds;
  Muls muls;
  uint8_t* result;
  unsigned long long* counters;  // inserted, found, failed
};

struct KernelSet {
  cudaError_t (*expand)(const ExpandArgs&, int grid, size_t smem, int carveout, cudaStream_t);  // carveout: percent, -1: default
  cudaError_t (*part_count)(const ExpandArgs&, const PartArgs&, size_t smem, cudaStream_t);
  cudaError_t (*part_scan)(const PartArgs&, cudaStream_t);
  cudaError_t (*part_scatter)(const ExpandArgs&, const PartArgs&, size_t smem, cudaStream_t);
  cudaError_t (*part_probe)(const ExpandArgs&, const uint32_t* succ, uint64_t n, int grid, cudaStream_t);
  cudaError_t (*init)(const InitArgs&, cudaStream_t);
  cudaError_t (*fop)(const FopArgs&, int grid, cudaStream_t);
  const void* expand_fn;  // for occupancy queries and attributes
  const void* fop_fn;
  const void* part_count_fn;
  const void* part_scatter_fn;
  const void* part_probe_fn;
  const void* init_fn;    // for graph kernel nodes
  const void* small_fn;   // levels of few states, many in one launch
  size_t small_queue_bytes;  // of its dynamic shared memory
  // the set whose lanes share a state's sources and a rule's combinations (nullptr: this is
  // that set; kernels_for)
  const KernelSet* sharing;
};
constexpr uint32_t kShareFrom = 16;

// Kernels for slot width W, bucket words B and group lanes G; nullptr if the
// combination is not built.
const KernelSet* kernels_w1(int B, int G);
const KernelSet* kernels_w2(int B, int G);
const KernelSet* kernels_w4(int B, int G);
inline const KernelSet* kernels_for(int W, int B, int G) {
  if (W == 1) return kernels_w1(B, G);
  if (W == 2) return kernels_w2(B, G);
  if (W == 4) return kernels_w4(B, G);
  return nullptr;
}
// The kernels for a network and a table of `slots` slots: the sharing set for networks with a
// source of kShareFrom successors or more, and for 4-word vectors in tables below 2^26
// slots.  Large levels of these lose 1-5 % with it (1.08e8 states 40.2 -> 40.7 ms, 3.4e8 in two
// passes 185 -> 195), levels of few states a warp gain as much as half (20,736 states, one
// pass 0.38 -> 0.31 ms, four 0.88 -> 0.54; 2^18 states of 124 processes in four passes 3.09
// -> 1.16, where the kernels before the staged ones took 2.19); 2^26 slots hold some 4e7
// states, whose levels are still mostly of the second kind.
inline const KernelSet* kernels_for(const Net& net, int B, int G, uint64_t slots) {
  const KernelSet* ks = kernels_for((int)net.slot_words, B, G);
  const bool share = net.lay.max_source >= kShareFrom || (net.slot_words == 4 && slots < (1ull << 26));
  return ks && share ? ks->sharing : ks;
}

// Lets a kernel take all the dynamic shared memory its static part leaves: the same
// value for every caller, as the attribute belongs to the function, which searches of
// other networks launch with other sizes, from cached graphs and other threads too.
cudaError_t allow_smem(const void* fn, size_t smem_optin, size_t* static_bytes = nullptr);

cudaError_t launch_digest(int W, const DigestArgs& a, int grid, cudaStream_t st);

// Hash-constant multipliers: odd 64-bit values drawn from splitmix64.
void hash_multipliers(uint64_t* out, int n);

// The caches of seen vectors of a search, as its options and its table decide
// (gx_explore_opts): for every entry point that runs the level kernel.
struct CachePlan {
  uint64_t entries = 0;   // of the GPU-wide one (0 = off), and its bytes
  uint64_t bytes = 0;
  SeenCache seen{};       // its layout (base left out)
  uint32_t warp_log2 = 0; // per-warp one: 2^warp_log2 entries (0 = off)
};
gx_status plan_caches(const Net& net, const gx_explore_opts& o, int lanes, uint64_t slots, uint32_t regions,
                      CachePlan& p);

// How the level kernel is launched: the shared memory of a CTA, CTAs per SM and the
// split with the L1.  Fills in a's stage and per-warp cache; a's gcache must be set.
struct ExpandLaunch {
  size_t smem = 0;
  int per_sm = 0;
  int carveout = -1;  // percent of shared memory, -1: default
};
gx_status plan_expand(const Net& net, const gx_explore_opts& o, const KernelSet& ks, uint32_t warp_log2,
                      size_t smem_optin, ExpandArgs& a, ExpandLaunch& l);

// GX_DL_GUIDED search (gx_guided.cu).
gx_status run_guided(gx_net* h, const gx_explore_opts* opts, void* ws, uint64_t ws_bytes, cudaStream_t st);

}  // namespace gx
