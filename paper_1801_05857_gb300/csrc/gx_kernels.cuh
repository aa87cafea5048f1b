// Templated kernels of the exploration path, instantiated per slot width W in
// gx_kernels_w{1,2,4}.cu.
//
//   expand_kernel  one BFS level (Sec. 3): claim open vectors, generate their
//                  successors from the staged network tables, find-or-put each
//                  (Sec. 4.1), append the new ones to the next level, count
//                  transitions, record deadlocks.
//   small_levels_kernel  levels of few states, many in one launch.
//   init_kernel    inserts the initial vector (level 0).
//   fop_kernel     the isolated hash-table experiment of Sec. 5.1.
#pragma once

#include "gx_device.cuh"
#include "gx_kernels.h"

namespace gxd {

using gx::Ctl;
using gx::NetBlobLayout;

// ---- network tables (a uint32 blob; see gx_net.cpp for its layout)

template <int W>
__device__ __forceinline__ uint32_t local_state(const uint32_t* t, const NetBlobLayout& L,
                                                const uint32_t (&v)[W], uint32_t p) {
  return (word_at<W>(v, t[L.proc_word + p]) >> t[L.proc_shift + p]) & t[L.proc_mask + p];
}

// Offsets [o[0], o[1]) of class c's deltas for local state s.
__device__ __forceinline__ const uint32_t* class_range(const uint32_t* t, const NetBlobLayout& L,
                                                       uint32_t c, uint32_t s) {
  return t + L.coff + t[L.cls_base + c] + s;
}

// Number of successors of v, with multiplicity: every local edge of every
// process, plus for every rule the product of its participants' edge counts.
template <int W>
__device__ __forceinline__ uint32_t count_succ(const uint32_t* t, const NetBlobLayout& L,
                                               const uint32_t (&v)[W]) {
  uint32_t n = 0;
  for (uint32_t p = 0; p < L.n_procs; ++p) {
    const uint32_t* o = class_range(t, L, p, local_state<W>(t, L, v, p));
    n += o[1] - o[0];
  }
  for (uint32_t r = 0; r < L.n_rules; ++r) {
    uint32_t prod = 1;
    const uint32_t j1 = t[L.rule_off + r + 1];
    for (uint32_t j = t[L.rule_off + r]; j < j1 && prod; ++j) {
      const uint32_t c = t[L.rule_cls + j];
      const uint32_t* o = class_range(t, L, c, local_state<W>(t, L, v, t[L.cls_proc + c]));
      prod *= o[1] - o[0];
    }
    n += prod;
  }
  return n;
}

// Resumable enumeration of the successors of one vector: first the local
// edges process by process, then each enabled rule's combinations in
// mixed-radix order.  next() must be called at most count_succ() times.
// The two phases share the iterator's four words (it keeps register use low
// in the level kernel): idx counts processes 0..n_procs-1 and then rules
// (n_procs + r); [e, e_end) is the current process's delta range, or the
// current rule's combination counter and count; wd is the current process's
// word, or the current rule.
struct SuccIter {
  uint32_t idx, e, e_end, wd;
  __device__ __forceinline__ void init() { idx = e = e_end = wd = 0; }
};

template <int W>
__device__ __forceinline__ void next_succ(SuccIter& it, const uint32_t* t, const NetBlobLayout& L,
                                          const uint32_t (&v)[W], uint32_t (&out)[W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) out[w] = v[w];
  if (it.idx <= L.n_procs) {  // local phase (or its end)
    while (it.e == it.e_end && it.idx < L.n_procs) {
      const uint32_t p = it.idx++;
      const uint32_t* o = class_range(t, L, p, local_state<W>(t, L, v, p));
      it.e = o[0];
      it.e_end = o[1];
      it.wd = t[L.proc_word + p];
    }
    if (it.e < it.e_end) {
      xor_at<W>(out, it.wd, t[L.cdelta + it.e]);
      ++it.e;
      return;
    }
  }
  while (it.e == it.e_end && it.idx < L.n_procs + L.n_rules) {
    const uint32_t r = it.idx++ - L.n_procs;
    uint32_t prod = 1;
    const uint32_t j1 = t[L.rule_off + r + 1];
    for (uint32_t j = t[L.rule_off + r]; j < j1 && prod; ++j) {
      const uint32_t c = t[L.rule_cls + j];
      const uint32_t* o = class_range(t, L, c, local_state<W>(t, L, v, t[L.cls_proc + c]));
      prod *= o[1] - o[0];
    }
    it.wd = r;
    it.e = 0;
    it.e_end = prod;
  }
  uint32_t x = it.e++;
  const uint32_t j1 = t[L.rule_off + it.wd + 1];
  for (uint32_t j = t[L.rule_off + it.wd]; j < j1; ++j) {
    const uint32_t c = t[L.rule_cls + j];
    const uint32_t p = t[L.cls_proc + c];
    const uint32_t* o = class_range(t, L, c, local_state<W>(t, L, v, p));
    const uint32_t cnt = o[1] - o[0];
    uint32_t i = 0;
    if (cnt > 1) {  // one matching edge is the common case: no division
      i = x % cnt;
      x /= cnt;
    }
    xor_at<W>(out, t[L.proc_word + p], t[L.cdelta + o[0] + i]);
  }
}

// Successor k (k < count_succ) of v, in next_succ's order, without walking
// the ones before it: O(processes + rules) table reads.  Lets the lanes of a
// warp take different successors of one state at once.
template <int W>
__device__ __forceinline__ void seek_succ(const uint32_t* t, const NetBlobLayout& L, const uint32_t (&v)[W],
                                          uint32_t k, uint32_t (&out)[W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) out[w] = v[w];
  for (uint32_t p = 0; p < L.n_procs; ++p) {
    const uint32_t* o = class_range(t, L, p, local_state<W>(t, L, v, p));
    const uint32_t c = o[1] - o[0];
    if (k < c) {
      xor_at<W>(out, t[L.proc_word + p], t[L.cdelta + o[0] + k]);
      return;
    }
    k -= c;
  }
  for (uint32_t r = 0; r < L.n_rules; ++r) {
    const uint32_t j0 = t[L.rule_off + r], j1 = t[L.rule_off + r + 1];
    uint32_t prod = 1;
    for (uint32_t j = j0; j < j1 && prod; ++j) {
      const uint32_t c = t[L.rule_cls + j];
      const uint32_t* o = class_range(t, L, c, local_state<W>(t, L, v, t[L.cls_proc + c]));
      prod *= o[1] - o[0];
    }
    if (k < prod) {
      uint32_t x = k;
      for (uint32_t j = j0; j < j1; ++j) {
        const uint32_t c = t[L.rule_cls + j];
        const uint32_t p = t[L.cls_proc + c];
        const uint32_t* o = class_range(t, L, c, local_state<W>(t, L, v, p));
        const uint32_t cnt = o[1] - o[0];
        uint32_t i = 0;
        if (cnt > 1) {
          i = x % cnt;
          x /= cnt;
        }
        xor_at<W>(out, t[L.proc_word + p], t[L.cdelta + o[0] + i]);
      }
      return;
    }
    k -= prod;
  }
}

// Order-free digest of one state: h = fold_p mix64(h ^ (p << 32 | s_p)).
template <int W>
__device__ __forceinline__ uint64_t state_digest(const uint32_t* t, const NetBlobLayout& L,
                                                 const uint32_t (&v)[W]) {
  uint64_t h = 0;
  for (uint32_t p = 0; p < L.n_procs; ++p)
    h = mix64(h ^ (((uint64_t)p << 32) | local_state<W>(t, L, v, p)));
  return h;
}

template <int W>
__device__ __forceinline__ void load_vec(const uint32_t* p, uint32_t (&v)[W]) {
  if constexpr (W == 1) {
    v[0] = p[0];
  } else if constexpr (W == 2) {
    uint2 x = *reinterpret_cast<const uint2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  } else {
    uint4 x = *reinterpret_cast<const uint4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  }
}

template <int W>
__device__ __forceinline__ void store_vec(uint32_t* p, const uint32_t (&v)[W]) {
  if constexpr (W == 1) {
    p[0] = v[0];
  } else if constexpr (W == 2) {
    *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
  } else {
    *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

// Safety check (Sec. 3: the negated property is one more automaton of the
// network): v violates when its watched field holds the automaton's error
// state.  A violation is counted, folded into the violation digest and kept
// while there is room.
template <int W>
__device__ __forceinline__ void check_watch(const gx::ExpandArgs& a, const uint32_t* t, const NetBlobLayout& L,
                                            const uint32_t (&v)[W]) {
  uint32_t w = v[0];
#pragma unroll
  for (int i = 1; i < W; ++i)
    if (a.watch_word == (uint32_t)i) w = v[i];
  if (((w >> a.watch_shift) & a.watch_mask) != a.watch_value) return;
  const uint64_t h = state_digest<W>(t, L, v);
  const unsigned long long vi = atomicAdd(&a.ctl->viol_count, 1ull);
  atomicAdd(&a.ctl->viol_sum, (unsigned long long)h);
  atomicXor(&a.ctl->viol_xor, (unsigned long long)h);
  if (vi < a.viol_cap) store_vec<W>(a.viol_buf + vi * W, v);
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULLMASK, x, o);
  return x;
}

// Shared-memory prologue shared by the kernels: hash multipliers, then
// (optionally) the network blob.
__device__ __forceinline__ const uint32_t* stage_tables(uint32_t* sm, const gx::Muls& muls,
                                                        int rounds, const uint32_t* blob,
                                                        uint32_t blob_words, int stage,
                                                        const uint64_t*& s_muls) {
  uint64_t* m = reinterpret_cast<uint64_t*>(sm);
  for (int i = threadIdx.x; i < rounds; i += blockDim.x) m[i] = muls.m[i];
  s_muls = m;
  if (!stage) return blob;
  uint32_t* s_tab = sm + 2 * kMaxRounds;
  const uint4* src = reinterpret_cast<const uint4*>(blob);
  uint4* dst = reinterpret_cast<uint4*>(s_tab);
  for (uint32_t i = threadIdx.x; i < blob_words / 4; i += blockDim.x) dst[i] = src[i];
  return s_tab;
}

// Where find-or-put inserts and where new vectors go: one network's table and
// frontier ring (the level being expanded starts at begin()).  Read from the
// kernel's parameters, which live in the constant bank and so take no registers in
// the inner loop; the batched kernel has its own (SmemTarget).
struct ParamTarget {
  const gx::ExpandArgs& a;
  const unsigned long long* range;  // [begin, end) of the level, in shared memory
  __device__ __forceinline__ uint32_t* table() const { return a.table; }
  __device__ __forceinline__ int log2nb() const { return a.log2nb; }
  __device__ __forceinline__ int rounds() const { return a.rounds; }
  __device__ __forceinline__ unsigned long long* next_end() const { return &a.ctl->next_end; }
  __device__ __forceinline__ uint32_t* frontier() const { return a.frontier; }
  __device__ __forceinline__ uint64_t fmask() const { return a.fmask; }
  __device__ __forceinline__ uint64_t begin() const { return range[0]; }
  __device__ __forceinline__ const gx::SeenCache& gcache() const { return a.gcache; }
};

// Per-warp staging of new vectors in shared memory: lanes that inserted a
// vector append it here (ballot + popc, no atomic); whenever 32 are staged the
// last 32 are written to the next level with one global atomicAdd and one
// coalesced store.  flush() writes what is left.  All 32 lanes call push/flush
// together.
constexpr int kStage = 64;  // vectors per warp (at most 31 + 32 are ever staged)

struct WarpStage {
  uint32_t* buf;  // kStage * W words of this warp
  int n;          // staged vectors (uniform in the warp)

  template <int W, class T>
  __device__ __forceinline__ void write_out(const T& a, int m, uint32_t& err) {
    const int lane = threadIdx.x & 31;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(a.next_end(), (unsigned long long)m);
    base = __shfl_sync(FULLMASK, base, 0);
    n -= m;
    if (lane < m) {
      const uint64_t pos = base + lane;
      uint32_t v[W];
      load_vec<W>(buf + (n + lane) * W, v);
      if (pos - a.begin() <= a.fmask()) store_vec<W>(a.frontier() + (pos & a.fmask()) * W, v);
      else err |= gx::ERR_FRONTIER;
    }
    __syncwarp();
  }

  template <int W, class T>
  __device__ __forceinline__ void push(const T& a, bool ins, const uint32_t (&v)[W],
                                       uint32_t& err) {
    const int lane = threadIdx.x & 31;
    const uint32_t im = __ballot_sync(FULLMASK, ins);
    if (ins) store_vec<W>(buf + (n + __popc(im & ((1u << lane) - 1u))) * W, v);
    n += __popc(im);
    __syncwarp();
    if (n >= 32) write_out<W>(a, 32, err);
  }

  template <int W, class T>
  __device__ __forceinline__ void flush(const T& a, uint32_t& err) {
    if (n > 0) write_out<W>(a, n, err);
  }
};

// Per-warp cache of recently seen vectors (the block-local state cache of
// Fig. 2, in shared memory, per warp): direct-mapped, overwritten on a miss,
// never cleared.  A vector written into it goes on to this warp's find-or-put
// (or was found in the GPU-wide cache), so a hit means the vector is in the table
// or will be put there by this warp, and its find-or-put can be skipped.
// A torn entry -- words of two vectors -- could equal a third one and drop it, so
// an entry must be read and written whole.  1- and 2-word entries are one 32- or
// 64-bit access, and so are 4-word vectors' whose fields fit 64 bits side by side
// (cache_key).  Longer ones take 16-byte entries, whose access is several accesses
// in no fixed order: the warp's reads, the choice of one writer per entry and the
// writes are kept apart.  (3.4e8 states of 4 words, 64 field bits, two passes: 185 ms
// with 2^7 entries of 8 bytes a warp, 189 with 2^6 of 16, 197 without a cache.)
struct WarpCache {
  uint32_t* base;  // the entries, or nullptr
  uint32_t mask;
  const uint32_t* key_at;  // 4-word vectors: bit offsets of words 1..3 in a 64-bit key, or nullptr
  // For every lane with `on` set: whether v is in the cache; else it is written.  All
  // 32 lanes call it together.
  template <int W>
  __device__ __forceinline__ bool seen(bool on, const uint32_t (&v)[W]) const {
    uint32_t m = v[0] * 0x9E3779B1u;
    if constexpr (W >= 2) m += v[1] * 0x85EBCA77u;
    if constexpr (W == 4) m += v[2] * 0xC2B2AE3Du + v[3] * 0x27D4EB2Fu;
    const uint32_t i = (m >> 20) & mask;  // (2^12 entries at most)
    if constexpr (W == 1) {
      if (!on) return false;
      uint32_t* e = base + i;
      if (*e == v[0]) return true;
      *e = v[0];
      return false;
    } else if constexpr (W == 2) {
      if (!on) return false;
      unsigned long long* e = reinterpret_cast<unsigned long long*>(base) + i;
      const unsigned long long x = (unsigned long long)v[0] | ((unsigned long long)v[1] << 32);
      if (*e == x) return true;
      *e = x;
      return false;
    } else {
      static_assert(W == 4, "slot width");
      if (key_at) {
        if (!on) return false;
        unsigned long long x = v[0] & ~kTag;
#pragma unroll
        for (int w = 1; w < 4; ++w)
          if (key_at[w - 1] < 64) x |= (unsigned long long)(v[w] & ~kTag) << key_at[w - 1];
        x += 1;  // 0 is an empty entry, and 2^64 - 1 the one key that is not cached
        unsigned long long* e = reinterpret_cast<unsigned long long*>(base) + i;
        if (x == 0) return false;
        if (*e == x) return true;
        *e = x;
        return false;
      }
      const uint32_t lane = threadIdx.x & 31;
      uint4* e = reinterpret_cast<uint4*>(base) + i;
      const uint4 c = *e;
      const bool hit = on && c.x == v[0] && c.y == v[1] && c.z == v[2] && c.w == v[3];
      const bool miss = on && !hit;
      __syncwarp();
      if (miss) e->x = lane;  // (no tag: never a stored vector's first word)
      __syncwarp();
      if (miss && e->x == lane) *e = make_uint4(v[0], v[1], v[2], v[3]);
      __syncwarp();
      return hit;
    }
  }
};

// GPU-wide cache of recently seen vectors (gx::SeenCache).  A vector is written
// into it after its find-or-put found or inserted it, so every entry is a vector
// of the table and a hit can skip the table probe.  An aligned load or store of
// an entry is one access, so an entry is never seen half-written.  Successors of
// a level mostly lead into the levels just before and after it, which were
// inserted or looked up moments earlier by some warp of the GPU.
// What bounds the searches that use it is DRAM traffic of random lines (128
// bytes per bucket read, entry missed in L2 or entry written back), so entries
// are as small as the vectors allow: the 62M-state mid network (40 bits)
// takes 2^25 entries of 16 bits in the 64 MiB that held 2^23 of 64 bits.
// Every successor is looked up, four in five are found, and the instructions
// of that are what is left: so the key is only split and one half xored with a
// hash of the other (a bijection whatever the hash is), and the table's 64-bit hash
// is left to those that go on to it.  Mid network 13.8 -> 12.3 ms, deadlock search of
// 4.5e7 states 12.9 -> 11.7, random network of 1.1e8 states (64 bits) 43.1 -> 40.2.
// A hash of one multiplication left 11 % more misses in the last (42.0 ms).
struct SeenEntry {
  uint32_t index;
  unsigned long long content;  // 0: this vector is never cached
};
template <int W>
__device__ __forceinline__ SeenEntry seen_entry(const gx::SeenCache& c, const uint32_t (&v)[W]) {
  uint64_t y = v[0] & ~kTag;
#pragma unroll
  for (int w = 1; w < W; ++w)
    if (c.word_at[w - 1] < 64) y |= (uint64_t)(v[w] & ~kTag) << c.word_at[w - 1];
  const uint64_t lo = y & c.tag_mask;
  uint32_t mix = (uint32_t)lo * 0x9E3779B1u + (uint32_t)(lo >> 32) * 0x85EBCA77u;
  mix = (mix ^ (mix >> 15)) * 0xC2B2AE3Du;
  SeenEntry e;
  e.index = ((uint32_t)(y >> c.shift) ^ (mix >> c.mix_shift)) & c.mask;
  e.content = lo + 1;
  if (c.log2_bytes == 1) e.content &= 0xFFFFull;  // (the one content that does not fit becomes 0)
  else if (c.log2_bytes == 2) e.content &= 0xFFFFFFFFull;
  return e;
}
__device__ __forceinline__ unsigned long long seen_get(const gx::SeenCache& c, uint32_t i) {
  if (c.log2_bytes == 1) return __ldcg(static_cast<const unsigned short*>(c.base) + i);
  if (c.log2_bytes == 2) return __ldcg(static_cast<const unsigned int*>(c.base) + i);
  return __ldcg(static_cast<const unsigned long long*>(c.base) + i);
}
__device__ __forceinline__ void seen_put(const gx::SeenCache& c, const SeenEntry& e) {
  if (c.log2_bytes == 1) __stcg(static_cast<unsigned short*>(c.base) + e.index, (unsigned short)e.content);
  else if (c.log2_bytes == 2) __stcg(static_cast<unsigned int*>(c.base) + e.index, (unsigned int)e.content);
  else __stcg(static_cast<unsigned long long*>(c.base) + e.index, e.content);
}

// One step of find-or-put for the vector x of every lane with has set: the
// bucket, read by G lanes, that hash-constant set k gives it.  A lane whose
// vector is settled (r >= 0) has the GPU-wide cache updated and a new vector
// staged for the next level.  All 32 lanes call it together.
template <int W, int B, int G, class T>
__device__ __forceinline__ int resolve_lanes(const T& a, const uint64_t* muls, bool has, const uint32_t (&x)[W],
                                             uint64_t h, uint32_t k, uint32_t& probes, uint32_t& err, WarpStage& st) {
  int r = -1;
  const uint64_t b = seq_bucket<B>(h, k, muls, a.log2nb());
  if constexpr (G == 1) {
    if (has) r = bucket_step<W, B>(a.table() + b * (uint64_t)B, x);
  } else {
    r = bucket_step_lanes<W, B, G>(a.table(), has, b, x);
  }
  probes += has;
  if (r >= 0 && a.gcache().base) seen_put(a.gcache(), seen_entry<W>(a.gcache(), x));
  st.push<W>(a, r == FOP_INSERTED, x, err);
  return r;
}

// What a warp needs of edge class c (class p < n_procs: the local edges of process
// p), one 16-byte shared-memory read: word, shift and mask of its process's field,
// and where the offsets of its edges start in the network tables.
__device__ __forceinline__ uint4 class_desc(const uint32_t* t, const NetBlobLayout& L, uint32_t c) {
  const uint32_t p = t[L.cls_proc + c];
  return make_uint4(t[L.proc_word + p], t[L.proc_shift + p], t[L.proc_mask + p], L.coff + t[L.cls_base + c]);
}
constexpr int kMaxProcs = 124;  // gx_load_network's limit

// The processes' descriptors in shared memory; a rule's class takes its process's.
struct ProcDescs {
  const uint4* staged;
  __device__ __forceinline__ uint4 proc(const uint32_t*, const NetBlobLayout&, uint32_t p) const { return staged[p]; }
  __device__ __forceinline__ uint4 cls(const uint32_t* t, const NetBlobLayout& L, uint32_t c) const {
    uint4 d = staged[t[L.cls_proc + c]];
    d.w = L.coff + t[L.cls_base + c];
    return d;
  }
};
// All threads of a CTA fill descs (kMaxProcs entries); the caller synchronises.
__device__ __forceinline__ ProcDescs stage_descs(const uint32_t* t, const NetBlobLayout& L, uint4* descs) {
  for (uint32_t p = threadIdx.x; p < L.n_procs; p += blockDim.x) descs[p] = class_desc(t, L, p);
  return ProcDescs{descs};
}

// The first n classes' descriptors in shared memory, the others from the tables.  For
// kernels whose network tables stay in global memory (256 networks: 9.1 ms with the
// processes' alone, 8.5 so); with the tables in shared memory it makes no difference.
struct ClassDescs {
  const uint4* staged;
  uint32_t n;
  __device__ __forceinline__ uint4 cls(const uint32_t* t, const NetBlobLayout& L, uint32_t c) const {
    return c < n ? staged[c] : class_desc(t, L, c);
  }
  __device__ __forceinline__ uint4 proc(const uint32_t* t, const NetBlobLayout& L, uint32_t p) const {
    return cls(t, L, p);
  }
};

// Successor generation by a warp.  Sources of successors are the processes, then
// the rules.  Either the lanes hold one state each (lanes without one hold no
// successors) and the warp walks the sources together -- open() finds, per lane, how
// many successors the current source gives its state; every table address but the
// edge offsets is uniform -- or all lanes hold the same state and take 32 sources
// at a time (open_wide), which costs a few dozen instructions a state instead of
// as many per source: what counts in a level of few states.  emit() appends one
// successor per lane that has any left to a queue in shared memory; a state's
// successors are counted on the way, without a pass of their own.
// Share: lanes whose source is exhausted take part of what is left of another lane's
// (share), where a warp has one or a few states: a rule of many combinations would be
// one lane's work.  (4096 states with one rule of 729: guided search 4.0 -> 0.29 ms,
// batch of one such network 4.4 -> 0.29, exploration 3.8 -> 0.32; 65,536 states with one of
// 6561: exploration 57 -> 16.7.)
// Kernels of their own, for networks with a source of kShareFrom successors or more
// (max_source): the others gain nothing and would pay for the check and a register (256
// networks: 8.2 ms, with it 8.4; mid network 12.4, 12.7).
using gx::kShareFrom;
template <int W, bool Share = false>
struct WarpGen {
  uint32_t src;       // next source: process src, then rule src - n_procs (uniform)
  uint32_t e, e_end;  // this lane's successors left of its source: edges, or combinations of the rule
  uint32_t word;      // word index of the source's process; W: a rule
  uint32_t cur;       // that word of this lane's state; a rule: its index
  uint32_t stride;    // Share: every how many of its source's successors are this lane's

  template <class Desc>
  __device__ __forceinline__ void open(const uint32_t* t, const NetBlobLayout& L, Desc& desc, bool valid,
                                       const uint32_t (&v)[W]) {
    if (src < L.n_procs) {
      const uint4 d = desc.proc(t, L, src);
      word = d.x;
      cur = word_at<W>(v, d.x);
      const uint32_t* o = t + d.w + ((cur >> d.y) & d.z);
      e = valid ? o[0] : 0u;
      e_end = valid ? o[1] : 0u;
    } else {
      const uint32_t r = src - L.n_procs;
      uint32_t prod = valid ? 1u : 0u;
      const uint32_t j1 = t[L.rule_off + r + 1];
      for (uint32_t j = t[L.rule_off + r]; j < j1; ++j) {
        const uint32_t c = t[L.rule_cls + j];
        const uint4 d = desc.cls(t, L, c);
        const uint32_t* o = t + d.w + ((word_at<W>(v, d.x) >> d.y) & d.z);
        prod *= o[1] - o[0];
        if (!__any_sync(FULLMASK, prod != 0)) break;
      }
      word = W;
      cur = r;
      e = 0;
      e_end = prod;
    }
    stride = 1;
    ++src;
  }

  // The next 2^sh sources of the state v that 2^sh neighbouring lanes hold, one per lane.
  template <class Desc>
  __device__ __forceinline__ void open_wide(const uint32_t* t, const NetBlobLayout& L, Desc& desc, bool valid,
                                            const uint32_t (&v)[W], uint32_t sh) {
    const uint32_t s = src + (threadIdx.x & ((1u << sh) - 1u));
    e = e_end = 0;
    if (!valid) {
    } else if (s < L.n_procs) {
      const uint4 d = desc.proc(t, L, s);
      word = d.x;
      cur = word_at<W>(v, d.x);
      const uint32_t* o = t + d.w + ((cur >> d.y) & d.z);
      e = o[0];
      e_end = o[1];
    } else if (s < L.n_procs + L.n_rules) {
      const uint32_t r = s - L.n_procs, j1 = t[L.rule_off + r + 1];
      uint32_t prod = 1;
      for (uint32_t j = t[L.rule_off + r]; j < j1 && prod; ++j) {
        const uint32_t c = t[L.rule_cls + j];
        const uint4 d = desc.cls(t, L, c);
        const uint32_t* o = t + d.w + ((word_at<W>(v, d.x) >> d.y) & d.z);
        prod *= o[1] - o[0];
      }
      word = W;
      cur = r;
      e_end = prod;
    }
    stride = 1;
    src += 1u << sh;
  }

  // When at most half of the 2^sh lanes that hold a state have successors left, and some
  // lane has many: the ones that have none take every 2nd, 4th, ... of theirs.  act: the
  // lanes with successors left.  All 32 lanes call it together.
  __device__ __forceinline__ void share(uint32_t act, uint32_t sh) {
    static_assert(Share, "only with strides");
    const uint32_t lane = threadIdx.x & 31, n = 1u << sh, sub = lane & (n - 1u), first = lane - sub;
    const uint32_t busy = (act >> first) & (0xFFFFFFFFu >> (32u - n));
    const uint32_t k = __popc(busy);
    // (sharing 8 successors takes about as long as the steps it saves)
    if (!__any_sync(FULLMASK, 2 * k <= n && e < e_end && (e_end - e) / stride >= 8)) return;
    const uint32_t log = k > 1 ? 32u - __clz(k - 1u) : 0u;  // 2^log >= k parts of the group
    const uint32_t m = 2 * k <= n && k > 0 ? sh - log : 0u;   // 2^m lanes each
    const uint32_t part = sub & ((1u << m) - 1u);
    const bool has = m == 0 || (sub >> m) < k;
    const int from = m == 0 || !has ? (int)lane : (int)(first + __fns(busy, 0, (int)(sub >> m) + 1));
    e = __shfl_sync(FULLMASK, e, from);
    e_end = __shfl_sync(FULLMASK, e_end, from);
    word = __shfl_sync(FULLMASK, word, from);
    cur = __shfl_sync(FULLMASK, cur, from);
    stride = __shfl_sync(FULLMASK, stride, from);
    if (!has || e_end - e <= part * stride) e = e_end;
    else e += part * stride;
    stride <<= m;
  }

  // One successor into the W words at q (a lane with e < e_end).
  template <class Desc>
  __device__ __forceinline__ void emit(const uint32_t* t, const NetBlobLayout& L, Desc& desc,
                                       const uint32_t (&v)[W], uint32_t* q) {
    if (word < (uint32_t)W) {
      store_vec<W>(q, v);
      q[word] = cur ^ t[L.cdelta + e];
    } else {
      uint32_t out[W];
#pragma unroll
      for (int w = 0; w < W; ++w) out[w] = v[w];
      uint32_t x = e;
      const uint32_t j1 = t[L.rule_off + cur + 1];
      for (uint32_t j = t[L.rule_off + cur]; j < j1; ++j) {
        const uint32_t c = t[L.rule_cls + j];
        const uint4 d = desc.cls(t, L, c);
        const uint32_t* o = t + d.w + ((word_at<W>(v, d.x) >> d.y) & d.z);
        const uint32_t cnt = o[1] - o[0];
        uint32_t i = 0;
        if (cnt > 1) {  // one matching edge is the common case: no division
          i = x % cnt;
          x /= cnt;
        }
        xor_at<W>(out, d.x, t[L.cdelta + o[0] + i]);
      }
      store_vec<W>(q, out);
    }
    if constexpr (Share) e = e_end - e > stride ? e + stride : e_end;  // (no overflow: ranges end below 2^32)
    else ++e;
  }
};

// The two queues a warp keeps in shared memory, used as stacks (the last
// entries are taken, so nothing is ever moved):
//   raw   successors as generated.  A source gives the 32 states of a warp
//         different numbers of successors, so generation runs with part of the
//         lanes; hashing and the filters (region, caches) then run on a batch of
//         32 or 64 successors, so that a lane's cache lookups are in flight
//         together.
//   kept  successors that passed the filters, with the hash-constant set to try;
//         only these are hashed.  32 of them at a time read one bucket each;
//         those that met a full one go back with the next set, so a lane in a
//         crowded part of the table holds up no other.
// Successors filtered at a time.  4-word vectors: one per lane, because shared
// memory beyond 196 KB an SM leaves so little L1 that it limits the loads in
// flight (irregular 1.08e8-state network: 42.1 ms with batches of 32, 68.0 ms
// with 64, the same instructions otherwise).
template <int W>
constexpr int kBatch = W == 4 ? 32 : 64;

template <int W, int Batch = kBatch<W>>
struct WarpQueues {
  static constexpr int kSlots = Batch + 32;  // at most 31 left of a batch of 32, or Batch - 1, before the next come in
  uint32_t raw[kSlots * W];
  uint32_t kept[kSlots * W];
  uint8_t seq[kSlots];  // hash-constant set to try for each of the kept ones
};

// Resident CTAs per SM the level kernel is compiled for (register budget): a
// lane holds a bucket of B words.
// (A sharing lane holds more: 4-word slots in 4-word buckets would spill 58 bytes with 5 CTAs,
// 3.8e6 states 3.38 ms, with 4 CTAs 2.47.)
template <int W, int B, int G, bool Share = false>
struct ExpandOcc {
  static constexpr int min_ctas = Share && W == 4 && B == 4 ? 4 : B <= 8 ? (G == 1 ? 5 : 4) : (B <= 16 && G == 1 ? 4 : 3);
};

// Up to this many states per warp are generated from by several lanes each, which take
// different sources of successors.  Token ring of 11 nodes, 22 sources: levels of 4 or 5
// states a warp 18 us instead of 26-28, the search 1.61 -> 1.33 ms.  (16 states: the same
// there; levels of 8 to 16 states a warp of the mid network 30 instead of 33 us, others
// up to 2 % slower.)
// With sharing, two lanes for each of 9 to 16 states still pay (16 networks of 4096 states
// with one rule of 729: 2.4 -> 1.6 ms).
template <bool Share>
constexpr uint32_t kWideStates = Share ? 16 : 8;

// The expansion of a warp's share of one level: generate successors of its
// states until a batch is queued, filter it, and resolve what is kept 32 at a
// time -- one loop with one copy of each step (a second copy of find-or-put
// costs registers).
//   next(pos, m)   the warp's next m <= 32 states, at absolute frontier
//                  positions pos.. (m = 0: none are left); up to kWideStates
//                  are generated from by several lanes each
//   desc           the descriptors of processes and classes (ProcDescs, ClassDescs)
//   seen(v)        a lane's state, once, when it is taken
//   done(v, n)     a lane's state and the number of its successors
//   keep(on, x)    the filters before the GPU-wide cache: whether a lane's successor x
//                  (if on) passes them; all 32 lanes call it together
// All 32 lanes call it together; returns with the queues empty.  Wide: whether
// few states are treated so at all; Share: see WarpGen.
template <int W, int B, int G, int Batch, bool Wide = true, bool Share = false, class T, class Desc, class Next, class Seen, class Done,
          class Keep>
__device__ __forceinline__ void expand_states(const T& tg, const uint64_t* muls, const uint32_t* t,
                                              const NetBlobLayout& L, WarpQueues<W, Batch>& q, WarpStage& st,
                                              uint32_t& probes, uint32_t& err, Desc desc, Next next, Seen seen,
                                              Done done, Keep keep) {
  const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  const uint32_t n_src = L.n_procs + L.n_rules;
  int n_raw = 0, n_kept = 0;  // queued (uniform in the warp)
  uint32_t m = 0;             // states the warp holds (lanes 0..m-1)
  uint32_t v[W];
#pragma unroll
  for (int w = 0; w < W; ++w) v[w] = 0;
  uint32_t sh = 0;    // 2^sh lanes hold the same state (uniform)
  uint32_t cnt = 0;   // successors this lane has found of its state
  WarpGen<W, Share> gen;
  gen.src = n_src;
  gen.e = gen.e_end = gen.cur = gen.word = 0;
  bool more = true;  // states may be left for this warp
  while (true) {
    while (n_raw < Batch) {
      uint32_t act = __ballot_sync(FULLMASK, gen.e < gen.e_end);
      if (act != 0) {
        if constexpr (Share) {
          if (sh != 0 && __popc(act) <= 16) {
            gen.share(act, sh);
            act = __ballot_sync(FULLMASK, gen.e < gen.e_end);
          }
        }
        if ((act >> lane) & 1u) gen.emit(t, L, desc, v, q.raw + (n_raw + __popc(act & below)) * W);
        n_raw += __popc(act);
      } else if (gen.src < n_src) {
        if (Wide && sh != 0) gen.open_wide(t, L, desc, (lane >> sh) < m, v, sh);
        else gen.open(t, L, desc, lane < m, v);
        cnt += gen.e_end - gen.e;
      } else {
        if (!more) break;
        if constexpr (Wide) {
          for (uint32_t o = 1u << sh; o > 1; o >>= 1) cnt += __shfl_xor_sync(FULLMASK, cnt, o >> 1);
          if ((lane >> sh) < m && (lane & ((1u << sh) - 1u)) == 0) done(v, cnt);
        } else {
          if (lane < m) done(v, cnt);
        }
        uint64_t pos = 0;
        next(pos, m);
        more = m != 0;
        if (!more) break;
        if constexpr (Wide) {
          sh = m <= kWideStates<Share> ? (uint32_t)__clz(m - 1) - 27u : 0u;
          if ((lane >> sh) < m) {
            load_words<W>(tg.frontier() + ((pos + (lane >> sh)) & tg.fmask()) * W, v);
            if ((lane & ((1u << sh) - 1u)) == 0) seen(v);
          }
        } else if (lane < m) {
          load_words<W>(tg.frontier() + ((pos + lane) & tg.fmask()) * W, v);
          seen(v);
        }
        cnt = 0;
        gen.src = 0;
      }
    }
    __syncwarp();
    {
      const int k = n_raw < Batch ? n_raw : Batch;
      n_raw -= k;
      constexpr int K = Batch / 32;
      bool on[K];
      uint32_t x[K][W];
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const int at = (int)lane + 32 * i;
        load_vec<W>(q.raw + (n_raw + at) * W, x[i]);  // (past the k-th entry: not used)
        on[i] = keep(at < k, x[i]);
      }
      if (tg.gcache().base) {
        SeenEntry e[K];
        unsigned long long c[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
          e[i] = seen_entry<W>(tg.gcache(), x[i]);
          c[i] = on[i] ? seen_get(tg.gcache(), e[i].index) : 0ull;
        }
#pragma unroll
        for (int i = 0; i < K; ++i) on[i] = on[i] && (c[i] != e[i].content || c[i] == 0);
      }
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const uint32_t km = __ballot_sync(FULLMASK, on[i]);
        if (on[i]) {
          const int at = n_kept + __popc(km & below);
          store_vec<W>(q.kept + at * W, x[i]);
          q.seq[at] = 0;
        }
        n_kept += __popc(km);
      }
    }
    const bool last = !more && n_raw == 0;
    while (n_kept >= 32 || (last && n_kept > 0)) {
      __syncwarp();
      const int k = n_kept < 32 ? n_kept : 32;
      n_kept -= k;
      const bool has = (int)lane < k;
      uint32_t x[W];
      load_vec<W>(q.kept + (n_kept + lane) * W, x);  // (past the k-th entry: not used)
      const uint32_t n = has ? q.seq[n_kept + lane] : 0u;
      bool again = resolve_lanes<W, B, G>(tg, muls, has, x, state_hash<W>(x), n, probes, err, st) < 0 && has;
      if (again && n + 1 == (uint32_t)tg.rounds()) {
        err |= gx::ERR_TABLE_FULL;
        again = false;
      }
      const uint32_t am = __ballot_sync(FULLMASK, again);
      if (again) {  // (the warp has read its entries: resolve_lanes synchronises it)
        const int at = n_kept + __popc(am & below);
        store_vec<W>(q.kept + at * W, x);
        q.seq[at] = (uint8_t)(n + 1);
      }
      n_kept += __popc(am);
    }
    if (last) break;
    __syncwarp();
  }
}

// Whether the level kernel does so: not with 4-word vectors, where the second way of
// generating spills registers in the loop that the large levels run (3.4e8 states in
// two passes 188 ms, without it 183).
// (The sharing set does, for tables whose levels are small: kernels_for.)
template <int W, bool Share>
constexpr bool kWide = Share || W < 4;

template <int W, int B, int G, bool Share>
__global__ void __launch_bounds__(gx::kBlock, ExpandOcc<W, B, G, Share>::min_ctas) expand_kernel(const gx::ExpandArgs a) {
  constexpr uint32_t kWarps = gx::kBlock / 32;
  extern __shared__ __align__(16) uint32_t sm[];
  // the level being expanded: from the parameters, or (device-driven level
  // loop) from the control block the previous level's advance step wrote.
  // Kept in shared memory, not registers, for the inner loop's sake.
  __shared__ unsigned long long s_range[2];
  const uint32_t nwarps = gridDim.x * kWarps;
  uint32_t unit;  // states a warp takes at a time
  {
    const uint64_t b0 = a.dev_range ? a.ctl->cur_begin : a.cur_begin;
    const uint64_t e0 = a.dev_range ? a.ctl->cur_end : a.cur_end;
    // a level of fewer states than lanes is spread over all warps: its time is
    // the latency of one warp's share, not throughput
    const uint64_t full = 32ull * nwarps;
    unit = e0 - b0 >= full ? 32u : ((uint32_t)(e0 - b0) + nwarps - 1) / nwarps;
    // a fixed full-size grid: CTAs beyond the level's states leave at once
    if ((uint64_t)blockIdx.x * kWarps * unit >= e0 - b0) return;
    if (threadIdx.x == 0) {
      s_range[0] = b0;
      s_range[1] = e0;
    }
  }
  const uint64_t* muls;
  const uint32_t* t = stage_tables(sm, a.muls, a.rounds, a.blob, a.blob_words, a.stage, muls);
  __shared__ uint4 descs[kMaxProcs];
  __syncthreads();
  const NetBlobLayout& L = a.lay;
  const ProcDescs desc = stage_descs(t, L, descs);
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31;
  uint32_t trans = 0;  // per thread and launch: far below 2^32
  uint32_t probes = 0, err = 0;
  __shared__ __align__(16) uint32_t stage_mem[kWarps][kStage * W];
  __shared__ __align__(16) WarpQueues<W> queue_mem[kWarps];
  WarpStage st{stage_mem[threadIdx.x >> 5], 0};
  const ParamTarget tg{a, s_range};
  // (a warp with a few states has no use for the cache of those it has seen)
  WarpCache cache{nullptr, 0, W == 4 && a.cache_key64 ? a.gcache.word_at : nullptr};
  if (a.cache_log2 > 0 && unit == 32) {
    uint32_t* cbase = sm + 2 * kMaxRounds + (a.stage ? a.blob_words : 0);  // 16-byte aligned
    const uint32_t per_warp = (1u << a.cache_log2) * (cache.key_at ? 2 : W);
    cache.base = cbase + (threadIdx.x >> 5) * per_warp;
    cache.mask = (1u << a.cache_log2) - 1u;
    for (uint32_t i = lane; i < per_warp; i += 32) cache.base[i] = 0u;  // 0 is never a stored vector
    __syncwarp();
  }
  const uint64_t own = s_range[0] + (uint64_t)(blockIdx.x * kWarps + (threadIdx.x >> 5)) * unit;
  bool first = true;
  expand_states<W, B, G, kBatch<W>, kWide<W, Share>, Share>(
      tg, muls, t, L, queue_mem[threadIdx.x >> 5], st, probes, err, desc,
      [&](uint64_t& pos, uint32_t& m) {
        // the first states of every warp are fixed by its index, a large level's
        // further ones are claimed
        m = 0;
        if (first) {
          pos = own;
          first = false;
        } else {
          if (unit < 32) return;
          unsigned long long c = 0;
          if (lane == 0) c = atomicAdd(&a.ctl->claim, 32ull);
          pos = s_range[0] + 32ull * nwarps + __shfl_sync(FULLMASK, c, 0);
        }
        if (pos < s_range[1]) m = s_range[1] - pos < unit ? (uint32_t)(s_range[1] - pos) : unit;
      },
      [&](const uint32_t(&v)[W]) {
        if (a.watch && a.count_states) check_watch<W>(a, t, L, v);
      },
      [&](const uint32_t(&v)[W], uint32_t n) {
        // with region passes, the level's states are accounted for in the first pass only
        if (!a.count_states) return;
        trans += n;
        if (n == 0) {
          const uint64_t h = state_digest<W>(t, L, v);
          const unsigned long long di = atomicAdd(&a.ctl->dl_count, 1ull);
          atomicAdd(&a.ctl->dl_sum, (unsigned long long)h);
          atomicXor(&a.ctl->dl_xor, (unsigned long long)h);
          if (di < a.dl_cap) store_vec<W>(a.dl_buf + di * W, v);
        }
      },
      [&](bool on, const uint32_t(&x)[W]) {
        // region passes: a vector whose first bucket lies outside this pass's region is
        // left to the pass of that region (tested before the caches, which may only hold
        // vectors that went to find-or-put).  A vector this warp has already sent to
        // find-or-put needs no second lookup, nor does one that any warp found or
        // inserted moments ago.
        if (a.region_mask && (bucket_of(state_hash<W>(x), muls[0], a.log2nb) & a.region_mask) != a.region_bits)
          on = false;
        const bool known = cache.base && cache.template seen<W>(on, x);
        return on && !known;
      });
  st.flush<W>(tg, err);
  // the CTA's totals, one atomic per counter: at the end of a level every warp
  // finishes at once, and per-warp atomics would queue on two addresses
  __shared__ unsigned long long s_tot[2][kWarps];
  __shared__ uint32_t s_err[kWarps];
  const unsigned long long trans_w = warp_sum((unsigned long long)trans);
  const unsigned long long pr = warp_sum((unsigned long long)probes);
  err = __reduce_or_sync(FULLMASK, err);
  if (lane == 0) {
    s_tot[0][threadIdx.x >> 5] = trans_w;
    s_tot[1][threadIdx.x >> 5] = pr;
    s_err[threadIdx.x >> 5] = err;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    unsigned long long x = 0;
    if (threadIdx.x < 2)
      for (uint32_t w = 0; w < kWarps; ++w) x += s_tot[threadIdx.x][w];
    if (threadIdx.x == 0 && x) atomicAdd(&a.ctl->transitions, x);
    if (threadIdx.x == 1 && x) atomicAdd(&a.ctl->probes, x);
    if (threadIdx.x == 2) {
      uint32_t e = 0;
      for (uint32_t w = 0; w < kWarps; ++w) e |= s_err[w];
      if (e) atomicOr(&a.ctl->error, e);
    }
  }
}


// ---- the device-driven level loop

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// What decides about going on, as the expansion of a level left it.
struct LevelEnd {
  unsigned long long next_end, dl_count, viol_count;
  unsigned int error;
};
__device__ __forceinline__ LevelEnd level_end(const gx::Ctl& c) {
  return LevelEnd{__ldcg(&c.next_end), __ldcg(&c.dl_count), __ldcg(&c.viol_count), __ldcg(&c.error)};
}

// The loop's bookkeeping of the control block, in registers.
struct LoopState {
  unsigned long long cur_begin, cur_end, n_levels, levels_done, explored, t_prev;
  long long first_dl, first_viol;
  unsigned int complete, yielded;
  __device__ __forceinline__ void load(const gx::Ctl& c) {
    cur_begin = c.cur_begin;
    cur_end = c.cur_end;
    n_levels = c.n_levels;
    levels_done = c.levels_done;
    explored = c.explored;
    t_prev = c.t_prev;
    first_dl = c.first_dl;
    first_viol = c.first_viol;
    complete = c.complete;
    yielded = c.yielded;
  }
  __device__ __forceinline__ void store(gx::Ctl& c) const {
    c.cur_begin = cur_begin;
    c.cur_end = cur_end;
    c.n_levels = n_levels;
    c.levels_done = levels_done;
    c.explored = explored;
    c.t_prev = t_prev;
    c.first_dl = first_dl;
    c.first_viol = first_viol;
    c.complete = complete;
    c.yielded = yielded;
  }
  // Level [cur_begin, cur_end) has been expanded: whether there is another one
  // to expand now, which is then [cur_begin, cur_end).
  __device__ __forceinline__ bool move(const gx::LoopArgs& L, const LevelEnd& e) {
    levels_done += 1;
    explored += cur_end - cur_begin;
    if (first_dl < 0 && e.dl_count > 0) first_dl = (long long)n_levels - 1;
    if (first_viol < 0 && e.viol_count > 0) first_viol = (long long)n_levels - 1;
    if (e.next_end > cur_end) n_levels += 1;
    if (e.error) return false;
    if (e.next_end == cur_end) {
      complete = 1;
      return false;
    }
    cur_begin = cur_end;
    cur_end = e.next_end;
    if ((L.stop_dl && e.dl_count > 0) || (L.stop_viol && e.viol_count > 0) ||
        (L.max_levels && levels_done >= L.max_levels))
      return false;
    if (n_levels >= L.cap) {  // arrays full: the host loop continues from here
      yielded = 1;
      return false;
    }
    return true;
  }
  // The same with the level's entries in the arrays.
  __device__ __forceinline__ bool advance(const gx::LoopArgs& L, const LevelEnd& e, unsigned long long probes,
                                          unsigned long long transitions) {
    const unsigned long long k = levels_done, end = cur_end, t = global_ns();
    if (k < L.cap) {
      L.lv_tns[k] = t - t_prev;
      L.lv_probes[k] = probes;
      L.lv_trans[k] = transitions;
    }
    t_prev = t;
    if (e.next_end > end && n_levels < L.cap) L.lv_size[n_levels] = e.next_end - end;
    return move(L, e);
  }
};

// (Not the .aligned forms: those want a warp whose lanes arrive together, and one lane
// keeps the books of a level just before.)
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Levels of at most kSmallLevel states, one after the other in one launch by one
// cluster of CTAs: what such a level costs elsewhere is launches, staging the
// tables and the loop's iteration (13-17 us a level), here two cluster barriers and
// the latency of one or a few states per warp (640-state network: 5-6 us a
// level).  Ends at the first larger level, which the large-level loop takes.
constexpr int kSmallCtas = 8, kSmallThreads = 512;
constexpr uint32_t kSmallWarps = kSmallCtas * kSmallThreads / 32;
constexpr unsigned long long kSmallLevel = 4 * kSmallWarps;

template <int W>
struct __align__(16) SmallQueues {  // of a warp, in dynamic shared memory
  WarpQueues<W, 32> queues;
  uint32_t stage[kStage * W];
};

template <int W, int B, bool Share>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads, 1)
    small_levels_kernel(const gx::ExpandArgs a, const gx::LoopArgs LA) {
  constexpr uint32_t kWarps = kSmallThreads / 32;
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ unsigned long long s_range[2];
  __shared__ uint4 descs[kMaxProcs];
  __shared__ unsigned long long s_tot[2];
  __shared__ uint32_t s_err, s_go;
  const uint64_t* muls;
  const uint32_t* t = stage_tables(sm, a.muls, a.rounds, a.blob, a.blob_words, a.stage, muls);
  __syncthreads();
  const NetBlobLayout& L = a.lay;
  const ProcDescs desc = stage_descs(t, L, descs);
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t gw = blockIdx.x * kWarps + wid;
  SmallQueues<W>& q = reinterpret_cast<SmallQueues<W>*>(sm + 2 * kMaxRounds + (a.stage ? a.blob_words : 0))[wid];
  WarpStage st{q.stage, 0};
  const ParamTarget tg{a, s_range};
  gx::Ctl& c = *a.ctl;
  LoopState ls;  // thread 0 of every CTA; CTA 0's is written back
  bool more = true;
  if (threadIdx.x == 0) {
    ls.load(c);
    s_go = ls.cur_end - ls.cur_begin <= kSmallLevel;
    s_range[0] = ls.cur_begin;
    s_range[1] = ls.cur_end;
    s_tot[0] = s_tot[1] = 0;
    s_err = 0;
  }
  __syncthreads();
  while (s_go) {
    uint32_t trans = 0, probes = 0, err = 0;
    // (at most 4 states a warp)
    const uint32_t unit = ((uint32_t)(s_range[1] - s_range[0]) + kSmallWarps - 1) / kSmallWarps;
    uint64_t own = s_range[0] + (uint64_t)gw * unit;
    expand_states<W, B, 1, 32, true, Share>(
        tg, muls, t, L, q.queues, st, probes, err, desc,
        [&](uint64_t& pos, uint32_t& m) {
          m = own >= s_range[1] ? 0u : s_range[1] - own < unit ? (uint32_t)(s_range[1] - own) : unit;
          pos = own;
          own = s_range[1];
        },
        [&](const uint32_t(&v)[W]) {
          if (a.watch) check_watch<W>(a, t, L, v);
        },
        [&](const uint32_t(&v)[W], uint32_t n) {
          trans += n;
          if (n == 0) {
            const uint64_t h = state_digest<W>(t, L, v);
            const unsigned long long di = atomicAdd(&c.dl_count, 1ull);
            atomicAdd(&c.dl_sum, (unsigned long long)h);
            atomicXor(&c.dl_xor, (unsigned long long)h);
            if (di < a.dl_cap) store_vec<W>(a.dl_buf + di * W, v);
          }
        },
        [](bool on, const uint32_t(&)[W]) { return on; });
    st.flush<W>(tg, err);
    const unsigned long long tr = warp_sum((unsigned long long)trans), pr = warp_sum((unsigned long long)probes);
    err = __reduce_or_sync(FULLMASK, err);
    if (lane == 0) {
      if (tr) atomicAdd(&s_tot[0], tr);
      if (pr) atomicAdd(&s_tot[1], pr);
      if (err) atomicOr(&s_err, err);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (s_tot[0]) atomicAdd(&c.transitions, s_tot[0]);
      if (s_tot[1]) atomicAdd(&c.probes, s_tot[1]);
      if (s_err) atomicOr(&c.error, s_err);
      s_tot[0] = s_tot[1] = 0;
      s_err = 0;
    }
    cluster_sync();  // the level is complete
    if (threadIdx.x == 0) {
      const LevelEnd e = level_end(c);
      if (blockIdx.x == 0) more = ls.advance(LA, e, __ldcg(&c.probes), __ldcg(&c.transitions));
      else more = ls.move(LA, e);
      s_range[0] = ls.cur_begin;
      s_range[1] = ls.cur_end;
      s_go = more && ls.cur_end - ls.cur_begin <= kSmallLevel;
    }
    cluster_sync();  // every CTA has read what the next level's expansion changes
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ls.store(c);
    c.claim = 0;
    c.small_launches += 1;
    cudaGraphSetConditional(LA.cond, more ? 1u : 0u);
    cudaGraphSetConditional(LA.cond_big, more ? 1u : 0u);
  }
}

// ---- partitioned expansion (see PartArgs)

// Exclusive scan of one value per thread over the block (blockDim.x == kBlock).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t& total, uint32_t* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULLMASK, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) scratch[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    uint32_t w = lane < (gx::kBlock / 32) ? scratch[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULLMASK, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < (gx::kBlock / 32)) scratch[lane] = wi - w;  // exclusive warp offsets
    if (lane == (gx::kBlock / 32) - 1) scratch[gx::kBlock / 32] = wi;
  }
  __syncthreads();
  const uint32_t r = scratch[wid] + inc - x;
  total = scratch[gx::kBlock / 32];
  __syncthreads();
  return r;
}

__device__ __forceinline__ void part_range(const gx::ExpandArgs& a, const gx::PartArgs& pa, int b,
                                           uint64_t& lo, uint64_t& hi) {
  lo = a.cur_begin + (uint64_t)b * pa.range;
  hi = lo + pa.range;
  if (hi > a.cur_end) hi = a.cur_end;
  if (lo > hi) lo = hi;
}

// Pass 1: successors per (CTA, slice).  No other side effect, so a level may still
// fall back to the direct kernel after it.
template <int W>
__global__ void __launch_bounds__(gx::kBlock) part_count_kernel(const gx::ExpandArgs a, const gx::PartArgs pa) {
  extern __shared__ __align__(16) uint32_t sm[];
  const uint64_t* muls;
  const uint32_t* t = stage_tables(sm, a.muls, 1, a.blob, a.blob_words, a.stage, muls);
  uint32_t* hist = sm + 2 * kMaxRounds + (a.stage ? a.blob_words : 0);
  __shared__ uint32_t scan_scratch[gx::kBlock / 32 + 1];
  const int P = 1 << pa.logp;
  for (int q = threadIdx.x; q < P; q += blockDim.x) hist[q] = 0;
  __syncthreads();
  const NetBlobLayout& L = a.lay;
  const uint64_t mul0 = muls[0];
  const int shift = 64 - pa.logp;
  uint64_t lo, hi;
  part_range(a, pa, blockIdx.x, lo, hi);
  for (uint64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    uint32_t v[W];
    load_vec<W>(a.frontier + (i & a.fmask) * W, v);
    const uint32_t cnt = count_succ<W>(t, L, v);
    SuccIter it;
    it.init();
    for (uint32_t k = 0; k < cnt; ++k) {
      uint32_t s[W];
      next_succ<W>(it, t, L, v, s);
      atomicAdd(&hist[(uint32_t)((state_hash<W>(s) * mul0) >> shift)], 1u);
    }
  }
  __syncthreads();
  uint32_t mine = 0;
  for (int q = threadIdx.x; q < P; q += blockDim.x) {
    pa.hist[(uint64_t)blockIdx.x * P + q] = hist[q];
    mine += hist[q];
  }
  uint32_t total;
  block_exclusive_scan(mine, total, scan_scratch);
  if (threadIdx.x == 0) pa.tot[blockIdx.x] = total;
}

// Pass 2: per slice q (one CTA each), exclusive scan over the batch's CTAs.
// (A template only so that every translation unit may include this header.)
template <int Unused>
__global__ void __launch_bounds__(gx::kBlock) part_scan_kernel(const gx::PartArgs pa) {
  __shared__ uint32_t scan_scratch[gx::kBlock / 32 + 1];
  const int q = blockIdx.x;
  const int P = 1 << pa.logp;
  uint32_t running = 0;
  for (int base = pa.b0; base < pa.b1; base += blockDim.x) {
    const int b = base + threadIdx.x;
    const uint32_t x = b < pa.b1 ? pa.hist[(uint64_t)b * P + q] : 0u;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan(x, total, scan_scratch);
    if (b < pa.b1) pa.off[(uint64_t)b * P + q] = running + ex;
    running += total;
  }
  if (threadIdx.x == 0) pa.ptot[q] = running;
}

// Pass 3: regenerate the successors and write them slice-major; transitions and
// deadlocks of the batch's frontier states are accounted here.
template <int W>
__global__ void __launch_bounds__(gx::kBlock) part_scatter_kernel(const gx::ExpandArgs a, const gx::PartArgs pa) {
  extern __shared__ __align__(16) uint32_t sm[];
  const uint64_t* muls;
  const uint32_t* t = stage_tables(sm, a.muls, 1, a.blob, a.blob_words, a.stage, muls);
  uint32_t* cur = sm + 2 * kMaxRounds + (a.stage ? a.blob_words : 0);
  __shared__ uint32_t scan_scratch[gx::kBlock / 32 + 1];
  const int P = 1 << pa.logp;
  const int b = pa.b0 + blockIdx.x;
  // cursor of slice q = (successors of the batch in slices < q) + (of CTAs before b in slice q)
  uint32_t running = 0;
  __syncthreads();
  for (int base = 0; base < P; base += blockDim.x) {
    const int q = base + threadIdx.x;
    const uint32_t x = q < P ? pa.ptot[q] : 0u;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan(x, total, scan_scratch);
    if (q < P) cur[q] = running + ex + pa.off[(uint64_t)b * P + q];
    running += total;
  }
  __syncthreads();
  const NetBlobLayout& L = a.lay;
  const uint64_t mul0 = muls[0];
  const int shift = 64 - pa.logp;
  uint64_t lo, hi;
  part_range(a, pa, b, lo, hi);
  unsigned long long trans = 0;
  for (uint64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    uint32_t v[W];
    load_vec<W>(a.frontier + (i & a.fmask) * W, v);
    const uint32_t cnt = count_succ<W>(t, L, v);
    trans += cnt;
    if (cnt == 0) {
      const uint64_t h = state_digest<W>(t, L, v);
      const unsigned long long di = atomicAdd(&a.ctl->dl_count, 1ull);
      atomicAdd(&a.ctl->dl_sum, (unsigned long long)h);
      atomicXor(&a.ctl->dl_xor, (unsigned long long)h);
      if (di < a.dl_cap) store_vec<W>(a.dl_buf + di * W, v);
    }
    if (a.watch) check_watch<W>(a, t, L, v);
    SuccIter it;
    it.init();
    for (uint32_t k = 0; k < cnt; ++k) {
      uint32_t s[W];
      next_succ<W>(it, t, L, v, s);
      const uint32_t q = (uint32_t)((state_hash<W>(s) * mul0) >> shift);
      const uint32_t pos = atomicAdd(&cur[q], 1u);
      store_vec<W>(pa.succ + (uint64_t)pos * W, s);
    }
  }
  trans = warp_sum(trans);
  if ((threadIdx.x & 31) == 0 && trans) atomicAdd(&a.ctl->transitions, trans);
}

// Pass 4: find-or-put of the buffered successors in buffer order (slice by slice).
template <int W, int B, int G>
__global__ void __launch_bounds__(gx::kBlock) part_probe_kernel(const gx::ExpandArgs a, const uint32_t* succ,
                                                                uint64_t n) {
  __shared__ uint64_t muls[kMaxRounds];
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  uint32_t probes = 0, err = 0;
  __shared__ __align__(16) uint32_t stage_mem[gx::kBlock / 32][kStage * W];
  WarpStage st{stage_mem[threadIdx.x >> 5], 0};
  __shared__ unsigned long long s_range[2];
  if (threadIdx.x == 0) {
    s_range[0] = a.cur_begin;
    s_range[1] = a.cur_end;
  }
  __syncthreads();
  const ParamTarget tg{a, s_range};
  while (true) {
    unsigned long long chunk = 0;
    if (lane == 0) chunk = atomicAdd(&a.ctl->claim, 32ull);
    chunk = __shfl_sync(FULLMASK, chunk, 0);
    if (chunk >= n) break;
    const uint64_t idx = chunk + lane;
    bool on = idx < n;
    uint32_t x[W];
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = 0;
    if (on) load_vec<W>(succ + idx * W, x);
    if (on && a.gcache.base) {  // the filter that the level kernel applies as it generates
      const SeenEntry e = seen_entry<W>(a.gcache, x);
      on = e.content == 0 || seen_get(a.gcache, e.index) != e.content;
    }
    const uint64_t h = state_hash<W>(x);
    for (uint32_t k = 0; __any_sync(FULLMASK, on); ++k) {
      if (k == (uint32_t)a.rounds) {
        if (on) err |= gx::ERR_TABLE_FULL;
        break;
      }
      on = resolve_lanes<W, B, G>(tg, muls, on, x, h, k, probes, err, st) < 0 && on;
    }
  }
  st.flush<W>(tg, err);
  const unsigned long long pr = warp_sum((unsigned long long)probes);
  err = __reduce_or_sync(FULLMASK, err);
  if (lane == 0) {
    if (pr) atomicAdd(&a.ctl->probes, pr);
    if (err) atomicOr(&a.ctl->error, err);
  }
}

template <int W, int B, int G>
__global__ void init_kernel(const gx::InitArgs a) {
  __shared__ uint64_t muls[kMaxRounds];
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  __syncthreads();
  if (threadIdx.x != 0) return;
  uint32_t v[W];
#pragma unroll
  for (int w = 0; w < W; ++w) v[w] = a.vec[w];
  uint32_t probes = 0;
  if (find_or_put_state<W, B>(a.table, a.log2nb, a.rounds, muls, v, probes) == FOP_INSERTED) {
    store_vec<W>(a.frontier, v);
    a.ctl->next_end = 1ull;
  } else {
    a.ctl->error |= gx::ERR_TABLE_FULL;
  }
}

// Sec. 5.1: key i of the sequence has result r.
__device__ __forceinline__ void fop_count(const gx::FopArgs& a, uint64_t i, int r, unsigned long long& ins,
                                          unsigned long long& fnd, unsigned long long& fail) {
  if (a.result) a.result[i] = (uint8_t)(r == FOP_INSERTED ? 1 : (r == FOP_FOUND ? 0 : 2));
  ins += r == FOP_INSERTED;
  fnd += r == FOP_FOUND;
  fail += r == FOP_FULL;
}

// The lanes of a warp take their own keys and read their buckets together
// (bucket_step_lanes), so a lane that is done takes its next key at once.  (With a group of lanes per key, which voted on every
// bucket, the same keys took 10.5 ms with a lane per slot of 8-word buckets, 22.6 of
// 32-word ones; now 4.8 and 5.6.)
template <int W, int B, int G>
__device__ __forceinline__ void fop_groups(const gx::FopArgs& a, const uint64_t* muls, unsigned long long& ins,
                                           unsigned long long& fnd, unsigned long long& fail) {
  const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  // the warp's keys: consecutive ones, of which 64 are held (base.., pos of them taken)
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
  const uint64_t len = (a.n + warps - 1) / warps;
  uint64_t base = ((uint64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5)) * len;
  const uint64_t end = base + len < a.n ? base + len : a.n;
  uint32_t pos = 0, cur[W], nxt[W];
  auto fetch = [&](uint64_t i, uint32_t(&x)[W]) {
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = i < end ? a.keys[i * W + w] : 0u;
  };
  fetch(base + lane, cur);
  fetch(base + 32 + lane, nxt);
  bool has = false;
  uint32_t v[W], k = 0;
  uint64_t h = 0, at = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) v[w] = 0;
  while (true) {
    const uint32_t need = __ballot_sync(FULLMASK, !has);
    if (need != 0 && base + pos < end) {
      const uint32_t src = pos + __popc(need & below);
      uint32_t x[W];
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t c = __shfl_sync(FULLMASK, cur[w], src & 31), d = __shfl_sync(FULLMASK, nxt[w], src & 31);
        x[w] = src < 32 ? c : d;
      }
      if (!has && base + src < end) {
#pragma unroll
        for (int w = 0; w < W; ++w) v[w] = x[w] | kTag;
        h = vec_hash<W>(v);
        at = base + src;
        k = 0;
        has = true;
      }
      pos += __popc(need);
      if (pos >= 32) {
        pos -= 32;
        base += 32;
#pragma unroll
        for (int w = 0; w < W; ++w) cur[w] = nxt[w];
        fetch(base + 32 + lane, nxt);
      }
    }
    if (!__any_sync(FULLMASK, has)) break;
    const int r = bucket_step_lanes<W, B, G>(a.table, has, seq_bucket<B>(h, k, muls, a.log2nb), v);
    if (has && (r >= 0 || ++k == (uint32_t)a.rounds)) {
      fop_count(a, at, r >= 0 ? r : FOP_FULL, ins, fnd, fail);
      has = false;
    }
  }
}

// A key per lane (G == 1), or per group of lanes where a lane's part of the bucket is 64 bytes
// or more (32-word buckets, 2 lanes: 25-50 G keys/s by duplication, 23-35 with fop_groups),
// key after key.  Bound by random 128-byte lines read and written back; a lane that took its
// next key while others of its warp read further buckets made it no faster (1.5e8 keys, 1e8
// of them new, 8-word buckets, G = 1: 4.75 ms, with that 4.92).  The loop stands here and
// not in a function: as one it took 46 registers for <2, 32, 2> instead of 40, a CTA an SM
// less (2e7 keys, each five times: 0.57 ms instead of 0.54).
template <int W, int B, int G>
__global__ void __launch_bounds__(gx::kBlock) fop_kernel(const gx::FopArgs a) {
  __shared__ uint64_t muls[kMaxRounds];
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  unsigned long long ins = 0, fnd = 0, fail = 0;
  if constexpr (G == 1 || B / G >= 16) {
    const Group<G> g;
    const uint64_t groups = (uint64_t)gridDim.x * blockDim.x / G;
    uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    uint32_t probes = 0;
    // the loop bound is uniform per warp: all groups of a warp leave together
    const uint64_t warp_first = ((uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) / G;
    for (uint64_t wi = warp_first; wi < a.n; wi += groups, i += groups) {
      if (i < a.n) {
        uint32_t v[W];
#pragma unroll
        for (int w = 0; w < W; ++w) v[w] = a.keys[i * W + w] | kTag;
        const int r = find_or_put<W, B, G>(a.table, a.log2nb, a.rounds, muls, v, g, probes);
        if (g.glane == 0) fop_count(a, i, r, ins, fnd, fail);
      }
    }
  } else {
    fop_groups<W, B, G>(a, muls, ins, fnd, fail);
  }
  ins = warp_sum(ins);
  fnd = warp_sum(fnd);
  fail = warp_sum(fail);
  if (lane == 0) {
    if (ins) atomicAdd(&a.counters[0], ins);
    if (fnd) atomicAdd(&a.counters[1], fnd);
    if (fail) atomicAdd(&a.counters[2], fail);
  }
}

}  // namespace gxd

namespace gx {

template <int W, int B, int G, bool Share>
cudaError_t launch_expand(const ExpandArgs& a, int grid, size_t smem, int carveout, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  at[0].val.sharedMemCarveout = (unsigned)carveout;
  cfg.attrs = at;
  cfg.numAttrs = carveout >= 0 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gxd::expand_kernel<W, B, G, Share>, a);
}
template <int W, int B, int G>
cudaError_t launch_init(const InitArgs& a, cudaStream_t st) {
  gxd::init_kernel<W, B, G><<<1, 32, 0, st>>>(a);
  return cudaGetLastError();
}
template <int W, int B, int G>
cudaError_t launch_fop(const FopArgs& a, int grid, cudaStream_t st) {
  gxd::fop_kernel<W, B, G><<<grid, kBlock, 0, st>>>(a);
  return cudaGetLastError();
}

template <int W>
cudaError_t launch_part_count(const ExpandArgs& a, const PartArgs& p, size_t smem, cudaStream_t st) {
  gxd::part_count_kernel<W><<<p.nb, kBlock, smem, st>>>(a, p);
  return cudaGetLastError();
}
inline cudaError_t launch_part_scan(const PartArgs& p, cudaStream_t st) {
  gxd::part_scan_kernel<0><<<1 << p.logp, kBlock, 0, st>>>(p);
  return cudaGetLastError();
}
template <int W>
cudaError_t launch_part_scatter(const ExpandArgs& a, const PartArgs& p, size_t smem, cudaStream_t st) {
  gxd::part_scatter_kernel<W><<<p.b1 - p.b0, kBlock, smem, st>>>(a, p);
  return cudaGetLastError();
}
template <int W, int B, int G>
cudaError_t launch_part_probe(const ExpandArgs& a, const uint32_t* succ, uint64_t n, int grid, cudaStream_t st) {
  gxd::part_probe_kernel<W, B, G><<<grid, kBlock, 0, st>>>(a, succ, n);
  return cudaGetLastError();
}

template <int W, int B, int G, bool Share = false>
const KernelSet* kernel_set() {
  const KernelSet* sharing = nullptr;
  if constexpr (!Share) sharing = kernel_set<W, B, G, true>();
  static const KernelSet ks{&launch_expand<W, B, G, Share>,
                            &launch_part_count<W>,
                            &launch_part_scan,
                            &launch_part_scatter<W>,
                            &launch_part_probe<W, B, G>,
                            &launch_init<W, B, G>,
                            &launch_fop<W, B, G>,
                            reinterpret_cast<const void*>(&gxd::expand_kernel<W, B, G, Share>),
                            reinterpret_cast<const void*>(&gxd::fop_kernel<W, B, G>),
                            reinterpret_cast<const void*>(&gxd::part_count_kernel<W>),
                            reinterpret_cast<const void*>(&gxd::part_scatter_kernel<W>),
                            reinterpret_cast<const void*>(&gxd::part_probe_kernel<W, B, G>),
                            reinterpret_cast<const void*>(&gxd::init_kernel<W, B, G>),
                            reinterpret_cast<const void*>(&gxd::small_levels_kernel<W, B, Share>),
                            sizeof(gxd::SmallQueues<W>) * (gxd::kSmallThreads / 32),
                            sharing};
  return &ks;
}

}  // namespace gx

// Dispatch helper: G must be a power of two dividing B / W.
#define GX_CASE(W, B, G) \
  if (b == B && g == G) return gx::kernel_set<W, B, G>();
