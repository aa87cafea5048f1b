// Batched exploration: many independent networks in one persistent launch (no
// counterpart in the paper, which explores one network at a time; the
// per-network work is the level expansion of Sec. 3 with the find-or-put of
// Sec. 4.1).
//
//   memset(all tables) -> init (initial vector of every network) -> expand
//
// Levels end network by network, not all together: a level's states are taken
// in claims by any warp, the warp that finishes a level's last claim opens the
// next one, and warps move on to another network meanwhile.  Nothing waits for
// a network but its own next level.  (One launch per level of all networks, on
// a device-side loop, left 85 of the 99 levels of the 256-network workload
// with less than one claim per warp: 3.1 of 9.8 ms.)
//
// Workspace: per-network descriptors | claims | counter | network blobs |
//            level arrays | frontier rings | tables (contiguous)

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "gx_kernels.cuh"

namespace gx {

struct BNet {
  const uint32_t* blob;
  NetBlobLayout lay;
  uint32_t* table;
  int log2nb;
  uint32_t* frontier;
  uint64_t fmask;
  // the level being expanded: its states, states per claim, claims, claims done
  unsigned long long cur_begin, cur_end, next_end;
  unsigned int unit, chunks, done;
  unsigned long long transitions, dl_count, dl_sum, dl_xor, probes;
  unsigned int error, active, n_levels;
  int first_dl;
  uint32_t init_vec[4];
};

struct BatchArgs {
  BNet* nets;  // largest table first
  int n;
  int rounds;
  uint32_t chunk;             // states per claim, at most
  uint32_t levels_cap;
  unsigned long long* levels; // level sizes: entry [level * n + network]
  // per network: claims taken of its level, and in the upper half how many it has
  // (0: finished, and then at least kFinished are taken)
  unsigned long long* claims;
  unsigned int* active;       // [0] networks that are not finished, [1] levels that ended
  unsigned long long give_up_ns;  // a warp's longest wait without either changing
  uint32_t warps;             // of the expansion's grid
  uint32_t wide;              // a level with at most this many states per warp that falls to
                              // its network is claimed state by state
  Muls muls;
};

constexpr unsigned long long kFinished = 0x80000000ull;
constexpr uint64_t kGiveUpNs = 20ull * 1000 * 1000 * 1000;  // (gx_batch_set_wait_limit)
constexpr unsigned int ERR_LEVELS = 8u;  // a network needed more levels than levels_cap

}  // namespace gx

namespace gxd {

using gx::BatchArgs;
using gx::BNet;

template <int W, int B, int G>
__global__ void __launch_bounds__(gx::kBlock) batch_init_kernel(const BatchArgs a) {
  __shared__ uint64_t muls[kMaxRounds];
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) muls[i] = a.muls.m[i];
  __syncthreads();
  const int net = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (net >= a.n || (threadIdx.x & 31) != 0) return;
  BNet& b = a.nets[net];
  uint32_t v[W];
#pragma unroll
  for (int w = 0; w < W; ++w) v[w] = b.init_vec[w];
  uint32_t probes = 0;
  const int r = find_or_put_state<W, B>(b.table, b.log2nb, a.rounds, muls, v, probes);
  if (r == FOP_INSERTED) store_vec<W>(b.frontier, v);
  b.cur_begin = 0;
  b.cur_end = 1;
  b.next_end = 1;
  b.unit = b.chunks = 1;
  b.done = 0;
  b.transitions = b.dl_count = b.dl_sum = b.dl_xor = 0;
  b.probes = probes;
  b.error = r == FOP_INSERTED ? 0u : gx::ERR_TABLE_FULL;
  b.active = r == FOP_INSERTED ? 1u : 0u;
  b.first_dl = -1;
  b.n_levels = 1;
  a.levels[net] = 1;
  a.claims[net] = r == FOP_INSERTED ? 1ull << 32 : gx::kFinished;
  if (r == FOP_INSERTED) atomicAdd(a.active, 1u);
}

// Network i has finished the level it was expanding: record the next one and
// open it, or finish the network (false).  One lane, after the level's last claim.
__device__ __forceinline__ bool batch_next_level(const BatchArgs& a, int i) {
  BNet& b = a.nets[i];
  using gx::kFinished;
  atomicAdd(a.active + 1, 1u);
  const unsigned long long end = __ldcg(&b.cur_end), next = __ldcg(&b.next_end), fresh = next - end;
  unsigned int err = __ldcg(&b.error), levels = __ldcg(&b.n_levels);
  if (__ldcg(&b.first_dl) < 0 && __ldcg(&b.dl_count) > 0) b.first_dl = (int)levels - 1;
  if (fresh > 0) {
    if (levels < a.levels_cap) {
      a.levels[(uint64_t)levels * a.n + i] = fresh;
    } else {
      err |= gx::ERR_LEVELS;
      b.error = err;
    }
    b.n_levels = levels + 1;
  }
  if (err || fresh == 0) {
    b.active = 0;
    atomicSub(a.active, 1u);
    __threadfence();
    atomicExch(a.claims + i, gx::kFinished);
    return false;
  }
  // a network's share of the warps, were all networks at work: a level that gives each
  // of them less than a full claim is taken in smaller ones
  const unsigned long long act = __ldcg(a.active), share = a.warps > act ? a.warps / act : 1;
  unsigned long long unit = (fresh + fresh / 4 + share - 1) / share;
  if (fresh <= a.wide * share) unit = 1;
  if (unit > a.chunk || a.wide == 0) unit = a.chunk;
  while ((fresh + unit - 1) / unit >= kFinished) unit *= 2;  // (the halves of a claims word hold them)
  const unsigned long long chunks = (fresh + unit - 1) / unit;
  b.cur_begin = end;
  b.cur_end = next;
  b.unit = (unsigned int)unit;
  b.chunks = (unsigned int)chunks;
  b.done = 0;
  __threadfence();
  atomicExch(a.claims + i, chunks << 32);
  return true;
}

// A claim of any network that has one left, of network `first` before others if that is
// one (the warp has just opened its next level).  False: all networks are finished, or this
// warp has waited give_up_ns in which no level ended and no claim was taken before its eyes.
// That is no error: the claims being worked on (a claim may hold up to 2^32 successors a
// state) are finished by their warps, and the one that ends a level goes on with the next.
// The host reports a network that was left unfinished, which only a lost claim can cause.
// A warp begins the search at a place of its own, so that the networks are worked on side by
// side: the claims words, queue ends and table lines of one network take only so many
// accesses at a time (256 networks: 9.2 ms; all warps on the first open network 12.8, on the
// first 8 of them 11.2, on 32 10.6).
// For the same reason warps that find nothing must not crowd the words of those that work:
// they look at kLook groups of 32 networks, then pause, twice as long each time (from 128 ns
// to 2 us for each of up to 8 unfinished networks), and a claim they got halves the pause.
// Without that -- all groups, pauses of 2 us at most, none after a claim taken by others --
// 32 networks of 640 states took 1.35 ms instead of 0.40, 32 of 118,098 5.3 instead of 2.15,
// 256 of the workload 8.5 instead of 8.3.  (Pauses up to 8, 16, 32 us for any number of
// networks: one network 1.6, 1.8, 2.0 ms instead of 1.39; looking at 1, 4 or 8 groups: the
// same within 5 %.)
struct Search {
  int base;        // networks below it are finished
  uint32_t place;  // the group of 32 networks to look at next
  uint32_t nap;    // ns
};
constexpr int kLook = 2;
constexpr uint32_t kShortNap = 128, kLongNap = 2048;
__device__ __forceinline__ unsigned long long batch_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool batch_claim(const BatchArgs& a, uint32_t warp, Search& at, int first, int& net,
                                            uint32_t& c) {
  const int lane = threadIdx.x & 31;
  unsigned long long since = 0;
  uint32_t ended = 0;  // levels, at the last look
  while (true) {
    int found = first;
    first = -1;
    const int span = (a.n - at.base + 31) / 32;
    int look = kLook;
    for (int k = 0; found < 0 && look > 0 && k < span; ++k) {
      const int w0 = at.base + 32 * (int)(at.place++ % span);
      const unsigned long long x = w0 + lane < a.n ? __ldcg(a.claims + w0 + lane) : gx::kFinished;
      if (__all_sync(FULLMASK, (x >> 32) == 0)) {
        if (w0 != at.base) continue;
        at.base += 32;
        break;
      }
      --look;
      const uint32_t open = __ballot_sync(FULLMASK, (uint32_t)x < (uint32_t)(x >> 32));
      if (open) found = w0 + (int)__fns(open, 0, warp % __popc(open) + 1);
    }
    if (found >= 0) {
      unsigned long long x = 0;
      if (lane == 0) x = atomicAdd(a.claims + found, 1ull);
      x = __shfl_sync(FULLMASK, x, 0);
      if ((uint32_t)x < (uint32_t)(x >> 32)) {
        net = found;
        c = (uint32_t)x;
        at.place = warp / 32;
        at.nap = at.nap > 2 * kShortNap ? at.nap / 2 : kShortNap;
        return true;
      }
      since = 0;  // taken by others
    }
    const unsigned long long state = __shfl_sync(FULLMASK, __ldcg(reinterpret_cast<const unsigned long long*>(a.active)), 0);
    const uint32_t active = (uint32_t)state;
    if (active == 0 || at.base >= a.n) return false;
    const unsigned long long now = __shfl_sync(FULLMASK, batch_now(), 0);
    if (since == 0 || ended != (uint32_t)(state >> 32)) {
      since = now;
      ended = (uint32_t)(state >> 32);
    }
    if (now - since > a.give_up_ns) return false;
    __nanosleep(at.nap);
    if (at.nap < kLongNap * (active < 8 ? active : 8)) at.nap *= 2;
  }
}

// Per-warp cache of seen vectors in the batched kernel (1- and 2-word slots).
// Networks have separate tables, so a hit is only valid for the network whose
// vectors filled the cache: a warp clears its cache whenever it moves to a
// chunk of another network.
constexpr int kBatchCacheLog2 = 8;

// The network a warp is working on, staged in shared memory when the warp
// moves to it, so that its layout and table pointers take no registers in the
// inner loop, with the level it is working on.
struct WarpNet {
  NetBlobLayout lay;
  uint32_t* table;
  unsigned long long* next_end;
  uint32_t* frontier;
  uint64_t fmask, cur_begin, cur_end;
  int log2nb;
  uint32_t unit, chunks;
};

struct SmemTarget {
  const WarpNet* w;
  int nrounds;
  __device__ __forceinline__ uint32_t* table() const { return w->table; }
  __device__ __forceinline__ int log2nb() const { return w->log2nb; }
  __device__ __forceinline__ int rounds() const { return nrounds; }
  __device__ __forceinline__ unsigned long long* next_end() const { return w->next_end; }
  __device__ __forceinline__ uint32_t* frontier() const { return w->frontier; }
  __device__ __forceinline__ uint64_t fmask() const { return w->fmask; }
  __device__ __forceinline__ uint64_t begin() const { return w->cur_begin; }
  __device__ __forceinline__ gx::SeenCache gcache() const { return gx::SeenCache{}; }
};

// The batched kernel keeps a network index and claim bounds besides the
// single-network kernel's state: one CTA per SM fewer (at most 4) keeps its
// common instantiations free of spills (256 networks: 9.55 ms with 4, 10.0 with 5,
// 10.4 with 3).
template <int W, int B, int G>
struct BatchOcc {
  static constexpr int min_ctas = ExpandOcc<W, B, G>::min_ctas < 4 ? ExpandOcc<W, B, G>::min_ctas : 4;
};

// Dynamic shared memory of the batched kernel, per warp: queues, staging, the
// cache of seen vectors, the network and descriptors of its edge classes.
template <int W>
struct __align__(16) BatchSmem {
  static constexpr int kWarps = gx::kBlock / 32;
  static constexpr int kCache = W <= 2 ? (1 << kBatchCacheLog2) * W : 4;
  WarpQueues<W, 32> queues[kWarps];
  uint32_t stage[kWarps][kStage * W];
  uint32_t cache[kWarps][kCache];
  uint4 descs[kWarps][32];  // of the first edge classes, one per lane to fetch
  WarpNet net[kWarps];
  unsigned long long muls[kMaxRounds];
};

template <int W, int B, int G, bool Share>
__global__ void __launch_bounds__(gx::kBlock, BatchOcc<W, B, G>::min_ctas) batch_expand_kernel(const BatchArgs a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  BatchSmem<W>& S = *reinterpret_cast<BatchSmem<W>*>(bsm);
  for (int i = threadIdx.x; i < a.rounds; i += blockDim.x) S.muls[i] = a.muls.m[i];
  __syncthreads();
  const uint64_t* muls = reinterpret_cast<const uint64_t*>(S.muls);
  const int wid = threadIdx.x >> 5;
  const uint32_t lane = threadIdx.x & 31;
  WarpNet& wn = S.net[wid];
  uint4* descs = S.descs[wid];
  WarpStage st{S.stage[wid], 0};
  WarpCache cache{W <= 2 ? S.cache[wid] : nullptr, (1u << kBatchCacheLog2) - 1u, nullptr};
  const SmemTarget tg{&wn, a.rounds};
  const uint32_t* t = nullptr;
  const uint32_t warp = blockIdx.x * (gx::kBlock / 32) + wid;
  Search at{0, warp / 32, kShortNap};
  int net = -1, first = -1;
  while (true) {
    int at_net;
    uint32_t c;
    if (!batch_claim(a, warp, at, first, at_net, c)) break;
    BNet& b = a.nets[at_net];
    if (at_net != net) {
      // stage the network; the cache holds one network's vectors at a time
      net = at_net;
      t = b.blob;
      if (lane == 0) {
        wn.lay = b.lay;
        wn.table = b.table;
        wn.next_end = &b.next_end;
        wn.frontier = b.frontier;
        wn.fmask = b.fmask;
        wn.log2nb = b.log2nb;
      }
      if (W <= 2)
        for (uint32_t i = lane; i < (uint32_t)BatchSmem<W>::kCache; i += 32) S.cache[wid][i] = 0u;
      __syncwarp();
      if (lane < wn.lay.n_classes) descs[lane] = class_desc(t, wn.lay, lane);
    }
    // the level (it cannot end before this claim is done)
    __threadfence();
    if (lane == 0) {
      wn.cur_begin = __ldcg(&b.cur_begin);
      wn.cur_end = __ldcg(&b.cur_end);
      wn.unit = __ldcg(&b.unit);
      wn.chunks = __ldcg(&b.chunks);
    }
    __syncwarp();
    const NetBlobLayout& L = wn.lay;
    uint32_t probes = 0, err = 0;
    unsigned long long trans = 0;
    uint64_t pos = 0, end = 0;  // what is left of the claim
    bool held = true;           // c is a claim that has not been started
    uint32_t taken = 1;
    expand_states<W, B, G, 32, true, Share>(
        tg, muls, t, L, S.queues[wid], st, probes, err,
        ClassDescs{descs, L.n_classes < 32u ? L.n_classes : 32u},
        [&](uint64_t& from, uint32_t& m) {
          m = 0;
          if (pos == end) {
            if (!held) {
              if (lane == 0) {
                c = (uint32_t)__ldcg(a.claims + net);
                if (c < wn.chunks) c = (uint32_t)atomicAdd(a.claims + net, 1ull);
              }
              c = __shfl_sync(FULLMASK, c, 0);
              if (c >= wn.chunks) return;
              ++taken;
            }
            pos = wn.cur_begin + (uint64_t)c * wn.unit;
            end = pos + wn.unit < wn.cur_end ? pos + wn.unit : wn.cur_end;
            held = false;
          }
          from = pos;
          m = end - pos < 32 ? (uint32_t)(end - pos) : 32u;
          pos += m;
        },
        [](const uint32_t(&)[W]) {},
        [&](const uint32_t(&v)[W], uint32_t n) {
          trans += n;
          if (n == 0) {
            const uint64_t h = state_digest<W>(t, L, v);
            atomicAdd(&b.dl_count, 1ull);
            atomicAdd(&b.dl_sum, (unsigned long long)h);
            atomicXor(&b.dl_xor, (unsigned long long)h);
          }
        },
        [&](bool on, const uint32_t(&x)[W]) {
          const bool known = cache.base && cache.template seen<W>(on, x);
          return on && !known;
        });
    st.flush<W>(tg, err);
    const unsigned long long tr = warp_sum(trans);
    const unsigned long long pr = warp_sum((unsigned long long)probes);
    err = __reduce_or_sync(FULLMASK, err);
    if (lane == 0) {
      if (tr) atomicAdd(&b.transitions, tr);
      if (pr) atomicAdd(&b.probes, pr);
      if (err) atomicOr(&b.error, err);
    }
    // (the warp's last use of the level: its states, counts and new states come before)
    __threadfence();  // before the level can be seen as done
    __syncwarp();
    bool opened = false;
    if (lane == 0 && atomicAdd(&b.done, taken) + taken == wn.chunks) {
      __threadfence();
      opened = batch_next_level(a, net);
    }
    first = __any_sync(FULLMASK, opened) ? net : -1;
  }
}

}  // namespace gxd

namespace gx {
namespace {

struct BatchKernels {
  const void* init;
  const void* expand;
  size_t smem;  // dynamic shared memory of expand
};

template <int W, int B, int G>
BatchKernels batch_kernels(bool share) {
  return BatchKernels{reinterpret_cast<const void*>(&gxd::batch_init_kernel<W, B, G>),
                      share ? reinterpret_cast<const void*>(&gxd::batch_expand_kernel<W, B, G, true>)
                            : reinterpret_cast<const void*>(&gxd::batch_expand_kernel<W, B, G, false>),
                      sizeof(gxd::BatchSmem<W>)};
}

// (B, G) pairs built for batches; the autotuner picks among them.
const int kCands[][2] = {{4, 1}, {8, 1}, {8, 2}, {16, 1}, {16, 2}, {32, 2}, {32, 4}};

bool lookup(int W, int B, int G, bool share, BatchKernels& out) {
#define GX_BK(w, b, g) \
  if (W == w && B == b && G == g) { out = batch_kernels<w, b, g>(share); return true; }
  GX_BK(1, 4, 1) GX_BK(1, 8, 1) GX_BK(1, 8, 2) GX_BK(1, 16, 1) GX_BK(1, 16, 2) GX_BK(1, 32, 2) GX_BK(1, 32, 4)
  GX_BK(2, 4, 1) GX_BK(2, 8, 1) GX_BK(2, 8, 2) GX_BK(2, 16, 1) GX_BK(2, 16, 2) GX_BK(2, 32, 2) GX_BK(2, 32, 4)
  GX_BK(4, 4, 1) GX_BK(4, 8, 1) GX_BK(4, 8, 2) GX_BK(4, 16, 1) GX_BK(4, 16, 2) GX_BK(4, 32, 2) GX_BK(4, 32, 4)
#undef GX_BK
  return false;
}

#define GB_CUDA(call)                                                                     \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return gx::fail(GX_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
  } while (0)

inline uint64_t a256(uint64_t x) { return (x + 255) & ~255ull; }
inline uint64_t p2ceil(uint64_t x) {
  uint64_t p = 1;
  while (p < x) p *= 2;
  return p;
}

struct BatchPlan {
  int W = 0, B = 0, G = 0, rounds = 0, chunk = 0;
  uint32_t levels_cap = 0, wide = 0;
  std::vector<uint64_t> slots, fcap;
  uint64_t off_nets = 0, off_claims = 0, off_active = 0, off_blobs = 0, off_levels = 0,
           off_fronts = 0, off_tables = 0, table_words = 0, total = 0;
  std::vector<uint64_t> blob_off, front_off, table_off;
  std::vector<uint32_t> order;  // networks by decreasing table size
  BatchKernels k{};
};

}  // namespace
}  // namespace gx

struct gx_batch {
  std::vector<gx::Net> nets;
  uint32_t W = 0;  // widest slot of the batch; narrower networks are padded to it
  // results of the last run
  bool have_result = false;
  std::vector<gx::BNet> res;
  std::vector<std::vector<uint64_t>> levels;
  double gpu_ms = 0;
  std::vector<uint64_t> last_plan_slots;
  uint64_t give_up_ns = gx::kGiveUpNs;
  uint32_t last_W = 0, last_B = 0, last_G = 0, last_rounds = 0;
};

namespace gx {
namespace {

gx_status batch_plan(const gx_batch* h, const gx_batch_opts* o, BatchPlan& P) {
  gx_batch_opts d{};
  if (!o) o = &d;
  const uint32_t n = (uint32_t)h->nets.size();
  P.W = (int)h->W;
  P.B = o->bucket_words ? (int)o->bucket_words : 8;
  P.G = o->group_lanes ? (int)o->group_lanes : 1;
  P.rounds = o->hash_rounds ? (int)o->hash_rounds : 8;
  P.chunk = o->chunk_states ? (int)o->chunk_states : 32;
  if (P.rounds < 1 || P.rounds > kMaxRounds) return fail(GX_ERR_INVALID, "hash_rounds must be 1..64");
  if (P.chunk < 32 || P.chunk % 32 || P.chunk > 4096)
    return fail(GX_ERR_INVALID, "chunk_states must be a multiple of 32 in 32..4096");
  bool share = false;  // of a rule's combinations, between lanes (WarpGen)
  for (const Net& net : h->nets) share |= net.lay.max_source >= gxd::kShareFrom;
  if (!lookup(P.W, P.B, P.G, share, P.k))
    return fail(GX_ERR_INVALID, "no batch kernel for bucket_words " + std::to_string(P.B) + ", group_lanes " +
                                    std::to_string(P.G) + " with " + std::to_string(P.W) + "-word slots");
  P.levels_cap = o->levels_cap ? o->levels_cap : 4096;
  P.wide = o->wide_factor ? o->wide_factor : 1u;
  P.slots.resize(n);
  P.fcap.resize(n);
  for (uint32_t i = 0; i < n; ++i) {
    uint64_t s = o->expected_states ? p2ceil(std::max<uint64_t>(1024, (o->expected_states[i] * 4 + 2) / 3))
                                    : (o->table_slots ? p2ceil(o->table_slots) : (1ull << 20));
    const uint64_t min_slots = std::max<uint64_t>(1024, 2ull * P.B / P.W);
    P.slots[i] = std::max(s, min_slots);
    // with expected sizes the ring holds a whole network (slots >= 4/3 of its states), so two
    // consecutive levels always fit; otherwise half the table
    P.fcap[i] = std::max<uint64_t>(4096, o->expected_states ? P.slots[i] : P.slots[i] / 2);
  }
  uint64_t off = 0;
  P.off_nets = off;
  off = a256(off + sizeof(BNet) * n);
  P.off_claims = off;
  off = a256(off + 8ull * (n + 1));
  P.off_active = off;
  off = a256(off + 24);
  P.off_blobs = off;
  P.blob_off.resize(n);
  for (uint32_t i = 0; i < n; ++i) {
    P.blob_off[i] = off;
    off = a256(off + 4ull * h->nets[i].blob.size());
  }
  P.off_levels = off;
  off = a256(off + 8ull * P.levels_cap * n);
  P.off_fronts = off;
  P.front_off.resize(n);
  for (uint32_t i = 0; i < n; ++i) {
    P.front_off[i] = off;
    off = a256(off + 4ull * P.W * P.fcap[i]);
  }
  P.off_tables = off;
  P.table_off.resize(n);
  for (uint32_t i = 0; i < n; ++i) {
    P.table_off[i] = off;
    off += 4ull * P.W * P.slots[i];  // power-of-two sizes of at least 4 KiB: stays aligned
  }
  P.table_words = (off - P.off_tables) / 4;
  P.total = a256(off);
  // large networks first: the levels of the last one left have the GPU to themselves
  P.order.resize(n);
  for (uint32_t i = 0; i < n; ++i) P.order[i] = i;
  std::stable_sort(P.order.begin(), P.order.end(), [&](uint32_t x, uint32_t y) { return P.slots[x] > P.slots[y]; });
  return GX_OK;
}

gx_status run_batch(gx_batch* h, const gx_batch_opts* o, void* ws, uint64_t ws_bytes, cudaStream_t st) {
  BatchPlan P;
  gx_status s = batch_plan(h, o, P);
  if (s != GX_OK) return s;
  if (!ws) return fail(GX_ERR_INVALID, "batched exploration needs a workspace (gx_batch_workspace_bytes)");
  if (ws_bytes < P.total)
    return fail(GX_ERR_OOM, "workspace holds " + std::to_string(ws_bytes) + " bytes, need " + std::to_string(P.total));
  if (reinterpret_cast<uintptr_t>(ws) % 256) return fail(GX_ERR_INVALID, "workspace is not 256-byte aligned");
  const int n = (int)h->nets.size();
  int dev = 0, sms = 0;
  GB_CUDA(cudaGetDevice(&dev));
  GB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  char* base = static_cast<char*>(ws);

  int per_sm = 0;
  GB_CUDA(cudaFuncSetAttribute(P.k.expand, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P.k.smem));
  GB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, P.k.expand, kBlock, P.k.smem));
  const int grid = sms * std::max(per_sm, 1);

  // the descriptors, and behind them the networks' encodings, as one copy (256 networks: 257
  // copies took 1.5 ms)
  std::vector<char> up(P.off_levels - P.off_nets, 0);
  BNet* const bn = reinterpret_cast<BNet*>(up.data());
  for (int k = 0; k < n; ++k) {
    const uint32_t i = P.order[k];
    const Net& net = h->nets[i];
    BNet& b = bn[k];
    b.blob = reinterpret_cast<const uint32_t*>(base + P.blob_off[i]);
    b.lay = net.lay;
    b.table = reinterpret_cast<uint32_t*>(base + P.table_off[i]);
    uint64_t nb = P.slots[i] * P.W / P.B;
    int l = 0;
    while ((1ull << l) < nb) ++l;
    b.log2nb = l;
    b.frontier = reinterpret_cast<uint32_t*>(base + P.front_off[i]);
    b.fmask = P.fcap[i] - 1;
    // the initial vector, padded to the batch's slot width (padding words carry only the tag)
    for (int w = 0; w < 4; ++w) b.init_vec[w] = w < P.W ? (net.init_vec[w] | kTag) : 0u;
    std::memcpy(up.data() + (P.blob_off[i] - P.off_nets), net.blob.data(), 4 * net.blob.size());
  }
  GB_CUDA(cudaMemcpyAsync(base + P.off_nets, up.data(), up.size(), cudaMemcpyHostToDevice, st));

  BatchArgs a{};
  a.nets = reinterpret_cast<BNet*>(base + P.off_nets);
  a.n = n;
  a.rounds = P.rounds;
  a.chunk = (uint32_t)P.chunk;
  a.levels_cap = P.levels_cap;
  a.levels = reinterpret_cast<unsigned long long*>(base + P.off_levels);
  a.claims = reinterpret_cast<unsigned long long*>(base + P.off_claims);
  a.active = reinterpret_cast<unsigned int*>(base + P.off_active);
  a.give_up_ns = h->give_up_ns;
  a.warps = (uint32_t)grid * (kBlock / 32);
  a.wide = P.wide == GX_BATCH_WIDE_OFF ? 0u : P.wide;
  hash_multipliers(a.muls.m, kMaxRounds);
  void* args[] = {&a};
  const int per_block = kBlock / 32;

  cudaEvent_t e0, e1;
  GB_CUDA(cudaEventCreate(&e0));
  GB_CUDA(cudaEventCreate(&e1));
  GB_CUDA(cudaEventRecord(e0, st));
  GB_CUDA(cudaMemsetAsync(base + P.off_tables, 0, 4 * P.table_words, st));
  GB_CUDA(cudaLaunchKernel(P.k.init, dim3((n + per_block - 1) / per_block), dim3(kBlock), args, 0, st));
  GB_CUDA(cudaLaunchKernel(P.k.expand, dim3(grid), dim3(kBlock), args, P.k.smem, st));
  GB_CUDA(cudaEventRecord(e1, st));
  GB_CUDA(cudaMemcpyAsync(bn, base + P.off_nets, sizeof(BNet) * n, cudaMemcpyDeviceToHost, st));
  GB_CUDA(cudaStreamSynchronize(st));
  float ms = 0;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  h->gpu_ms = ms;
  // as many levels as the deepest network has
  uint32_t deepest = 0;
  for (int k = 0; k < n; ++k) deepest = std::max(deepest, std::min<uint32_t>(bn[k].n_levels, P.levels_cap));
  std::vector<unsigned long long> lv((uint64_t)n * deepest);
  GB_CUDA(cudaMemcpyAsync(lv.data(), base + P.off_levels, 8ull * lv.size(), cudaMemcpyDeviceToHost, st));
  GB_CUDA(cudaStreamSynchronize(st));
  h->res.resize(n);
  h->levels.assign(n, {});
  gx_status rs = GX_OK;
  std::vector<uint32_t> slot(n);  // where network i is on the device
  for (int k = 0; k < n; ++k) slot[P.order[k]] = (uint32_t)k;
  for (int i = 0; i < n; ++i) {
    h->res[i] = bn[slot[i]];
    if (h->res[i].active && !h->res[i].error) h->res[i].error = ERR_SPIN;  // its warps gave up waiting
    const uint32_t k = std::min<uint32_t>(h->res[i].n_levels, P.levels_cap);
    h->levels[i].resize(k);
    for (uint32_t l = 0; l < k; ++l) h->levels[i][l] = lv[(uint64_t)l * n + slot[i]];
    if (h->res[i].error && rs == GX_OK) {
      const unsigned e = h->res[i].error;
      rs = (e & ERR_TABLE_FULL)  ? fail(GX_ERR_TABLE_FULL, "network " + std::to_string(i) + ": hash table full")
         : (e & ERR_FRONTIER)    ? fail(GX_ERR_FRONTIER_OVERFLOW, "network " + std::to_string(i) + ": frontier overflow")
         : (e & ERR_LEVELS)      ? fail(GX_ERR_OOM, "network " + std::to_string(i) + ": more levels than levels_cap")
                                 : fail(GX_ERR_SPIN_LIMIT, "network " + std::to_string(i) + ": left unfinished after waits that gave up");
    }
  }
  h->have_result = true;
  h->last_plan_slots = P.slots;
  h->last_W = (uint32_t)P.W;
  h->last_B = (uint32_t)P.B;
  h->last_G = (uint32_t)P.G;
  h->last_rounds = (uint32_t)P.rounds;
  return rs;
}

}  // namespace
}  // namespace gx

extern "C" {

gx_status gx_batch_create(const gx_net* const* nets, uint32_t n, gx_batch** out) {
  gx::clear_error();
  if (!nets || !out || n == 0) return gx::fail(GX_ERR_INVALID, "nets, n or out is invalid");
  gx_batch* h = new gx_batch();
  for (uint32_t i = 0; i < n; ++i) {
    if (!nets[i]) {
      delete h;
      return gx::fail(GX_ERR_INVALID, "nets[" + std::to_string(i) + "] is NULL");
    }
    h->nets.push_back(nets[i]->net);
    h->W = std::max(h->W, nets[i]->net.slot_words);
  }
  *out = h;
  return GX_OK;
}

void gx_batch_free(gx_batch* b) { delete b; }

gx_status gx_batch_set_wait_limit(gx_batch* b, uint64_t ns) {
  gx::clear_error();
  if (!b) return gx::fail(GX_ERR_INVALID, "batch is NULL");
  b->give_up_ns = ns ? ns : gx::kGiveUpNs;
  return GX_OK;
}

gx_status gx_batch_workspace_bytes(const gx_batch* b, const gx_batch_opts* opts, uint64_t* bytes) {
  gx::clear_error();
  if (!b || !bytes) return gx::fail(GX_ERR_INVALID, "batch or bytes is NULL");
  gx::BatchPlan P;
  gx_status s = gx::batch_plan(b, opts, P);
  if (s != GX_OK) return s;
  *bytes = P.total;
  return GX_OK;
}

gx_status gx_batch_explore(gx_batch* b, const gx_batch_opts* opts, void* ws, uint64_t ws_bytes, void* stream) {
  gx::clear_error();
  if (!b) return gx::fail(GX_ERR_INVALID, "batch is NULL");
  return gx::run_batch(b, opts, ws, ws_bytes, static_cast<cudaStream_t>(stream));
}

gx_status gx_batch_stats(const gx_batch* b, uint32_t i, gx_stats_t* out) {
  gx::clear_error();
  if (!b || !out) return gx::fail(GX_ERR_INVALID, "batch or out is NULL");
  if (!b->have_result) return gx::fail(GX_ERR_STATE, "no batched exploration has run");
  if (i >= b->res.size()) return gx::fail(GX_ERR_INVALID, "network index out of range");
  const gx::BNet& r = b->res[i];
  std::memset(out, 0, sizeof(*out));
  out->states = r.next_end;
  out->explored = r.cur_end;  // end of the last level that was expanded
  out->transitions = r.transitions;
  out->n_levels = r.n_levels;
  out->deadlock_count = r.dl_count;
  out->deadlock_sum = r.dl_sum;
  out->deadlock_xor = r.dl_xor;
  out->first_deadlock_level = r.first_dl;
  out->table_slots = b->last_plan_slots[i];
  out->vector_words = b->nets[i].vector_words;
  out->slot_words = b->last_W;
  out->bucket_words = b->last_B;
  out->group_lanes = b->last_G;
  out->hash_rounds = b->last_rounds;
  out->complete = (!r.active && !r.error) ? 1u : 0u;
  out->status = r.error ? 1u : 0u;
  out->fill = (double)r.next_end / (double)out->table_slots;
  out->gpu_ms = b->gpu_ms;
  out->probes = r.probes;
  return GX_OK;
}

gx_status gx_batch_levels(const gx_batch* b, uint32_t i, uint64_t* out, uint32_t cap, uint32_t* n) {
  gx::clear_error();
  if (!b) return gx::fail(GX_ERR_INVALID, "batch is NULL");
  if (!b->have_result) return gx::fail(GX_ERR_STATE, "no batched exploration has run");
  if (i >= b->levels.size()) return gx::fail(GX_ERR_INVALID, "network index out of range");
  if (cap && !out) return gx::fail(GX_ERR_INVALID, "out is NULL");
  const auto& L = b->levels[i];
  for (size_t k = 0; k < L.size() && k < cap; ++k) out[k] = L[k];
  if (n) *n = (uint32_t)L.size();
  return GX_OK;
}

gx_status gx_batch_autotune(gx_batch* b, gx_batch_opts* io, void* ws, uint64_t ws_bytes, void* stream,
                            double* best_ms) {
  gx::clear_error();
  if (!b || !io) return gx::fail(GX_ERR_INVALID, "batch or opts is NULL");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const uint32_t chunks[] = {32, 64, 128};
  gx_batch_opts best = *io;
  double best_t = 1e30;
  for (const auto& c : gx::kCands) {
    if (c[0] < (int)b->W) continue;
    for (uint32_t ch : chunks) {
      gx_batch_opts o = *io;
      o.bucket_words = (uint32_t)c[0];
      o.group_lanes = (uint32_t)c[1];
      o.chunk_states = ch;
      gx::BatchPlan P;
      if (gx::batch_plan(b, &o, P) != GX_OK || P.total > ws_bytes) continue;
      // one warm-up, then the median of three timed runs
      gx_status s = gx::run_batch(b, &o, ws, ws_bytes, st);
      if (s != GX_OK) continue;
      double t[3];
      for (double& x : t) {
        if (gx::run_batch(b, &o, ws, ws_bytes, st) != GX_OK) x = 1e30;
        else x = b->gpu_ms;
      }
      std::sort(t, t + 3);
      if (t[1] < best_t) {
        best_t = t[1];
        best = o;
      }
    }
  }
  gx::clear_error();
  if (best_t >= 1e30) return gx::fail(GX_ERR_INVALID, "no candidate configuration ran");
  *io = best;
  if (best_ms) *best_ms = best_t;
  return GX_OK;
}

}  // extern "C"
