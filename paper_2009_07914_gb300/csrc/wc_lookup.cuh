// Lookups of windows of at most 64 bytes: one query per thread, straight-line.
//
// With the table in L2 a lookup is bound by instruction issue and by the SM's load path,
// not by memory latency, so this kernel spends as little as it can per query: no group
// votes, no key hand-out, one probe of the first window per query (which ends about four
// of five lookups at load 0.9).  The queries it leaves open go to a queue of their warp in
// shared memory and are probed 32 at a time, so no lane waits for the warp's longest walk.
// The stop rules are those of sv_retrieve_range, the group-per-key engine that lookups of
// every window used to run on and wider windows still do.
//
// 4+4-byte pairs, 2^27 queries, one GB300, that engine (its best lane shape) against this
// kernel: 9 MiB table at load 0.9 with overflow bits, half absent 75.7 -> 105 G lookups/s
// (counters: issue 63 % busy, load path 70 %); 16 MiB at load 0.5 66.6 -> 146; 142 MiB at
// 0.9 44.5 -> 64.5; 1.1 GiB, from HBM, 26.0 -> 28.5 (one 64-byte request per window either
// way: bound by the random-line rate).  8+8-byte pairs: 18 MiB 42.0 -> 87.3.
#pragma once

#include <type_traits>

#include "wc_launch.cuh"
#include "wc_partition.cuh"
#include "wc_sv_kernels.cuh"

namespace wc {

constexpr int kLookThreads = 256;
constexpr uint32_t kLookChunk = 512;  // keys a warp of the group-per-key engine takes from the sweep counter at a time
constexpr uint64_t kSweepLead = 8ull << 20;  // table bytes a sweep's prefetch runs ahead (BatchBlocks::prefetch)

template <class L>
constexpr int slot_size() {
  return L::kHalf ? 4 : L::kWords * 8;
}

// Windows this kernel serves: at most 64 bytes (16 registers of slots per query).
template <class L>
constexpr bool lookup_window(int W) {
  return W * slot_size<L>() <= 64;
}

template <class L>
struct EmitLookup {
  typename L::Val* __restrict__ out;
  uint8_t* __restrict__ found;
  const void* vals;  // struct-of-arrays value array (else unused)
  __device__ __forceinline__ void operator()(uint32_t pos, bool hit, typename L::Val v, uint64_t idx) const {
    if (out != nullptr) {
      if constexpr (L::kSoA) {
        out[pos] = hit ? static_cast<const typename L::Val*>(vals)[idx] : L::kNotFound;
      } else {
        out[pos] = hit ? v : L::kNotFound;
      }
    }
    if (found != nullptr) found[pos] = hit ? 1 : 0;
  }
};

// What a query's probe of one window found.
template <class L>
struct Probe {
  typename L::Val v;  // its value (struct-of-arrays layouts: not read here)
  uint32_t sub;       // struct-of-arrays layouts: slot number of the key
  bool hit;           // the key
};

// S slots looked through for the key k; `at` = slot number of the first of them.
template <class L, int S>
__device__ __forceinline__ Probe<L> find_in(const typename L::Slot (&s)[S], typename L::Key k, uint32_t at) {
  Probe<L> r;
  r.v = typename L::Val(0);
  r.sub = 0;
  r.hit = false;
#pragma unroll
  for (int i = 0; i < S; ++i) {
    if (L::key(s[i]) == k) {
      r.hit = true;
      if constexpr (L::kSoA) r.sub = at + i;
      else if constexpr (!L::kHalf) r.v = L::val(s[i]);
    }
  }
  return r;
}

// Lanes without a key load a window as well (clearing the registers instead costs more), so
// in a step of a warp's queue they are handed the one of lane 0, which its warp reads
// anyway: with the table's first window for all of them the tails of all warps met on one
// line of the L2 (222,476 lookups at load 0.9, half absent, 8+8 bytes 44.7 -> 27.4 us;
// 317,816 of 4+4 bytes 32.0 -> 18.6).  Every lane calls; lane 0 holds an entry of the queue.
__device__ __forceinline__ uint32_t window_for_all(bool on, uint32_t w) {
  const uint32_t first = __shfl_sync(kFull, w, 0);
  return on ? w : first;
}

// Probe window w for the key k (not a sentinel) in every lane with `on`; every lane of the
// warp calls, with a window of the table.  `full`: the window holds no empty slot.  Inserts claim the first empty or
// tombstoned slot of a window and no slot becomes empty again, so the empty slots of a
// window are always its last ones: it holds one exactly when its last slot is empty.
//
// A window of at most 32 bytes is one load of its lane.  A 64-byte window is read by a pair
// of lanes, 32 bytes each in one instruction, so it is one request and one tag look-up of
// the SM's load path instead of two (the path looks up one line per clock, which bounds
// lookups in L2; from HBM two requests per window halve the rate): the pair reads the
// windows of both its queries, each lane looks for both keys in its half and hands the
// other lane what it found.
template <class L, int W>
__device__ __forceinline__ Probe<L> probe_window(const typename L::Slot* slots, bool on, typename L::Key k,
                                                 uint32_t w, bool& full) {
  using Slot = typename L::Slot;
  Probe<L> r;
  if constexpr (W * slot_size<L>() <= 32) {
    Slot s[W];
    load_slots<L, W>(slots + static_cast<uint64_t>(w) * W, s);
    r = find_in<L, W>(s, k, 0);
    full = L::key(s[W - 1]) != L::kEmpty;
  } else {
    constexpr int S = W / 2;
    const bool odd = threadIdx.x & 1;
    const uint32_t ow = __shfl_xor_sync(kFull, w, 1);
    const typename L::Key ok = __shfl_xor_sync(kFull, k, 1);
    const uint32_t half = odd ? S : 0;
    Slot a[S], b[S];  // my half of the even lane's window and of the odd lane's
    load_slots<L, S>(slots + static_cast<uint64_t>(odd ? ow : w) * W + half, a);
    load_slots<L, S>(slots + static_cast<uint64_t>(odd ? w : ow) * W + half, b);
    const Probe<L> ra = find_in<L, S>(a, odd ? ok : k, half), rb = find_in<L, S>(b, odd ? k : ok, half);
    r = odd ? rb : ra;
    const Probe<L> o = odd ? ra : rb;  // what I found for the other lane's key
    // bit 0: hit; bit 1 (from the odd lane, which has the last slots): the even lane's window is full
    const bool fa = L::key(a[S - 1]) != L::kEmpty, fb = L::key(b[S - 1]) != L::kEmpty;
    uint32_t msg = (o.hit ? 1u : 0u) | (fa ? 2u : 0u);
    if constexpr (L::kSoA) msg |= o.sub << 2;
    const uint32_t of = __shfl_xor_sync(kFull, msg, 1);
    if constexpr (!L::kHalf && !L::kSoA) {
      const typename L::Val ov = __shfl_xor_sync(kFull, o.v, 1);
      if (of & 1u) r.v = ov;
    }
    if constexpr (L::kSoA) {
      if (of & 1u) r.sub = of >> 2;
    }
    r.hit = r.hit || (of & 1u) != 0;
    full = odd ? fb : (of & 2u) != 0;
  }
  r.hit = r.hit && on;
  full = full && on;
  return r;
}

// Regions that a batch of queries is split into (MiB), and the inputs of a chunk of its
// sweep.  Small ones sweep faster: 2^27 queries of 4+4 bytes over 1.2 GiB in regions of 32
// MiB and chunks of 512 1.67 ms, 16 and 512 1.52, 16 and 256 1.45 (32 and 256 1.60); 8 MiB
// 1.49.  Twice the regions split and put back slower (0.04 ms there), which large tables
// do not get back: 2^28 Zipf queries of 8+8 bytes over 4.8 GiB sweep in 2.89 ms with 32 and
// 512 (3.07 with 256) and 2.84 with 16, for 0.6 ms more before and after.
constexpr uint64_t kSmallSweep = 2ull << 30;
__host__ __device__ constexpr int look_region_mib(uint64_t slots_bytes) { return slots_bytes > kSmallSweep ? 32 : 16; }
__host__ __device__ constexpr uint32_t look_chunk(uint64_t slots_bytes) { return slots_bytes > kSmallSweep ? 512 : 256; }

// A warp's blocks of 32 consecutive inputs (warp-uniform).  kSwept: chunks of inputs are taken
// from a counter in order, so the grid sweeps the batch front to back; otherwise the blocks
// are strided over the grid (kernels of their own: a direct batch carries none of the sweep's
// registers).  Inputs are numbered in 32 bits (n < 2^32).
//
// What the warps of a sweep hold together is the part of the table that has to stay in L2,
// so chunks are short, and a sweep of lookups asks for the next one when one is begun
// (early), so no warp waits for the counter.  Chunks of 192, 128 and 64: 1.47, 1.65 and 2.9
// ms for 2^27 lookups, as the counter takes only some 0.3 to 0.7 atomics per ns.  It takes
// fewest beside inserts, which are fastest with 512 asked for when needed (2^27 pairs of 4+4
// bytes: early 8 % slower, early 256 6 %; 2^26 Zipf counting inserts 0.63 ms, early 256
// 0.88).  Batches below 2^21 take shorter chunks: there are about 5000 warps.
template <bool kSwept>
struct BatchBlocks {
  uint32_t n, next, end;  // end of the taken chunk
  uint32_t stride;        // between a warp's blocks; of a sweep, inputs of a chunk
  unsigned long long* counter;
  unsigned long long later;  // first input of the chunk after this one (lane 0)
  const char* tab = nullptr;  // prefetch: the table, its bytes, bytes per input << 16
  uint64_t tab_bytes = 0, ratio = 0;
  bool early;  // ask for the next chunk when one is begun
  // most: inputs of a chunk
  __device__ __forceinline__ BatchBlocks(uint64_t n_, unsigned long long* c, uint32_t most, bool early_)
      : n(static_cast<uint32_t>(n_)), next(kSwept ? n : (blockIdx.x * blockDim.x + threadIdx.x) & ~31u), end(n),
        stride(kSwept ? min(most, max(32u, n >> 12 & ~31u)) : gridDim.x * blockDim.x), counter(c), later(0),
        early(early_) {
    if (kSwept && early) ask();
  }
  // all of n inputs for this warp (one tile of the batched executor)
  __device__ __forceinline__ explicit BatchBlocks(uint32_t n_)
      : n(n_), next(0), end(n_), stride(32), counter(nullptr), later(0), early(false) {}
  __device__ __forceinline__ void ask() {
    if ((threadIdx.x & 31) == 0) later = atomicAdd(counter, static_cast<unsigned long long>(stride));
  }
  // A sweep of inserts copies the table to L2 kSweepLead ahead of itself, in order, as much
  // per chunk as its share of the batch: the windows it reads next are not fetched one by one
  // from DRAM.  A batch that would not touch most windows is left alone; for a skewed one the
  // place in the table is a guess and the copies are at most the table's size.
  // 2^27 pairs of 4+4 bytes 2.97 -> 2.74 ms, 2^28 of 8+8 8.19 -> 7.94 (16 MiB ahead 2.76 and
  // 8.15), counting and set inserts 2 and 1 %.  Lookups gain nothing (1.46 ms both ways,
  // 8-byte ones 2.94 -> 3.1), inserts of open-addressing multi-value tables lose (2^26 1.81
  // -> 1.91): neither calls this.
  __device__ __forceinline__ void prefetch(const void* slots, uint64_t bytes) {
    if (!kSwept || bytes > static_cast<uint64_t>(n) * 64) return;
    tab = static_cast<const char*>(slots);
    tab_bytes = bytes & ~127ull;
    ratio = (bytes << 16) / n;  // n > 0: a table has bytes
  }
  __device__ __forceinline__ void prefetch_for(uint64_t c) const {
    const uint64_t a = (c * ratio >> 16 & ~127ull) + kSweepLead;
    uint64_t e = ((c + stride) * ratio >> 16 & ~127ull) + kSweepLead;
    if (e > tab_bytes) e = tab_bytes;
    if (a < e)  // at most 32 KiB: 512 inputs of up to 64 bytes of table each
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(tab + a), "r"(static_cast<uint32_t>(e - a))
                   : "memory");
  }
  // first input of the next block, n when there is none
  __device__ __forceinline__ uint32_t take() {
    if constexpr (!kSwept) {
      const uint32_t b = next;
      next = b < n && n - b > stride ? b + stride : n;
      return b < n ? b : n;
    }
    if (next >= end) {
      if (!early) ask();
      const unsigned long long c = __shfl_sync(kFull, later, 0);
      if (c >= n) return n;  // and so every time from now on
      if (early) ask();
      if (tab != nullptr && (threadIdx.x & 31) == 0) prefetch_for(c);
      next = static_cast<uint32_t>(c);
      end = n - next > stride ? next + stride : n;
    }
    const uint32_t b = next;
    next = end - b > 32 ? b + 32 : end;
    return b;
  }
};

// A warp's queue of open queries: at most 31 left over + 32 of one step.
constexpr int kWarpQueue = 64;
template <class KIn>
struct LookupQueue {
  KIn key[kWarpQueue];
  uint32_t pos[kWarpQueue], w[kWarpQueue], j[kWarpQueue];
};

// The lookups of a warp's blocks; every lane calls.
template <class L, int W, bool kSwept, class Emit, class KIn>
__device__ __forceinline__ void lookup_blocks(const TableDesc& t, const KIn* __restrict__ keys, BatchBlocks<kSwept>& blocks,
                                              LookupQueue<KIn>& q, const Emit& emit, uint32_t& flags) {
  using Slot = typename L::Slot;
  using Key = typename L::Key;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  const Slot* slots = static_cast<const Slot*>(t.slots);
  uint32_t cnt = 0;

  // one step for the last (at most 32) queries of the queue: the next window of their
  // sequence, and where that is full its overflow bit
  auto drain = [&]() {
    const uint32_t m = cnt < 32 ? cnt : 32;
    cnt -= m;
    __syncwarp();
    const bool on = lane < m;
    KIn kin = 0;
    uint32_t pos = 0, w = 0, j = 0;
    if (on) {
      kin = q.key[cnt + lane];
      pos = q.pos[cnt + lane];
      w = q.w[cnt + lane];
      j = q.j[cnt + lane] + 1;
    }
    __syncwarp();
    const Key k = static_cast<Key>(kin);
    uint32_t w0, step, tag;
    probe_init(static_cast<uint64_t>(k), t.seed, t.p, w0, step, tag);
    const bool go = on && j < t.p;
    if (go) w = probe_next(w, step, t.p);
    w = window_for_all(on, w);
    bool full;
    const Probe<L> r = probe_window<L, W>(slots, go, k, w, full);
    bool again = full && !r.hit;
    if (t.ovf != nullptr && again) again = ovf_bit(ovf_word(t.ovf, w), w, tag);
    const uint32_t b = __ballot_sync(kFull, again);
    if (again) {
      const uint32_t at = cnt + __popc(b & below);
      q.key[at] = kin;
      q.pos[at] = pos;
      q.w[at] = w;
      q.j[at] = j;
    }
    cnt += __popc(b);
    if (on && !again) emit(pos, r.hit, r.v, static_cast<uint64_t>(w) * W + r.sub);
  };

  const uint32_t nn = blocks.n;
  uint32_t base = blocks.take();
  KIn kn = nn - base > lane ? ldg_stream(keys + base + lane) : KIn(0);
  while (base != nn) {
    const KIn kin = kn;
    const bool in = nn - base > lane;
    const uint32_t pos = base + lane;
    base = blocks.take();
    kn = nn - base > lane ? ldg_stream(keys + base + lane) : KIn(0);  // the next block's queries
    const bool bad = in && is_sentinel(kin);
    if (bad) flags |= kFlagInvalid;
    const Key k = static_cast<Key>(kin);
    const uint64_t h = fmix64(static_cast<uint64_t>(k) ^ t.seed);  // as probe_init
    const uint32_t w = __umulhi(static_cast<uint32_t>(h >> 32), t.p);
    const bool on = in && !bad;
    bool full;
    const Probe<L> r = probe_window<L, W>(slots, on, k, w, full);
    bool open = full && !r.hit;
    if (t.ovf != nullptr && open) open = ovf_bit(ovf_word(t.ovf, w), w, static_cast<uint32_t>(h) & 7u);
    const uint32_t b = __ballot_sync(kFull, open);
    if (open) {
      const uint32_t at = cnt + __popc(b & below);
      q.key[at] = kin;
      q.pos[at] = pos;
      q.w[at] = w;
      q.j[at] = 0;
    }
    cnt += __popc(b);
    if (in && !open) emit(pos, r.hit, r.v, static_cast<uint64_t>(w) * W + r.sub);
    while (cnt >= 32) drain();
  }
  while (cnt > 0) drain();
}

// kSwept: a batch sorted by table region, swept in order by `counter`.
template <class L, int W, class Emit, class KIn, bool kSwept>
__global__ void __launch_bounds__(kLookThreads, 5) k_lookup(TableDesc t, const KIn* __restrict__ keys, uint64_t n,
                                                            unsigned long long* counter, Emit emit) {
  __shared__ LookupQueue<KIn> q[kLookThreads / 32];
  uint32_t flags = 0;
  const uint64_t bytes = static_cast<uint64_t>(t.p) * W * slot_size<L>();
  BatchBlocks<kSwept> blocks(n, counter, look_chunk(bytes), true);
  lookup_blocks<L, W>(t, keys, blocks, q[threadIdx.x >> 5], emit, flags);
  flush_flags(t.status, flags);
}

// Lookups of a batch split by region (the blocked scheme) sweep the table region by region
// in L2: 2^27 queries of 4+4-byte pairs over a 1.1 GiB table take 0.20 ms to count the
// regions, 0.48 ms to split, 1.45 ms to probe and 0.44 ms to put back, against 4.71 ms in
// input order (5.14 on the group-per-key engine).
//
// Results of a batch split by region, back in input order: the split kept every input
// tile's elements of a region together (runs[tile * R + r] = where that run starts in the
// split batch and in the tile's own region order), so the block of a tile reads the tile's
// R runs, puts every result at its input position (lidx) in shared memory and writes the
// tile out in order -- no scattered store leaves the SM.
template <class V, class Out = V>
__global__ void __launch_bounds__(kPartThreads, 3) k_unsplit(const uint16_t* __restrict__ lidx, const V* __restrict__ rv,
                                                          const uint8_t* __restrict__ rf, uint64_t n, uint32_t R,
                                                          const uint2* __restrict__ runs, Out* __restrict__ out,
                                                          uint8_t* __restrict__ found) {
  __shared__ V s_v[kPartTile];
  __shared__ __align__(4) uint8_t s_f[kPartTile];
  __shared__ uint32_t s_pos[kMaxRegions];
  __shared__ uint16_t s_off[kMaxRegions + 1];
  const uint64_t ntiles = (n + kPartTile - 1) / kPartTile;
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    for (uint32_t r = threadIdx.x; r < R; r += kPartThreads) {
      const uint2 x = runs[tile * R + r];
      s_pos[r] = x.x;
      s_off[r] = static_cast<uint16_t>(x.y);
    }
    if (threadIdx.x == 0) s_off[R] = 0xffffu;
    __syncthreads();
    const uint64_t t0 = tile * kPartTile;
    const uint32_t tn = static_cast<uint32_t>(n - t0 < kPartTile ? n - t0 : kPartTile);
    // a warp takes consecutive elements of the region order, so each row of 32 starts in the
    // run where the row before it ended or a few runs on
    const uint32_t first = (threadIdx.x >> 5) * (32 * kPartItems) + (threadIdx.x & 31);
    uint32_t r = 0, hi = R - 1;  // the last run starting at or before `first` (an empty run starts where the next does)
    while (r < hi) {
      const uint32_t mid = (r + hi + 1) >> 1;
      if (s_off[mid] <= first) r = mid;
      else hi = mid - 1;
    }
#pragma unroll
    for (int h = 0; h < kPartItems; h += 4) {
      uint32_t p[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t i = first + (h + k) * 32;
        while (s_off[r + 1] <= i) ++r;  // s_off[R] is past every element
        p[k] = s_pos[r] + (i - s_off[r]);
      }
      uint16_t li[4];
      V v[4];
      uint8_t f[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (first + (h + k) * 32 >= tn) continue;
        li[k] = lidx[p[k]];
        if (out != nullptr) v[k] = rv[p[k]];
        if (found != nullptr) f[k] = rf[p[k]];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (first + (h + k) * 32 >= tn) continue;
        if (out != nullptr) s_v[li[k]] = v[k];
        if (found != nullptr) s_f[li[k]] = f[k];
      }
    }
    __syncthreads();
    if (out != nullptr) {
#pragma unroll
      for (int k = 0; k < kPartItems; ++k) {
        const uint32_t i = k * kPartThreads + threadIdx.x;
        if (i < tn) out[t0 + i] = s_v[i];
      }
    }
    if (found != nullptr) {
      if (tn == kPartTile && (reinterpret_cast<uintptr_t>(found) & 3) == 0) {
        const auto* s4 = reinterpret_cast<const uint32_t*>(s_f);
        auto* f4 = reinterpret_cast<uint32_t*>(found + t0);
        for (uint32_t i = threadIdx.x; i < kPartTile / 4; i += kPartThreads) f4[i] = s4[i];
      } else {
        for (uint32_t i = threadIdx.x; i < tn; i += kPartThreads) found[t0 + i] = s_f[i];
      }
    }
    __syncthreads();
  }
}

// ---- host side ---------------------------------------------------------------------------

// Lookups in input order run as many blocks as fit (five an SM) while the table stays within
// reach of the L2, three above 160 MiB: their window reads then come from DRAM, and with all
// five in flight those get in each other's way.  Five against three blocks, queries all
// present / half absent: 140 MiB of 4+4-byte slots at load 0.6 138 / 149 us against 155 / 161,
// 200 MiB of 8+8 at 0.9 316 / 531 against 295 / 514, 430 MiB 878 / 1604 against 772 / 1451,
// 500 MiB of 4+4 at 0.6 895 / 954 against 834 / 888; above 1 GiB and on Zipf queries the two
// are within 2 % of each other.  (Two blocks: 2 to 5 % slower below 300 MiB, the same above.)
constexpr uint64_t kLookFewer = 160ull << 20;
inline int look_blocks_per_sm(const wc_table* t, int most, bool swept) {
  return swept || t->table_bytes <= kLookFewer ? most : std::min(most, 3);
}

template <class L, int W, class Emit, class KIn = typename L::Key>
cudaError_t lookup_launch(const wc_table* t, const KIn* keys, uint64_t n, unsigned long long* counter,
                          const Emit& emit, cudaStream_t s) {
  auto kern = counter != nullptr ? k_lookup<L, W, Emit, KIn, true> : k_lookup<L, W, Emit, KIn, false>;
  const uint64_t want = (n + kLookThreads - 1) / kLookThreads;
  const int per_sm = look_blocks_per_sm(t, occupancy(kern, kLookThreads), counter != nullptr);
  const uint64_t most = static_cast<uint64_t>(per_sm) * t->sm_count;
  return launch_k(t, kern, static_cast<unsigned>(std::min(want, most)), kLookThreads, 0, s, desc_of(t), keys, n,
                  counter, emit);
}

// A batch of queries split by table region, with room for the results in split order.
template <class K, class V>
struct QuerySplit {
  RegionSplit<K, uint16_t> sp;
  V* rv;
  uint8_t* rf;
  uint2* runs;
  uint32_t R;
};

template <class K, class V>
cudaError_t query_split(const wc_table* t, int region_mib, const K* keys, uint64_t n, cudaStream_t s,
                        QuerySplit<K, V>& q) {
  const uint64_t slots_bytes = t->windows * t->W * t->slot_bytes;
  const RegionMap m = region_map(t, region_mib > 0 ? region_mib : look_region_mib(slots_bytes));
  q.R = m.R;
  const uint64_t ntiles = (n + kPartTile - 1) / kPartTile;
  const uint64_t rv_bytes = align256(n * sizeof(V)), rf_bytes = align256(n);
  const uint64_t runs_bytes = ntiles * q.R * sizeof(uint2);
  const cudaError_t e = region_split<K, uint16_t, kValsLocal>(t, m, keys, nullptr, n, s, q.sp,
                                                              rv_bytes + rf_bytes + runs_bytes, rv_bytes + rf_bytes);
  if (e != cudaSuccess) return e;
  q.rv = reinterpret_cast<V*>(q.sp.extra);
  q.rf = reinterpret_cast<uint8_t*>(q.sp.extra + rv_bytes);
  q.runs = reinterpret_cast<uint2*>(q.sp.extra + rv_bytes + rf_bytes);
  return cudaSuccess;
}

template <class K, class V, class Out = V>
cudaError_t unsplit_launch(const wc_table* t, const QuerySplit<K, V>& q, uint64_t n, Out* out, uint8_t* found,
                           cudaStream_t s) {
  auto kern = k_unsplit<V, Out>;
  const uint64_t ntiles = (n + kPartTile - 1) / kPartTile;
  const unsigned grid = static_cast<unsigned>(
      std::min<uint64_t>(ntiles, static_cast<uint64_t>(occupancy(kern, kPartThreads)) * t->sm_count));
  kern<<<grid, kPartThreads, 0, s>>>(q.sp.vals, q.rv, q.rf, n, q.R, q.runs, out, found);
  return cudaGetLastError();
}

}  // namespace wc
