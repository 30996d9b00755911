// Multi-split of a batch by table region (the partition step of the paper's distributed
// mode, Sec. IV-E, applied to L2-sized regions of one table instead of to GPUs).
//
// Region of a key = (first window of its probing sequence) / windows_per_region.  After
// the split the batch is ordered by region, so a probe kernel that sweeps it front to
// back touches one table region (a few tens of MB) at a time: its window loads and CAS
// claims hit L2 instead of HBM, and every region is read from and written back to HBM
// about once.  The order of keys inside a region is unspecified (bulk operations are
// sets of independent element operations).
#pragma once

#include <algorithm>
#include <type_traits>

#include "wc_device.cuh"
#include "wc_internal.h"
#include "wc_launch.cuh"

namespace wc {

constexpr int kPartThreads = 512;
constexpr int kPartItems = 8;
constexpr int kPartTile = kPartThreads * kPartItems;
constexpr int kMaxRegions = 1024;      // of a sweep (region_map)
constexpr int kMaxSplitRegions = 2048; // of any split (header areas)

struct RegionMap {
  uint64_t seed;
  uint32_t p;      // windows of the table
  uint32_t shift;  // 2^shift windows per region
  uint32_t R;      // regions
  template <class K>
  __device__ __forceinline__ uint32_t of(K key) const {
    uint32_t w, step;
    probe_init(static_cast<uint64_t>(key), seed, p, w, step);
    return w >> shift;  // below R = ceil(p / 2^shift), since w < p
  }
};

// Regions of a table: a power of two of windows each (a shift instead of a division per
// key), the largest one within region_mib MiB (0 = 32), doubled until there are at most
// kMaxRegions of them.
inline RegionMap region_map(const wc_table* t, int region_mib) {
  const uint64_t region_bytes = static_cast<uint64_t>(region_mib > 0 ? region_mib : 32) << 20;
  const uint64_t window_bytes = t->W * t->slot_bytes;
  uint32_t shift = 0;
  while ((window_bytes << (shift + 1)) <= region_bytes && shift < 31) ++shift;
  while (((t->windows + (1ull << shift) - 1) >> shift) > static_cast<uint64_t>(kMaxRegions)) ++shift;
  RegionMap m;
  m.seed = t->cfg.seed;
  m.p = static_cast<uint32_t>(t->windows);
  m.shift = shift;
  m.R = static_cast<uint32_t>((t->windows + (1ull << shift) - 1) >> shift);
  return m;
}

// Per-region counts of the batch (hist[R], zeroed by the caller).  Warps share `copies`
// shared-memory histograms (one each while the regions are few), so few atomics collide.
constexpr int kHistWarps = kPartThreads / 32;

inline uint32_t hist_copies(uint32_t R) { return R <= 512 ? kHistWarps : R <= 1024 ? 8 : 4; }

template <class K>
__global__ void __launch_bounds__(kPartThreads) k_part_hist(const K* __restrict__ keys, uint64_t n, RegionMap m,
                                                            unsigned int* __restrict__ hist, uint32_t copies,
                                                            const unsigned long long* n_dev) {
  extern __shared__ __align__(16) unsigned int s_hw[];  // copies * R
  if (n_dev != nullptr) n = *n_dev;
  for (uint32_t i = threadIdx.x; i < copies * m.R; i += kPartThreads) s_hw[i] = 0;
  __syncthreads();
  unsigned int* mine = s_hw + ((threadIdx.x >> 5) & (copies - 1)) * m.R;
  // kPartItems independent loads in flight per thread (block b takes elements
  // [b * kPartTile, (b + 1) * kPartTile) of every grid-wide stride, one per thread per item)
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * kPartTile;
  for (uint64_t e0 = static_cast<uint64_t>(blockIdx.x) * kPartTile + threadIdx.x; e0 < n; e0 += stride) {
    K x[kPartItems];
#pragma unroll
    for (int u = 0; u < kPartItems; ++u) {
      const uint64_t e = e0 + static_cast<uint64_t>(u) * kPartThreads;
      x[u] = e < n ? ldg_stream(keys + e) : K(0);
    }
#pragma unroll
    for (int u = 0; u < kPartItems; ++u)
      if (e0 + static_cast<uint64_t>(u) * kPartThreads < n) atomicAdd(mine + m.of(x[u]), 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < m.R; i += kPartThreads) {
    unsigned int c = 0;
    for (uint32_t w = 0; w < copies; ++w) c += s_hw[w * m.R + i];
    if (c) atomicAdd(hist + i, c);
  }
}

// Words of shared memory that scan_regions takes for the counts and for their scan.
__host__ __device__ constexpr uint32_t scan_cnt_words(uint32_t R) { return (R + 3) / 4 * 4; }
__host__ __device__ constexpr uint32_t scan_off_words(uint32_t R) { return scan_cnt_words(R) + 4; }

// Exclusive scan of cnt[0..R) into off[0..R], off[R] the total, by the whole block
// (R <= kMaxSplitRegions; both 16-byte aligned, counts behind R up to scan_cnt_words are zero);
// ends with a barrier.  Up to 512 regions are scanned by the first warp alone while the
// others wait: a lane takes up to 16 neighbouring counts in 16-byte words, so the chain that
// the block waits for is one scan over lanes.
__device__ __forceinline__ void scan_regions(const uint32_t* cnt, uint32_t* off, uint32_t R, uint32_t* s_w) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (R <= 512) {
    if (warp == 0) {
      const uint32_t b = lane * ((R + 127) / 128) * 4, end = min(b + (R + 127) / 128 * 4, scan_cnt_words(R));
      uint32_t sum = 0;
#pragma unroll 1
      for (uint32_t i = b; i < end; i += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(cnt + i);
        sum += v.x + v.y + v.z + v.w;
      }
      uint32_t inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
      }
      uint32_t run = inc - sum;
#pragma unroll 1
      for (uint32_t i = b; i < end; i += 4) {  // the counts again: few registers held
        const uint4 v = *reinterpret_cast<const uint4*>(cnt + i);
        const uint4 o = make_uint4(run, run + v.x, run + v.x + v.y, run + v.x + v.y + v.z);
        *reinterpret_cast<uint4*>(off + i) = o;
        run = o.w + v.w;
      }
      if (lane == 31) off[R] = inc;  // what a word past the counts holds there already
    }
    __syncthreads();
    return;
  }
  constexpr int kPer = kMaxSplitRegions / kPartThreads;
  const uint32_t b0 = threadIdx.x * kPer;
  uint32_t v[kPer], sum = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    v[k] = b0 + k < R ? cnt[b0 + k] : 0u;
    sum += v[k];
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  uint32_t run = inc - sum;
#pragma unroll
  for (int w = 0; w < kPartThreads / 32; ++w)
    if (w < warp) run += s_w[w];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (b0 + k < R) off[b0 + k] = run;
    run += v[k];
    if (b0 + k == R - 1) off[R] = run;
  }
  __syncthreads();
}

// Asynchronous global -> shared copy of one 4- or 8-byte element (cp.async, L1 bypassed
// for the streamed input with an evict-first L2 policy), and the wait for all of them.
template <class T>
__device__ __forceinline__ void cp_async_elem(T* smem_dst, const T* gmem_src) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "element size");
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], %2, %3;"
               :
               : "r"(d), "l"(gmem_src), "n"(static_cast<int>(sizeof(T))), "l"(evict_first_policy())
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Where the values of a split come from: read from `vals`, element i's position inside its
// tile, or there are none (vals is read in the first only, ovals not written in the last).
// With kValsLocal the split also leaves runs[tile * R + r] = (start of the tile's run of
// region r in the output, its start in the tile's own region order), from which k_unsplit
// puts results back in input order.
enum { kValsRead = 0, kValsLocal = 1, kValsNone = 2 };

// Scatter (keys, vals) into region order.  Per tile: rank every element inside its region
// with shared-memory atomics, reserve one run per region in the output with one global
// atomic on cursor[r] (zeroed by the caller), stage the tile in shared memory grouped by
// region, then copy the runs out with consecutive threads on consecutive addresses.
// Issue and the shared-memory pipe bound it (both about two thirds busy), so what an
// element takes is kept short: its place in the output is delta[region] + its place in the
// staged tile, position and region of a split with positions share one staged word.  What a
// tile's barriers wait for is short too: the scan over the regions is one warp's and only
// shared memory, the reservations (a global round trip) are made by all threads side by side.
// 4-byte inputs come through buffers that cp.async fills for the next tile while this one is
// written out (4-byte keys only if their values come that way too); 8-byte ones are read
// into registers: through buffers 2^28 pairs of 8+8 bytes take 2.03 ms against 1.69, and
// 8-byte keys beside buffered 4-byte values 1.80 against 1.49.  Pairs of at most 8 bytes hold
// no input in registers and run three blocks an SM, wider ones two.
// One GB300, with the reservations inside the one warp's scan -> as it is: 2^28 pairs of 8+8
// bytes 2.09 -> 1.69 ms (5.1 TB/s), 8+4 1.85 -> 1.49, 2^28 queries of 8 bytes (with
// positions) 1.66 -> 1.23, of 4 bytes 2^27 0.495 -> 0.473, 2^27 pairs of 4+4 0.662 -> 0.635,
// 2^27 keys alone into 1300 regions 0.77 -> 0.59, 60 M into 256 0.188 -> 0.185.
template <class K, class V, int kVals>
struct SplitTile {
  static constexpr bool kRead = kVals == kValsRead;
  static constexpr bool kPreKey = sizeof(K) == 4 && (!kRead || sizeof(V) == 4);
  static constexpr bool kPreVal = kRead && sizeof(V) == 4;
  static constexpr int kMinBlocks = sizeof(K) + (kRead ? sizeof(V) : 0) <= 8 && sizeof(K) == 4 ? 3 : 2;
  // shared bytes of one element: staged key, value and region, input buffers
  static constexpr size_t kElem = sizeof(K) + (kRead ? sizeof(V) : 0) + (kVals == kValsLocal ? 4 : 2) +
                                  (kPreKey ? sizeof(K) : 0) + (kPreVal ? sizeof(V) : 0);
  static constexpr size_t smem_bytes(uint32_t R, int tile) {
    return kElem * tile + 4 * (2ull * scan_cnt_words(R) + 2ull * scan_off_words(R) + kPartThreads / 32);
  }
};

template <class K, class V, int kVals = kValsRead, int kItems = kPartItems>
__global__ void __launch_bounds__(kPartThreads, (SplitTile<K, V, kVals>::kMinBlocks))
    k_part_scatter(const K* __restrict__ keys, const V* __restrict__ vals, uint64_t n, RegionMap m,
                   const unsigned int* __restrict__ hist, unsigned int* __restrict__ cursor, K* __restrict__ okeys,
                   V* __restrict__ ovals, uint2* __restrict__ runs, const unsigned long long* n_dev) {
  if (n_dev != nullptr) n = *n_dev;
  using Tile = SplitTile<K, V, kVals>;
  constexpr bool kPreKey = Tile::kPreKey, kPreVal = Tile::kPreVal, kPre = kPreKey || kPreVal, kRead = Tile::kRead;
  constexpr int kTile = kPartThreads * kItems;
  extern __shared__ __align__(16) unsigned long long scatter_smem[];
  char* at = reinterpret_cast<char*>(scatter_smem);
  auto carve = [&](size_t bytes) {
    char* p = at;
    at += bytes;
    return p;
  };
  // 4+4-byte pairs are staged together (one store and one load of 8 bytes)
  constexpr bool kPair = kRead && sizeof(K) == 4 && sizeof(V) == 4;
  uint2* s_pair = reinterpret_cast<uint2*>(at);
  K* s_key = reinterpret_cast<K*>(carve(sizeof(K) * kTile));
  V* s_val = reinterpret_cast<V*>(carve(kRead ? sizeof(V) * kTile : 0));
  K* in_key = reinterpret_cast<K*>(carve(kPreKey ? sizeof(K) * kTile : 0));
  V* in_val = reinterpret_cast<V*>(carve(kPreVal ? sizeof(V) * kTile : 0));
  using Reg = typename std::conditional<kVals == kValsLocal, uint32_t, uint16_t>::type;
  Reg* s_reg = reinterpret_cast<Reg*>(carve(sizeof(Reg) * kTile));  // region (<< 16 | position, with kValsLocal)
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(carve(4ull * scan_cnt_words(m.R)));
  uint32_t* s_off = reinterpret_cast<uint32_t*>(carve(4ull * scan_off_words(m.R)));   // start in the staged tile
  uint32_t* s_base = reinterpret_cast<uint32_t*>(carve(4ull * scan_off_words(m.R)));  // the region's start in the output
  uint32_t* s_delta = reinterpret_cast<uint32_t*>(carve(4ull * scan_cnt_words(m.R)));  // output place - staged place
  uint32_t* s_w = reinterpret_cast<uint32_t*>(carve(4ull * (kPartThreads / 32)));
  const uint32_t nn = static_cast<uint32_t>(n);  // n < 2^32: places and counts are 32 bits
  const uint32_t ntiles = static_cast<uint32_t>((n + kTile - 1) / kTile);
  // copy tile `tl`'s input into the input buffer
  auto prefetch = [&](uint32_t tl) {
    const uint32_t b = tl * kTile;
    const uint32_t cnt = nn - b < kTile ? nn - b : kTile;
    for (uint32_t i = threadIdx.x; i < cnt; i += kPartThreads) {
      if constexpr (kPreKey) cp_async_elem(in_key + i, keys + b + i);
      if constexpr (kPreVal) cp_async_elem(in_val + i, vals + b + i);
    }
  };
  if constexpr (kPre) {
    if (blockIdx.x < ntiles) prefetch(blockIdx.x);
  }
  // region bases: exclusive prefix of the histogram (every block recomputes it)
  for (uint32_t i = threadIdx.x; i < scan_cnt_words(m.R); i += kPartThreads) s_cnt[i] = i < m.R ? hist[i] : 0u;
  __syncthreads();
  scan_regions(s_cnt, s_base, m.R, s_w);
  for (uint32_t i = threadIdx.x; i < m.R; i += kPartThreads) s_cnt[i] = 0;
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint32_t t0 = tile * kTile;
    const uint32_t tn = nn - t0 < kTile ? nn - t0 : kTile;
    if constexpr (kPre) cp_async_wait_all();  // this tile's input is in shared memory
    __syncthreads();
    K kk[kPreKey ? 1 : kItems];
    V vv[kPreVal || !kRead ? 1 : kItems];
    uint32_t rr[kItems];  // region << 16 | rank (a tile holds fewer than 2^16 elements)
    if constexpr (!kPreKey || (kRead && !kPreVal)) {
#pragma unroll
      for (int k = 0; k < kItems; ++k) {
        const uint32_t i = k * kPartThreads + threadIdx.x;
        if constexpr (!kPreKey) kk[k] = i < tn ? ldg_stream(keys + t0 + i) : K(0);
        if constexpr (kRead && !kPreVal) vv[k] = i < tn ? ldg_stream(vals + t0 + i) : V(0);
      }
    }
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const uint32_t i = k * kPartThreads + threadIdx.x;
      if (i < tn) {
        uint32_t r;
        if constexpr (kPreKey) r = m.of(in_key[i]);
        else r = m.of(kk[k]);
        rr[k] = r << 16 | atomicAdd(s_cnt + r, 1u);
      }
    }
    __syncthreads();
    scan_regions(s_cnt, s_off, m.R, s_w);
    for (uint32_t r = threadIdx.x; r < m.R; r += kPartThreads) {
      const uint32_t before = s_off[r], c = s_cnt[r];
      const uint32_t p = c ? s_base[r] + atomicAdd(cursor + r, c) : 0u;
      s_delta[r] = p - before;
      if constexpr (kVals == kValsLocal) runs[static_cast<uint64_t>(tile) * m.R + r] = make_uint2(p, before);
    }
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const uint32_t i = k * kPartThreads + threadIdx.x;
      if (i < tn) {
        const uint32_t r = rr[k] >> 16, o = s_off[r] + (rr[k] & 0xffffu);
        if constexpr (kPair) {
          s_pair[o] = make_uint2(in_key[i], in_val[i]);
        } else {
          if constexpr (kPreKey) s_key[o] = in_key[i];
          else s_key[o] = kk[k];
          if constexpr (kPreVal) s_val[o] = in_val[i];
          else if constexpr (kRead) s_val[o] = vv[k];
        }
        if constexpr (kVals == kValsLocal) s_reg[o] = r << 16 | i;
        else s_reg[o] = static_cast<Reg>(r);
      }
    }
    __syncthreads();
    // the input buffer and the counters are free again
    if constexpr (kPre) {
      if (ntiles - tile > gridDim.x) prefetch(tile + gridDim.x);
    }
    for (uint32_t i = threadIdx.x; i < m.R; i += kPartThreads) s_cnt[i] = 0;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < tn; i += kPartThreads) {
      const uint32_t x = s_reg[i];
      const uint32_t o = s_delta[kVals == kValsLocal ? x >> 16 : x] + i;
      if (o < nn) {  // always true when hist holds this batch's counts
        if constexpr (kPair) {
          const uint2 p = s_pair[i];
          okeys[o] = p.x;
          ovals[o] = p.y;
        } else {
          okeys[o] = s_key[i];
          if constexpr (kVals == kValsLocal) ovals[o] = static_cast<V>(x & 0xffffu);
          else if constexpr (kRead) ovals[o] = s_val[i];
        }
      }
    }
  }
  if constexpr (kPre) cp_async_wait_all();
}

// ---- host side -------------------------------------------------------------------------
// A batch split by table region in the table's scratch buffer, plus kSplitCounters zeroed
// chunk counters for the ordered sweeps of the kernels that consume it, and `extra` bytes
// the caller asked for.
constexpr int kSplitCounters = 32;
constexpr uint64_t kSplitHist = 0, kSplitCursor = 8192, kSplitCnt = 16384, kSplitHeader = 16640;
static_assert(kMaxSplitRegions * sizeof(unsigned int) <= kSplitCursor - kSplitHist, "hist area");
static_assert(kMaxSplitRegions * sizeof(unsigned int) <= kSplitCnt - kSplitCursor, "cursor area");
static_assert(kSplitCounters * sizeof(unsigned long long) <= kSplitHeader - kSplitCnt, "counter area");

template <class K, class V>
struct RegionSplit {
  const K* keys;
  const V* vals;
  const unsigned int* hist;  // keys of every region
  unsigned long long* counters;
  char* extra;  // `extra` bytes, 256-byte aligned (not zeroed)
};

inline uint64_t align256(uint64_t x) { return (x + 255) / 256 * 256; }

// The two kernels of a split: hist and cursor are m.R zeroed words each.  n_dev (or null): the
// batch's size on the device, at most n.
template <class K, class V, int kVals = kValsRead, int kItems = kPartItems>
cudaError_t split_launch(const wc_table* t, const RegionMap& m, const K* keys, const V* vals, uint64_t n,
                         unsigned int* hist, unsigned int* cursor, K* okeys, V* ovals, uint2* runs, cudaStream_t s,
                         const unsigned long long* n_dev = nullptr) {
  auto hk = k_part_hist<K>;
  auto sk = k_part_scatter<K, V, kVals, kItems>;
  using Tile = SplitTile<K, V, kVals>;
  constexpr int kTile = kPartThreads * kItems;
  const uint32_t copies = hist_copies(m.R);
  const size_t hsm = static_cast<size_t>(copies) * m.R * sizeof(unsigned int);
  const size_t ssm = Tile::smem_bytes(m.R, kTile);
  static_assert(kHistWarps * 512 * 4 <= 48 << 10, "the histogram needs no raised limit");
  const cudaError_t attr = allow_smem(sk, Tile::smem_bytes(kMaxSplitRegions, kTile));
  if (attr != cudaSuccess) return attr;
  const uint64_t hist_most = static_cast<uint64_t>(occupancy_smem(hk, kPartThreads, hsm)) * t->sm_count;
  const uint64_t split_most = static_cast<uint64_t>(occupancy_smem(sk, kPartThreads, ssm)) * t->sm_count;
  const unsigned hg = static_cast<unsigned>(std::min<uint64_t>((n + kPartTile - 1) / kPartTile, hist_most));
  const unsigned sg = static_cast<unsigned>(std::min<uint64_t>((n + kTile - 1) / kTile, split_most));
  hk<<<hg, kPartThreads, hsm, s>>>(keys, n, m, hist, copies, n_dev);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;  // no split without its counts
  sk<<<sg, kPartThreads, ssm, s>>>(keys, vals, n, m, hist, cursor, okeys, ovals, runs, n_dev);
  return cudaGetLastError();
}

// Regions of m.  Scratch layout: [header kSplitHeader B | keys | vals | extra], grown on
// demand.  kVals: where the values come from (kValsLocal: uint16 positions inside the tile,
// run starts to extra + runs_at).  The caller hands the scratch on with scratch_release.
template <class K, class V, int kVals = kValsRead, int kItems = kPartItems>
cudaError_t region_split(const wc_table* t, const RegionMap& m, const K* keys, const V* vals, uint64_t n,
                         cudaStream_t s, RegionSplit<K, V>& out, uint64_t extra = 0, uint64_t runs_at = 0,
                         const unsigned long long* n_dev = nullptr) {
  const uint64_t keys_off = kSplitHeader;
  const uint64_t vals_off = keys_off + align256(n * sizeof(K));
  const uint64_t extra_off = vals_off + (kVals == kValsNone ? 0 : align256(n * sizeof(V)));
  char* sc = nullptr;
  cudaError_t e = ensure_scratch(t, extra_off + extra, s, &sc, lookup_scratch_likely(t, n));
  if (e != cudaSuccess) return e;
  out.keys = reinterpret_cast<K*>(sc + keys_off);
  out.vals = kVals == kValsNone ? nullptr : reinterpret_cast<V*>(sc + vals_off);
  auto* hist = reinterpret_cast<unsigned int*>(sc + kSplitHist);
  out.hist = hist;
  out.counters = reinterpret_cast<unsigned long long*>(sc + kSplitCnt);
  out.extra = sc + extra_off;
  e = cudaMemsetAsync(sc, 0, kSplitHeader, s);
  if (e != cudaSuccess) return e;
  return split_launch<K, V, kVals, kItems>(t, m, keys, vals, n, hist,
                                           reinterpret_cast<unsigned int*>(sc + kSplitCursor), const_cast<K*>(out.keys),
                                           const_cast<V*>(out.vals), reinterpret_cast<uint2*>(out.extra + runs_at), s,
                                           n_dev);
}

}  // namespace wc
