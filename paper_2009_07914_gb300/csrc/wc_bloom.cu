// Bloom filters (the paper's BloomFilter: set membership with false positives), blocked
// for the GPU: a key owns one 256-bit block (32 bytes, one sector) chosen by its hash and
// sets k bits inside it, so an insert is at most four atomic ORs into one sector and a lookup
// is one 32-byte read.
//   h = fmix64(key ^ seed); block = floor(hi32(h) * blocks / 2^32);
//   bit positions: bytes 0..7 of g1 = fmix64(h ^ 0x9e3779b97f4a7c15), then bytes of
//   g2 = fmix64(g1), ... (position i = byte i % 8 of g_{i / 8 + 1}); bits may coincide.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "wc.h"
#include "wc_device.cuh"
#include "wc_internal.h"
#include "wc_launch.cuh"
#include "wc_lookup.cuh"
#include "wc_partition.cuh"

namespace wc {
namespace {

// The key's hash; its block is the high half scaled to the filter (RegionMap's first window).
__device__ __forceinline__ uint64_t bloom_hash(uint64_t key, uint64_t seed) { return fmix64(key ^ seed); }
__device__ __forceinline__ uint32_t bloom_block(uint64_t h, uint32_t blocks) {
  return __umulhi(static_cast<uint32_t>(h >> 32), blocks);
}

// Calls bit(pos) for the key's k bit positions 0..255.
template <class Bit>
__device__ __forceinline__ void bloom_bits(uint64_t h, int k, Bit bit) {
  uint64_t g = h ^ 0x9e3779b97f4a7c15ull;
  for (int i = 0; i < k; i += 8) {
    g = fmix64(g);
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if (i + b < k) bit(static_cast<uint32_t>(g >> (8 * b)) & 255u);
  }
}

// Calls at(i) for the batch's positions: strided over the grid, or (counter != nullptr) in
// order, a warp taking 512 at a time (a batch split by filter region then finds the region's
// blocks in L2).
template <class At>
__device__ __forceinline__ void for_batch(uint64_t n, unsigned long long* counter, At at) {
  if (counter == nullptr) {
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) at(i);
    return;
  }
  const uint32_t lane = threadIdx.x & 31;
  while (true) {
    unsigned long long c = 0;
    if (lane == 0) c = atomicAdd(counter, 512ull);
    c = __shfl_sync(kFull, c, 0);
    if (c >= n) break;
    const uint64_t end = n - c < 512 ? n : c + 512;
#pragma unroll 4
    for (uint64_t i = c + lane; i < end; i += 32) at(i);
  }
}

// Every key's bits by atomic ORs on 64-bit words: at most four per key (32-bit words took
// up to eight; at k = 7 about 3.5 against 4.9).  The L2's atomics bound it: 2^20 keys of a
// 1.2 MiB filter 37.8 G/s, 2^26 of 80 MiB 57.7; 20.7 with 32-bit words.
template <class K>
__global__ void __launch_bounds__(256) k_bloom_insert(TableDesc t, const K* __restrict__ keys, uint64_t n, int k,
                                                      unsigned long long* counter) {
  auto* bits = static_cast<unsigned long long*>(t.slots);
  uint32_t flags = 0;
  long long added = 0;
  for_batch(n, counter, [&](uint64_t i) {
    const K key = ldg_stream(keys + i);
    if (key == K(0) || key == K(~K(0))) {
      flags |= kFlagInvalid;
      return;
    }
    const uint64_t h = bloom_hash(static_cast<uint64_t>(key), t.seed);
    unsigned long long m0 = 0, m1 = 0, m2 = 0, m3 = 0;
    bloom_bits(h, k, [&](uint32_t pos) {
      const unsigned long long x = 1ull << (pos & 63u);
      const uint32_t w = pos >> 6;
      if (w == 0) m0 |= x;
      if (w == 1) m1 |= x;
      if (w == 2) m2 |= x;
      if (w == 3) m3 |= x;
    });
    unsigned long long* b = bits + static_cast<uint64_t>(bloom_block(h, t.p)) * 4;
    if (m0) atomicOr(b, m0);
    if (m1) atomicOr(b + 1, m1);
    if (m2) atomicOr(b + 2, m2);
    if (m3) atomicOr(b + 3, m3);
    ++added;
  });
  flush_flags(t.status, flags);
  flush_delta(t.size, added);
}

// Insert of a batch split by filter region: a block sets the bits of a region's keys in a
// copy of the region in shared memory (a shared OR per bit) and then ORs the copy's
// non-zero words into the filter, consecutive threads on consecutive words -- one global
// atomic per word of the region instead of 3.5 per key on random words.  A region of many
// keys (a skewed batch) is worked on in parts of at most `part` keys, each with a copy of
// its own, so no block is left with a hot key's share.  Concurrent inserts stay correct:
// the filter only ever changes by ORs.  2^27 keys of a 160 MiB filter, k = 7: 0.93 ms (1.60
// with 512 threads: one block of a 128 KiB region fills an SM), 1.73 ms with the split,
// against 3.89 ms by k_bloom_insert and 6.65 ms with its former 32-bit words.
// A part is at most kFillPart keys, so its size and the parts' number stay far below 2^32
// for any batch, and a filter of one region is still filled by many blocks (the unit words
// are 32 bits wide; a batch has up to 2^32 - 1 keys).
constexpr int kFillThreads = 1024;
constexpr uint64_t kFillPart = 1ull << 20;
constexpr uint32_t fill_words(uint32_t R) { return scan_cnt_words(R) + 2 * scan_off_words(R); }

template <class K>
__global__ void __launch_bounds__(kFillThreads) k_bloom_fill(TableDesc t, const K* __restrict__ keys, RegionMap m,
                                                             const unsigned int* __restrict__ hist, uint32_t part,
                                                             unsigned long long* next_unit, int k) {
  extern __shared__ __align__(16) unsigned long long fill_smem[];
  const uint32_t words = 4u << m.shift;  // 64-bit words of a region
  unsigned long long* s_bits = fill_smem;
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(fill_smem + words);
  uint32_t* s_off = s_cnt + scan_cnt_words(m.R);   // first key of every region
  uint32_t* s_unit = s_off + scan_off_words(m.R);  // first unit of every region (part, region)
  __shared__ uint32_t s_w[kFillThreads / 32];  // scan_regions: the first kPartThreads threads do the work
  __shared__ unsigned long long s_next;
  for (uint32_t r = threadIdx.x; r < scan_cnt_words(m.R); r += kFillThreads) s_cnt[r] = r < m.R ? hist[r] : 0u;
  __syncthreads();
  scan_regions(s_cnt, s_off, m.R, s_w);
  for (uint32_t r = threadIdx.x; r < m.R; r += kFillThreads)
    if (s_cnt[r] != 0) s_cnt[r] = (s_cnt[r] - 1) / part + 1;
  __syncthreads();
  scan_regions(s_cnt, s_unit, m.R, s_w);
  const uint32_t units = s_unit[m.R];
  uint32_t flags = 0;
  long long added = 0;
  while (true) {
    if (threadIdx.x == 0) s_next = atomicAdd(next_unit, 1ull);
    for (uint32_t i = threadIdx.x; i < words; i += kFillThreads) s_bits[i] = 0;
    __syncthreads();
    if (s_next >= units) break;
    const uint32_t u = static_cast<uint32_t>(s_next);
    uint32_t lo = 0, hi = m.R - 1;  // the last region starting at or before unit u (an empty one has no unit)
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (s_unit[mid] <= u) lo = mid;
      else hi = mid - 1;
    }
    const uint32_t len = hist[lo], done = (u - s_unit[lo]) * part;
    const uint32_t cnt = len - done < part ? len - done : part;
    const K* in = keys + s_off[lo] + done;
    auto* b32 = reinterpret_cast<uint32_t*>(s_bits);
    const uint32_t mask = (1u << m.shift) - 1u;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < cnt; i += kFillThreads) {
      const K key = ldg_stream(in + i);
      if (key == K(0) || key == K(~K(0))) {
        flags |= kFlagInvalid;
        continue;
      }
      const uint64_t h = bloom_hash(static_cast<uint64_t>(key), t.seed);
      const uint32_t b = (bloom_block(h, t.p) & mask) * 8;
      bloom_bits(h, k, [&](uint32_t pos) { atomicOr(b32 + b + (pos >> 5), 1u << (pos & 31u)); });
      ++added;
    }
    __syncthreads();
    const uint64_t w0 = static_cast<uint64_t>(lo) * words, end = static_cast<uint64_t>(t.p) * 4;
    auto* bits = static_cast<unsigned long long*>(t.slots);
    for (uint32_t i = threadIdx.x; i < words; i += kFillThreads) {
      const unsigned long long x = s_bits[i];
      if (x != 0 && w0 + i < end) atomicOr(bits + w0 + i, x);
    }
    __syncthreads();
  }
  flush_flags(t.status, flags);
  flush_delta(t.size, added);
}

// Membership: one 32-byte read per key, its k bits picked from the eight words by selects
// (building the 256-bit mask of the key first took twice the instructions, which bound the
// kernel: 2^27 keys over 160 MiB 26.2 -> 91 G/s).
template <class K>
__global__ void __launch_bounds__(256) k_bloom_contains(TableDesc t, const K* __restrict__ keys, uint64_t n, int k,
                                                        uint8_t* __restrict__ found, unsigned long long* counter) {
  const unsigned long long* bits = static_cast<const unsigned long long*>(t.slots);
  uint32_t flags = 0;
  for_batch(n, counter, [&](uint64_t i) {
    const K key = ldg_stream(keys + i);
    if (key == K(0) || key == K(~K(0))) {
      flags |= kFlagInvalid;
      found[i] = 0;
      return;
    }
    const uint64_t h = bloom_hash(static_cast<uint64_t>(key), t.seed);
    unsigned long long u[4];
    ldcg4(bits + static_cast<uint64_t>(bloom_block(h, t.p)) * 4, u);
    uint32_t all = 1;
    bloom_bits(h, k, [&](uint32_t pos) {
      const unsigned long long a = pos & 64u ? u[1] : u[0], b = pos & 64u ? u[3] : u[2];
      const unsigned long long x = pos & 128u ? b : a;
      const uint32_t y = pos & 32u ? static_cast<uint32_t>(x >> 32) : static_cast<uint32_t>(x);
      all &= y >> (pos & 31u);
    });
    found[i] = all & 1u;
  });
  flush_flags(t.status, flags);
}

// Inserts are split where the shared-memory copies save more global atomics than merging
// them takes: k = 7, 10 bits per key, in input order against split, 2^22 keys 79.8 / 119.7
// us, 2^24 287 / 278, 2^26 (80 MiB) 1164 / 976, 2^27 (160 MiB) 3892 / 1730.  A copy is merged
// whatever the batch, so a batch below a quarter key per byte of the filter stays in order.
// Filters of more regions than a split takes (above 256 MiB) are swept by k_bloom_insert
// over a split into L2-sized regions (2^28 keys, 320 MiB: 11.7 ms in input order).
template <class K>
cudaError_t insert(const wc_table* t, const K* keys, uint64_t n, cudaStream_t s) {
  const int k = t->cfg.window_width;
  auto direct = k_bloom_insert<K>;
  const uint64_t most = static_cast<uint64_t>(occupancy(direct, 256)) * t->sm_count;
  if (n >= (1ull << 24) && n >= t->table_bytes / 4 && !stream_capturing(s)) {
    // regions of a power of two of blocks, at most 128 KiB, about a thousand of them
    RegionMap m;
    m.seed = t->cfg.seed;
    m.p = static_cast<uint32_t>(t->windows);
    m.shift = 5;
    while (m.shift < 12 && (t->windows - 1) >> m.shift >= 1536) ++m.shift;
    m.R = static_cast<uint32_t>(((t->windows - 1) >> m.shift) + 1);
    const bool fill = m.R <= kMaxSplitRegions;
    if (!fill) m = region_map(t, 0);
    RegionSplit<K, K> sp;
    cudaError_t e = region_split<K, K, kValsNone, 16>(t, m, keys, nullptr, n, s, sp);
    if (e == cudaSuccess) {
      if (fill) {
        auto kern = k_bloom_fill<K>;
        const size_t smem = (32ull << m.shift) + fill_words(m.R) * 4;
        const cudaError_t attr = allow_smem(kern, (32 << 12) + fill_words(kMaxSplitRegions) * 4);
        const uint64_t part = std::min(std::max<uint64_t>(4 * (n / m.R + 1), 4ull << m.shift), kFillPart);
        const unsigned grid = static_cast<unsigned>(occupancy_smem(kern, kFillThreads, smem) * t->sm_count);
        e = attr != cudaSuccess ? attr
                                : launch_k(t, kern, grid, kFillThreads, smem, s, desc_of(t), sp.keys, m, sp.hist,
                                           static_cast<uint32_t>(part), sp.counters, k);
      } else {
        e = launch_k(t, direct, static_cast<unsigned>(most), 256u, 0, s, desc_of(t), sp.keys, n, k, sp.counters);
      }
      const cudaError_t r = scratch_release(t, s);
      return e != cudaSuccess ? e : r;
    }
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();  // no room for the split: set the bits in input order
  }
  const uint64_t want = (n + 255) / 256;
  return launch_k(t, direct, static_cast<unsigned>(want < most ? want : most), 256u, 0, s, desc_of(t), keys, n, k,
                  static_cast<unsigned long long*>(nullptr));
}

// Queries are split where the filter no longer fits L2: in input order against split, 2^27
// queries over 160 MiB 1.48 / 1.79 ms, 2^28 over 320 MiB 4.92 / 3.54 ms.
template <class K>
cudaError_t contains(const wc_table* t, const K* keys, uint64_t n, uint8_t* found, cudaStream_t s) {
  const int k = t->cfg.window_width;
  auto kern = k_bloom_contains<K>;
  const uint64_t most = static_cast<uint64_t>(occupancy(kern, 256)) * t->sm_count;
  if (t->table_bytes > (224ull << 20) && n >= t->table_bytes / 32 && !stream_capturing(s)) {
    QuerySplit<K, uint8_t> q;
    cudaError_t e = query_split(t, 0, keys, n, s, q);
    if (e == cudaSuccess) {
      e = launch_k(t, kern, static_cast<unsigned>(most), 256u, 0, s, desc_of(t), q.sp.keys, n, k, q.rf, q.sp.counters);
      if (e == cudaSuccess) e = unsplit_launch(t, q, n, static_cast<uint8_t*>(nullptr), found, s);
      const cudaError_t r = scratch_release(t, s);
      return e != cudaSuccess ? e : r;
    }
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();  // no room for the split: query in input order
  }
  const uint64_t want = (n + 255) / 256;
  return launch_k(t, kern, static_cast<unsigned>(want < most ? want : most), 256u, 0, s, desc_of(t), keys, n, k, found,
                  static_cast<unsigned long long*>(nullptr));
}

}  // namespace

// op: WC_OP_INSERT (set the keys' bits) or WC_OP_RETRIEVE (membership into found).
cudaError_t bloom_launch(const wc_table* t, int op, const void* keys, uint64_t n, uint8_t* found, cudaStream_t s) {
  if (t->cfg.key_bytes == 4) {
    const auto* k = static_cast<const uint32_t*>(keys);
    return op == WC_OP_INSERT ? insert(t, k, n, s) : contains(t, k, n, found, s);
  }
  const auto* k = static_cast<const unsigned long long*>(keys);
  return op == WC_OP_INSERT ? insert(t, k, n, s) : contains(t, k, n, found, s);
}

}  // namespace wc
