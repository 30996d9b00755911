// Instantiation and dispatch of the open-addressing multi-value kernels for one slot
// layout.  Ops: WC_OP_INSERT (append), WC_OP_COUNT (per-query counts; the caller scans),
// WC_OP_RETRIEVE (CSR write of the matches), WC_OP_ERASE (tombstone every copy).
#pragma once

#include "wc_launch.cuh"
#include "wc_mvoa_kernels.cuh"
#include "wc_partition.cuh"

namespace wc {

template <class L, int G, int S>
cudaError_t oa_run(const wc_table* t, int op, const void* keys, const void* vals, uint64_t n, uint64_t* offs,
                   void* out, cudaStream_t s) {
  using Key = typename L::Key;
  using Val = typename L::Val;
  const wc_launch& lc = t->launch[op];
  const int block = lc.block_threads;
  TableDesc d = desc_of(t);
  // A count recorded into a graph does not use the walk bits: between its replays the slots may
  // be handed to a user kernel, which sets none (recorded inserts do set them).
  d.ovf = t->walk_off || (op == WC_OP_COUNT && stream_capturing(s)) ? nullptr : t->d_walk;
  const Key* k = static_cast<const Key*>(keys);
  constexpr int W = G * S;
  if (op == WC_OP_INSERT) {
    const Val* v = static_cast<const Val*>(vals);
    // Swept batches run one pair per thread; batches in input order stay on the group engine,
    // whose copies of a key get in each other's way less (2^20 pairs, 1 / 4 / 16 per key: 51.7
    // / 62.3 / 91.1 us against 52.3 / 68.4 / 104; swept, 2^24: 558 / 641 / 1008 against 504 /
    // 583 / 854).
    auto put = [&](const Key* pk, const Val* pv, unsigned long long* counter) {
      if constexpr (lookup_window<L>(W)) {
        if (counter != nullptr) {
          auto kern = k_oa_put<L, W>;
          const unsigned grid = static_cast<unsigned>(occupancy(kern, kLookThreads) * t->sm_count);
          return launch_k(t, kern, grid, kLookThreads, 0, s, d, pk, pv, n, counter);
        }
      }
      auto kern = k_oa_insert<L, G, S>;
      const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
      const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
      const unsigned grid =
          counter != nullptr ? static_cast<unsigned>(bps) * static_cast<unsigned>(t->sm_count) : g.blocks;
      return launch_k(t, kern, grid, block, 0, s, d, pk, pv, n, g.per_warp, counter,
                      counter != nullptr ? kLookChunk : 0u);
    };
    if (scheme_for(t, op, n) != WC_SCHEME_BLOCKED) return put(k, v, nullptr);
    RegionSplit<Key, Val> sp;
    cudaError_t e = region_split(t, region_map(t, lc.region_mib), k, v, n, s, sp);
    if (e == cudaSuccess) e = put(sp.keys, sp.vals, sp.counters);
    const cudaError_t r = scratch_release(t, s);
    return e != cudaSuccess ? e : r;
  }
  if constexpr (lookup_window<L>(W)) {
    if (op == WC_OP_COUNT) {
      // split by region like lookups (lookup_splits): counts of 32 bits, widened on the way back
      if (lookup_splits(t, n) && !stream_capturing(s)) {
        QuerySplit<Key, uint32_t> q;
        cudaError_t e = query_split(t, 0, k, n, s, q);
        if (e == cudaSuccess) {
          auto kern = k_oa_count<L, W, uint32_t>;
          const unsigned grid = static_cast<unsigned>(occupancy(kern, kLookThreads) * t->sm_count);
          e = launch_k(t, kern, grid, kLookThreads, 0, s, d, q.sp.keys, n, q.sp.counters, q.rv);
          if (e == cudaSuccess) e = unsplit_launch<Key, uint32_t, uint64_t>(t, q, n, offs, nullptr, s);
          const cudaError_t r = scratch_release(t, s);
          return e != cudaSuccess ? e : r;
        }
        if (e != cudaErrorMemoryAllocation) return e;
        cudaGetLastError();  // no room for the split: count in input order
      }
      auto kern = k_oa_count<L, W, uint64_t>;
      const uint64_t want = (n + kLookThreads - 1) / kLookThreads;
      const uint64_t most = static_cast<uint64_t>(occupancy(kern, kLookThreads)) * t->sm_count;
      return launch_k(t, kern, static_cast<unsigned>(std::min(want, most)), kLookThreads, 0, s, d, k, n,
                      static_cast<unsigned long long*>(nullptr), offs);
    }
  }
  if (op == WC_OP_COUNT || op == WC_OP_RETRIEVE) {
    auto kern = k_oa_walk<L, G, S, true>;
    if constexpr (!lookup_window<L>(W))
      if (op == WC_OP_COUNT) kern = k_oa_walk<L, G, S, false>;
    const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
    const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
    return launch_k(t, kern, g.blocks, block, 0, s, d, k, n, offs, static_cast<Val*>(out));
  }
  auto kern = k_oa_erase<L, G, S>;
  const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
  const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
  return launch_k(t, kern, g.blocks, block, 0, s, d, k, n);
}

// Distinct live keys into the table's nkeys word (zeroed first).
template <class L>
cudaError_t oa_count_keys(const wc_table* t, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(t->d_nkeys, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  auto kern = k_oa_num_keys<L>;
  const uint64_t want = (t->capacity + 255) / 256;
  const uint64_t most = static_cast<uint64_t>(occupancy(kern, 256)) * t->sm_count;
  const unsigned grid = static_cast<unsigned>(want < most ? want : most);
  return launch_k(t, kern, grid, 256u, 0, s, desc_of(t), t->capacity);
}

}  // namespace wc

#define WC_OA_CASE(L, Wv, Gv) \
  if (W == (Wv) && G == (Gv)) return oa_run<L, (Gv), (Wv) / (Gv)>(t, op, keys, vals, n, offs, out, s);
