// Instantiation and dispatch of the single-value kernels for one slot layout.
#pragma once

#include "wc_insert.cuh"
#include "wc_launch.cuh"
#include "wc_lookup.cuh"
#include "wc_partition.cuh"
#include "wc_sv_kernels.cuh"

namespace wc {

// Retrieve by the blocked scheme: split the queries by table region, probe region by region
// in L2 with the results in split order, and put them back in input order tile by tile.
template <class L, int G, int S, int H = 1>
cudaError_t sv_retrieve_blocked(const wc_table* t, const wc_launch& lc, const typename L::Key* k, uint64_t n,
                                typename L::Val* out, uint8_t* found, cudaStream_t s) {
  using Key = typename L::Key;
  using Val = typename L::Val;
  constexpr int W = G * S * H;
  QuerySplit<Key, Val> q;
  cudaError_t e = query_split(t, lc.region_mib, k, n, s, q);
  if (e != cudaSuccess) return e;
  Val* rv = out != nullptr ? q.rv : nullptr;
  uint8_t* rf = found != nullptr ? q.rf : nullptr;
  if constexpr (lookup_window<L>(W)) {
    e = lookup_launch<L, W>(t, q.sp.keys, n, q.sp.counters, EmitLookup<L>{rv, rf, t->d_vals}, s);
  } else {
    auto kern = k_sv_retrieve<L, G, S, H>;
    const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, lc.block_threads);
    e = launch_k(t, kern, static_cast<unsigned>(bps) * static_cast<unsigned>(t->sm_count), lc.block_threads, 0, s,
                 desc_of(t), q.sp.keys, n, static_cast<uint64_t>(0), rv, rf, q.sp.counters, kLookChunk);
  }
  if (e == cudaSuccess) e = unsplit_launch(t, q, n, out, found, s);
  const cudaError_t r = scratch_release(t, s);
  return e != cudaSuccess ? e : r;
}

// The insert kernel of a window: counter != nullptr for a batch split by region.  n_dev (one
// key per thread only, or null): the batch's size on the device, at most n.
template <class L, int G, int S, int H = 1>
cudaError_t insert_kernel(const wc_table* t, const typename L::Key* keys, const typename L::Val* vals, uint64_t n,
                          unsigned long long* counter, cudaStream_t s, const unsigned long long* n_dev = nullptr) {
  if constexpr (lookup_window<L>(G * S * H)) {
    return insert_launch<L, G * S * H>(t, keys, vals, n, counter, n_dev, s);
  } else {
    const wc_launch& lc = t->launch[WC_OP_INSERT];
    auto kern = k_sv_insert<L, G, S, H>;
    const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, lc.block_threads);
    const EngineGrid g = engine_grid(n, G, lc.block_threads, bps, t->sm_count);
    const unsigned grid =
        counter != nullptr ? static_cast<unsigned>(bps) * static_cast<unsigned>(t->sm_count) : g.blocks;
    return launch_k(t, kern, grid, lc.block_threads, 0, s, desc_of(t), keys, vals, n, g.per_warp, counter,
                    counter != nullptr ? kLookChunk : 0u);
  }
}

// Insert (direct, or the blocked scheme: split the batch by table region, then insert it
// region by region).  vals == nullptr (counting tables): every key counts 1.
template <class L, int G, int S, int H = 1>
cudaError_t sv_insert_op(const wc_table* t, const void* keys, const void* vals, uint64_t n, cudaStream_t s,
                         const unsigned long long* n_dev = nullptr) {
  using Key = typename L::Key;
  using Val = typename L::Val;
  constexpr int W = G * S * H;
  const wc_launch& lc = t->launch[WC_OP_INSERT];
  const Key* k = static_cast<const Key*>(keys);
  const Val* v = static_cast<const Val*>(vals);
  if (scheme_for(t, WC_OP_INSERT, n) != WC_SCHEME_BLOCKED) return insert_kernel<L, G, S, H>(t, k, v, n, nullptr, s, n_dev);
  RegionSplit<Key, Val> sp;
  const RegionMap m = region_map(t, lc.region_mib);
  cudaError_t e = v != nullptr ? region_split(t, m, k, v, n, s, sp, 0, 0, n_dev)
                               : region_split<Key, Val, kValsNone>(t, m, k, nullptr, n, s, sp, 0, 0, n_dev);
  if (e == cudaSuccess) e = insert_kernel<L, G, S, H>(t, sp.keys, sp.vals, n, sp.counters, s, n_dev);
  const cudaError_t r = scratch_release(t, s);
  return e != cudaSuccess ? e : r;
}

// H > 1: a window of G * S * H slots is walked in H steps of G * S slots.
template <class L, int G, int S, int H = 1>
cudaError_t sv_run(const wc_table* t, int op, const void* keys, const void* vals, uint64_t n, void* out,
                   uint8_t* found, cudaStream_t s) {
  using Key = typename L::Key;
  using Val = typename L::Val;
  if (op == WC_OP_INSERT) return sv_insert_op<L, G, S, H>(t, keys, vals, n, s);
  const wc_launch& lc = t->launch[op];
  const int block = lc.block_threads;
  const TableDesc d = desc_of(t);
  const Key* k = static_cast<const Key*>(keys);
  if (op == WC_OP_RETRIEVE) {
    const int scheme = lookup_scheme(t, n, s);
    Val* o = static_cast<Val*>(out);
    if (scheme == WC_SCHEME_BLOCKED) {
      const cudaError_t e = sv_retrieve_blocked<L, G, S, H>(t, lc, k, n, o, found, s);
      if (e != cudaErrorMemoryAllocation || lc.scheme == WC_SCHEME_BLOCKED) return e;
      cudaGetLastError();  // no room for the split: probe in input order
    }
    if (scheme == WC_SCHEME_DEDUP) {
      auto kern = k_sv_retrieve_dedup<L, G, S, H>;
      const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
      const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
      return launch_k(t, kern, g.blocks, block, 0, s, d, k, n, g.per_warp, o, found);
    }
    if constexpr (lookup_window<L>(G * S * H)) {
      return lookup_launch<L, G * S * H>(t, k, n, nullptr, EmitLookup<L>{o, found, t->d_vals}, s);
    } else {
      // two keys per group: windows of at most 32 bytes per lane (register budget)
      if constexpr (S * L::kWords * 8 <= 32 || (L::kHalf && S * 4 <= 32))
        if (lc.keys_in_flight == 2) {
          auto kern = k_sv_retrieve2<L, G, S, H>;
          const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
          const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
          return launch_k(t, kern, g.blocks, block, 0, s, d, k, n, g.per_warp, o, found);
        }
      auto kern = k_sv_retrieve<L, G, S, H>;
      const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
      const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
      return launch_k(t, kern, g.blocks, block, 0, s, d, k, n, g.per_warp, o, found,
                      static_cast<unsigned long long*>(nullptr), 0u);
    }
  }
  auto kern = k_sv_erase<L, G, S, H>;
  const int bps = lc.blocks_per_sm > 0 ? lc.blocks_per_sm : occupancy(kern, block);
  const EngineGrid g = engine_grid(n, G, block, bps, t->sm_count);
  return launch_k(t, kern, g.blocks, block, 0, s, d, k, n, erase_chunk(g.per_warp));
}

}  // namespace wc

#define WC_SV_CASE(L, Wv, Gv)                                               \
  if (W == (Wv) && G == (Gv)) return sv_run<L, (Gv), (Wv) / (Gv)>(t, op, keys, vals, n, out, found, s);
// A window of Wv slots walked by Gv lanes in Hv steps.
#define WC_SV_CASE_H(L, Wv, Gv, Hv) \
  if (W == (Wv) && G == (Gv)) return sv_run<L, (Gv), (Wv) / (Gv) / (Hv), (Hv)>(t, op, keys, vals, n, out, found, s);
