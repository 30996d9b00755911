// Inserts into windows of at most 64 bytes: one pair per thread, straight-line, like the
// lookups of wc_lookup.cuh.
//
// Swept region by region (or into a table that fits L2) an insert is bound by the L2's rate
// of window reads followed by CASes (ldcg1 ff. in wc_device.cuh: 68 G/s at best) and by its
// chain of those two round trips.  The first window of a key takes most of them, so it is
// probed straight from the input; pairs that are not placed there (a full window, a slot lost
// to another pair and no other in the window) go to the warp's queue in shared memory and are
// worked on 32 at a time.  The claim rules are those of sv_insert_range (the group-per-key
// engine that wider windows run on): the earliest candidate of the key's sequence once the
// walk has met an empty slot or its end.
//
// The sweep of 2^27 pairs, one GB300, that engine against this kernel (with half-line
// reads): 4+4 bytes at load 0.9 with overflow bits 3.51 -> 2.97 ms (2.73 with the table
// copied to L2 ahead of the sweep, BatchBlocks::prefetch), at 0.5 3.11 -> 2.30; 8+8 bytes at
// 0.9 5.02 -> 4.35; sets of 8-byte keys at 0.9 4.6 -> 3.2.
//
// In input order it is races for slots that take the time: all pairs of a batch into a fresh
// table want the first slots of its windows at once.  A pair that loses one tries the next of
// the window with another CAS and nothing read in between; reading window and slot again for
// each lost race was slower than the group engine.  131,072 pairs of 4+4 bytes, load 0.6, that
// engine / read again / next slot 18.8 / 21.6 / 12.8 us, at 0.9 32.4 / 35.4 / 26.3; 2^20 at
// 0.9 55.9 / 53.3 / 48.7; 1000 at 0.6 14.8 / 15.2 / 8.6; sets of 8-byte keys, 222,476 at 0.9
// 34.7 / 39.7 / 31.2.
#pragma once

#include "wc_launch.cuh"
#include "wc_lookup.cuh"
#include "wc_sv_kernels.cuh"

namespace wc {

// What an insert needs to know of a window.
struct Spot {
  uint32_t at;    // slot of the key (hit)
  uint32_t tomb;  // first tombstone (has_tomb)
  uint32_t empty;  // first empty slot (see spot_word), W when there is none
  bool hit, has_tomb;
};

// S slots, the first of them slot `first` of the window, in one word: bit 0 the key is here,
// bit 1 a tombstone is, bits 2..7 the key's slot, 8..13 the first tombstone, 14.. the first
// empty slot, first + S when there is none.
// kCounted: the number of slots in use instead, plus `first` -- the same, as the empty slots
// are the last ones, but for a window that is read in two halves with other pairs claiming
// its slots in between: the count is then that of a slot which is taken by now.  It costs less
// (the sweep of 2^27 pairs of 4+4 bytes 3.58 against 3.70 ms with the split) and will do where
// one CAS is tried.
template <class L, int S, bool kCounted>
__device__ __forceinline__ uint32_t spot_word(const typename L::Slot (&s)[S], typename L::Key k, uint32_t first) {
  uint32_t hit = 0, tomb = 0, empty = kCounted ? first << 14 : (first + S) << 14;
#pragma unroll
  for (int i = S - 1; i >= 0; --i) {
    const typename L::Key kk = L::key(s[i]);
    if (kk == k) hit = 1u | (first + i) << 2;
    if (kk == L::kTomb) tomb = 2u | (first + i) << 8;
    if constexpr (kCounted) {
      if (kk != L::kEmpty) empty += 1u << 14;
    } else {
      if (kk == L::kEmpty) empty = (first + i) << 14;
    }
  }
  return hit | tomb | empty;
}

// Window w seen by the key k; every lane of the warp calls, with a window of the table.  As in
// probe_window, a pair of lanes reads a 64-byte window in one request.
template <class L, int W, bool kCounted>
__device__ __forceinline__ Spot spot_of(const typename L::Slot* slots, typename L::Key k, uint32_t w) {
  using Slot = typename L::Slot;
  uint32_t lo, hi = W << 14;  // the window's first half (or all of it), its second
  if constexpr (W * slot_size<L>() <= 32) {
    Slot s[W];
    load_slots<L, W, true>(slots + static_cast<uint64_t>(w) * W, s);
    lo = spot_word<L, W, kCounted>(s, k, 0);
  } else {
    constexpr int S = W / 2;
    const bool odd = threadIdx.x & 1;
    const uint32_t ow = __shfl_xor_sync(kFull, w, 1);
    const typename L::Key ok = __shfl_xor_sync(kFull, k, 1);
    const uint32_t half = odd ? S : 0;
    Slot sa[S], sb[S];  // my half of the even lane's window and of the odd lane's
    load_slots<L, S, true>(slots + static_cast<uint64_t>(odd ? ow : w) * W + half, sa);
    load_slots<L, S, true>(slots + static_cast<uint64_t>(odd ? w : ow) * W + half, sb);
    const uint32_t ma = spot_word<L, S, kCounted>(sa, odd ? ok : k, half);
    const uint32_t mb = spot_word<L, S, kCounted>(sb, odd ? k : ok, half);
    const uint32_t o = __shfl_xor_sync(kFull, odd ? ma : mb, 1);  // mine, as the other lane sees it
    lo = odd ? o : ma;
    hi = odd ? mb : o;
  }
  Spot r;
  r.hit = (lo | hi) & 1u;
  r.has_tomb = (lo | hi) & 2u;
  r.at = ((lo | hi) >> 2) & 63u;  // the key is in one half at most
  r.tomb = ((lo & 2u ? lo : hi) >> 8) & 63u;
  r.empty = lo >> 14;
  if (W * slot_size<L>() > 32 && r.empty == W / 2) r.empty = hi >> 14;
  return r;
}

template <class Key, class Val>
struct InsertQueue {
  Key key[kWarpQueue];
  Val val[kWarpQueue];
  uint32_t w[kWarpQueue], j[kWarpQueue];
  uint64_t tomb[kWarpQueue];
};

// The inserts of a warp's blocks; every lane calls.  vals == nullptr: every value is 1 (sets;
// counting tables without weights).  added: new keys stored by this lane.
template <class L, int W, bool kSwept>
__device__ __forceinline__ void insert_blocks(const TableDesc& t, const typename L::Key* __restrict__ keys,
                                              const typename L::Val* __restrict__ vals, BatchBlocks<kSwept>& blocks,
                                              InsertQueue<typename L::Key, typename L::Val>& q, uint32_t& flags,
                                              long long& added) {
  using Slot = typename L::Slot;
  using Key = typename L::Key;
  using Val = typename L::Val;
  // first tombstone of a walk: none; none, and the pair has lost a slot before; else its index
  constexpr uint64_t kNone = ~0ull, kLost = ~1ull;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  Slot* slots = static_cast<Slot*>(t.slots);
  uint32_t cnt = 0;

  // A pair on its walk: hash h, window w, the j-th of the sequence, `tomb` the first
  // tombstone met before it.
  struct Pair {
    Key k;
    Val v;
    uint32_t w, j;
    uint64_t tomb, h;
  };
  // One window of the walk, in every lane with `on` (cleared when the pair is done).
  auto step = [&](bool& on, Pair& x) {
    const Spot s = spot_of<L, W, kSwept>(slots, x.k, x.w);
    if (!on) return;
    const uint64_t base = static_cast<uint64_t>(x.w) * W;
    auto stored = [&](uint64_t at) {  // the key is there: overwrite the value (duplicate warning, Sec. IV-B3)
      slot_store_value<L>(slots, t.vals, at, x.v);
      if constexpr (!L::kCount) flags |= kFlagDuplicate;
      on = false;
    };
    if (s.hit) {
      stored(base + s.at);
      return;
    }
    // A pair that lost a slot has walked to its end without meeting the key, so the first
    // free slot it meets now is its own: had a copy of the key gone to a later window since,
    // it would have passed that free slot (tombstones only get fewer during an insert).
    const bool at_once = x.tomb == kLost && s.has_tomb;
    if (s.has_tomb && x.tomb >= kLost) x.tomb = base + s.tomb;
    const bool from_tomb = x.tomb < kLost;
    if (s.empty == W && x.j + 1 < t.p && !at_once) {  // no empty slot: walk on
      if (t.ovf != nullptr) ovf_mark(t.ovf, x.w, static_cast<uint32_t>(x.h) & 7u);
      x.w = probe_next(x.w, 1u + __umulhi(static_cast<uint32_t>(x.h), t.p - 1u), t.p);
      ++x.j;
      return;
    }
    if (!from_tomb && s.empty == W) {
      flags |= kFlagProbeLimit;  // every window visited, nothing to claim
      on = false;
      return;
    }
    // Claim the earliest candidate: the remembered tombstone, else the first empty slot, taken
    // to hold the word that clears and erases leave.  Where the slot went to another key, the
    // next one of the window is tried at once: slots fill in order, so the key is in none
    // behind the one that is claimed, and every one before it was seen here or by a CAS.
    // (Not in sweeps: few pairs race there, and the code around the loop cost 3 %.)
    uint64_t c = from_tomb ? x.tomb : base + s.empty;
    const uint64_t last = from_tomb ? c : base + (W - 1);
    Slot old = from_tomb ? L::tomb() : Slot{};
    const Slot pair = L::make(x.k, x.v);
    while (true) {
      Slot seen;
      if (L::cas(slots + c, old, pair, seen)) {
        if constexpr (L::kSoA) slot_store_value<L>(slots, t.vals, c, x.v);
        ++added;
        on = false;
        return;
      }
      const Key kk = L::key(seen);
      if (kk == x.k) {  // by another copy of the pair's key
        stored(c);
        return;
      }
      if (kk == (from_tomb ? L::kTomb : L::kEmpty)) {
        old = seen;  // still free, with another word
        continue;
      }
      if (kSwept || c == last) break;
      ++c;
      old = Slot{};
    }
    // on from the slot's window (the ones before it hold no free slot)
    x.w = static_cast<uint32_t>(c / W);
    if (from_tomb) x.j = 0;
    x.tomb = kLost;
  };
  auto enqueue = [&](bool yes, const Pair& x) {
    const uint32_t b = __ballot_sync(kFull, yes);
    if (yes) {
      const uint32_t at = cnt + __popc(b & below);
      q.key[at] = x.k;
      q.val[at] = x.v;
      q.w[at] = x.w;
      q.j[at] = x.j;
      q.tomb[at] = x.tomb;
    }
    cnt += __popc(b);
    __syncwarp();
  };
  // a step for the last (at most 32) pairs of the queue
  auto drain = [&]() {
    const uint32_t m = cnt < 32 ? cnt : 32;
    cnt -= m;
    bool on = lane < m;
    Pair x{};
    if (on) {
      x.k = q.key[cnt + lane];
      x.v = q.val[cnt + lane];
      x.w = q.w[cnt + lane];
      x.j = q.j[cnt + lane];
      x.tomb = q.tomb[cnt + lane];
    }
    __syncwarp();
    x.w = window_for_all(on, x.w);
    x.h = fmix64(static_cast<uint64_t>(x.k) ^ t.seed);
    step(on, x);
    enqueue(on, x);
  };

  const uint32_t nn = blocks.n;
  uint32_t base = blocks.take();
  Key kn = nn - base > lane ? ldg_stream(keys + base + lane) : Key(0);
  Val vn = vals == nullptr ? Val(1) : nn - base > lane ? ldg_stream(vals + base + lane) : Val(0);
  while (base != nn) {
    const Key k = kn;
    const Val v = vn;
    const bool in = nn - base > lane, bad = in && is_sentinel(k);
    base = blocks.take();
    kn = nn - base > lane ? ldg_stream(keys + base + lane) : Key(0);  // the next block's pairs
    if (vals != nullptr) vn = nn - base > lane ? ldg_stream(vals + base + lane) : Val(0);
    // counting inserts run on aggregated batches whose padding is key 0 (the aggregation
    // pass already flagged the caller's sentinel keys)
    if (bad && !(L::kCount && k == Key(0))) flags |= kFlagInvalid;
    Pair x{k, v, 0, 0, kNone, fmix64(static_cast<uint64_t>(k) ^ t.seed)};  // as probe_init
    x.w = __umulhi(static_cast<uint32_t>(x.h >> 32), t.p);
    bool on = in && !bad;
    if (!__any_sync(kFull, on)) continue;  // padding of an aggregated batch
    step(on, x);
    enqueue(on, x);
    while (cnt >= 32) drain();
  }
  while (cnt > 0) drain();
}

// kSwept: a batch split by table region, swept in order by `counter`.  n_dev (or null): the
// batch's size on the device, at most n.
template <class L, int W, bool kSwept>
__global__ void __launch_bounds__(kLookThreads, 4)
    k_insert(TableDesc t, const typename L::Key* __restrict__ keys, const typename L::Val* __restrict__ vals,
             uint64_t n, unsigned long long* counter, const unsigned long long* n_dev) {
  if (n_dev != nullptr) n = *n_dev;
  __shared__ InsertQueue<typename L::Key, typename L::Val> q[kLookThreads / 32];
  uint32_t flags = 0;
  long long added = 0;
  BatchBlocks<kSwept> blocks(n, counter, 512, false);
  blocks.prefetch(t.slots, static_cast<uint64_t>(t.p) * W * slot_size<L>());
  insert_blocks<L, W>(t, keys, vals, blocks, q[threadIdx.x >> 5], flags, added);
  flush_flags(t.status, flags);
  flush_delta(t.size, added);
}

// As many blocks as fit, at every size: with fewer, so that fewer pairs race for slots, batches
// of 2^17 to 2^21 pairs took longer (two or three blocks an SM against four, load 0.9: 222,476
// pairs of 4+4 bytes 31.3 / 29.2 us, 600,000 45.3 / 40.3, 2^20 52.0 / 48.7; 317,816 8-byte
// set keys at 0.6 20.7 / 18.8).
template <class L, int W>
cudaError_t insert_launch(const wc_table* t, const typename L::Key* keys, const typename L::Val* vals, uint64_t n,
                          unsigned long long* counter, const unsigned long long* n_dev, cudaStream_t s) {
  auto kern = counter != nullptr ? k_insert<L, W, true> : k_insert<L, W, false>;
  const uint64_t want = (n + kLookThreads - 1) / kLookThreads;
  const uint64_t most = static_cast<uint64_t>(occupancy(kern, kLookThreads)) * t->sm_count;
  return launch_k(t, kern, static_cast<unsigned>(std::min(want, most)), kLookThreads, 0, s, desc_of(t), keys, vals, n,
                  counter, n_dev);
}

}  // namespace wc
