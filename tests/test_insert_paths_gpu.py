"""Inserts one pair per thread, in input order and swept by region: the sizes where a warp's
block, its queue and a chunk of the sweep begin and end, repeated keys, tombstones that many
pairs want at once, and a table that is filled to its last slot -- against the oracle's plain
map and the reachability check of the slot dump."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import wc_inputs

pytestmark = pytest.mark.gpu

SEED = 0x5EED_C0DE


@pytest.fixture(scope="module")
def wc():
    from paper_2009_07914_gb300 import build
    build.build()
    import paper_2009_07914_gb300 as m
    return m


def _inputs(kb, n, seed):
    if kb == 4:
        return wc_inputs.distinct_u32(seed, n), wc_inputs.uniform_u32(seed + 1, n)
    return wc_inputs.distinct_u64(seed, n), wc_inputs.uniform_u64(seed + 1, n)


def _same(wc, t, o, q):
    out, found, _ = t.retrieve(q)
    eo, ef, _ = o.retrieve(q)
    np.testing.assert_array_equal(found, ef)
    np.testing.assert_array_equal(out, eo)
    assert t.size() == o.size()


def _layout(wc, t, soa):
    from paper_2009_07914_gb300 import api
    if soa:
        return
    i = t.info
    bits = api.wc_table_dump_overflow_bits(t.handle) if i["options"] & wc.WC_OPT_OVERFLOW_BITS else None
    r = oracle.check_slots(api.wc_table_dump_slots(t.handle), i["windows"], i["window_width"], i["slot_bytes"], SEED,
                           True, bits)
    assert r["dups"] == 0 and r["unreachable"] == 0


@pytest.mark.parametrize("blocked", [False, True], ids=["direct", "swept"])
@pytest.mark.parametrize("kb,W,soa,bits", [(4, 8, 0, 1), (4, 4, 0, 0), (8, 4, 0, 1), (8, 2, 0, 0), (4, 16, 1, 0),
                                           (8, 8, 1, 0)])
def test_batches_erases_and_reinserts(wc, kb, W, soa, bits, blocked):
    opt = (wc.WC_OPT_SOA if soa else 0) | (wc.WC_OPT_OVERFLOW_BITS if bits else 0)
    for n in (1, 31, 33, 511, 513, 4097, 60_013):
        keys, vals = _inputs(kb, n + 64, 0x1A5 + n)
        t = wc.SingleValueTable(kb, kb, min_capacity=int(n / 0.95) + 1, window_width=W, options=opt, seed=SEED)
        if blocked:
            lc = wc.wc_table_get_launch(t.handle, wc.WC_OP_INSERT)
            t.set_launch(wc.WC_OP_INSERT, lc["group_size"], scheme=wc.WC_SCHEME_BLOCKED, region_mib=1)
        o = oracle.SingleValue(kb, kb)
        k = keys[:n].copy()
        if n > 100:
            k[50] = 0
            k[51] = 2 ** (8 * kb) - 1
        assert t.insert(k, vals[:n]) == o.insert(k, vals[:n])
        _same(wc, t, o, keys)
        t.erase(k[::2])
        o.erase(k[::2])
        # the erased keys with new values; what is stored already is overwritten
        again, v2 = np.concatenate([k[::2], k[1::4]]), wc_inputs.uniform_u64(n, n)[:k[::2].size + k[1::4].size]
        v2 = v2.astype(vals.dtype)
        assert t.insert(again, v2) == o.insert(again, v2)
        _same(wc, t, o, keys)
        _layout(wc, t, soa)


@pytest.mark.parametrize("kb,W", [(4, 8), (8, 4)])
def test_last_slots_and_repeats(wc, kb, W):
    """More distinct keys than slots, in a table full of tombstones: every slot is taken, the
    rest raises PROBE_LIMIT; each key of a batch of repeats is stored once, with one of its
    values."""
    t = wc.SingleValueTable(kb, kb, min_capacity=5 * W, window_width=W, seed=SEED)
    cap = t.capacity
    keys, vals = _inputs(kb, cap + 40, 0x7A8)
    t.insert(keys[:cap], vals[:cap])
    t.erase(keys[:cap])
    assert t.size() == 0
    flags = t.insert(keys, vals)
    assert flags & wc.WC_FLAG_PROBE_LIMIT and t.size() == cap
    out, found, _ = t.retrieve(keys)
    assert found.sum() == cap and np.array_equal(out[found == 1], vals[found == 1])
    big = wc.SingleValueTable(kb, kb, min_capacity=1 << 12, window_width=W, seed=SEED)
    pick = np.arange(200_000) % 997
    v = np.arange(200_000).astype(vals.dtype)
    k = _inputs(kb, 997, 0x99)[0][pick]
    assert big.insert(k, v) == wc.WC_FLAG_DUPLICATE_KEY and big.size() == 997
    out, found, _ = big.retrieve(k[:997])
    assert found.all() and np.array_equal(out.astype(np.int64) % 997, pick[:997])


@pytest.mark.parametrize("kb,n,load", [(4, (1 << 19) + 13, 0.9), (4, (1 << 21) + 5, 0.9), (8, (1 << 22) + 77, 0.9),
                                       (4, (1 << 19) + 31, 0.05), (8, (1 << 18) + 1, 0.005)])
def test_sweeps_of_every_chunk_length(wc, kb, n, load):
    """Chunks of 32 to 256 inputs; tables that end inside the prefetched range, in front of
    it, or are so large beside the batch that nothing is prefetched."""
    keys, vals = _inputs(kb, n, n)
    t = wc.SingleValueTable(kb, kb, min_capacity=int(n / load) + 1, seed=SEED)
    for op in (wc.WC_OP_INSERT, wc.WC_OP_RETRIEVE):
        lc = wc.wc_table_get_launch(t.handle, op)
        t.set_launch(op, lc["group_size"], scheme=wc.WC_SCHEME_BLOCKED, region_mib=1)
    assert t.insert(keys, vals) == 0 and t.size() == n
    out, found, _ = t.retrieve(keys)
    assert found.all()
    np.testing.assert_array_equal(out, vals)


@pytest.mark.parametrize("kb,W", [(4, 8), (4, 4), (8, 4), (8, 2)])
@pytest.mark.parametrize("windows,copies", [(7, 1), (7, 40), (1009, 8), (40_009, 3)])
def test_pairs_that_race_for_the_same_slots(wc, kb, W, windows, copies):
    """Every pair of a batch for the same few windows at once, each key several times side by
    side and far apart: each key stored once, the empty slots of a window behind all others;
    counts of a counting table exact."""
    from paper_2009_07914_gb300 import api
    n = int(windows * W * 0.97)
    keys, _ = _inputs(kb, n, windows + W)
    batch = np.concatenate([np.repeat(keys, copies), np.tile(keys, copies)])
    vals = np.arange(batch.size).astype(keys.dtype)
    t = wc.SingleValueTable(kb, kb, min_capacity=windows * W, window_width=W, seed=SEED)
    c = wc.CountingTable(kb, min_capacity=windows * W, window_width=W, seed=SEED)
    for _ in range(3):
        t.clear()
        assert t.insert(batch, vals) == wc.WC_FLAG_DUPLICATE_KEY and t.size() == n
        out, found, _ = t.retrieve(keys)
        assert found.all()
        np.testing.assert_array_equal(batch[out.astype(np.int64)], keys)  # one of the key's values
        _layout(wc, t, 0)
        dump = api.wc_table_dump_slots(t.handle).view(np.uint64)
        k = (dump & np.uint64(0xFFFFFFFF) if kb == 4 else dump[::2]).reshape(-1, W)
        empty = k == 0
        assert (empty[:, 1:] >= empty[:, :-1]).all()
        c.clear()
        c.insert(batch)
        assert c.size() == n
        got, found, _ = c.retrieve(keys)
        assert found.all() and (got == 2 * copies).all()


@pytest.mark.parametrize("kb,W", [(4, 8), (8, 4)])
def test_free_slots_with_other_words(wc, kb, W):
    """A slot is free by its key: an empty slot or a tombstone whose value word is not what
    clears and erases leave (left by a user kernel; written here by a copy) is claimed."""
    import ctypes

    import torch
    from paper_2009_07914_gb300 import api
    t = wc.SingleValueTable(kb, kb, min_capacity=5 * W, window_width=W, seed=SEED)
    cap, tomb = t.capacity, 2 ** (8 * kb) - 1
    words = np.zeros((cap, 2), np.uint32 if kb == 4 else np.uint64)
    words[:, 1] = 9
    words.reshape(-1, W, 2)[:, : W // 2, 0] = tomb  # each window: tombstones, then empty slots
    src = torch.from_numpy(words.view(np.int32 if kb == 4 else np.int64)).cuda()
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.13")  # the runtime instance libwc.so is linked against
    assert rt.cudaMemcpy(ctypes.c_void_p(api.wc_table_device_view(t.handle).slots), ctypes.c_void_p(src.data_ptr()),
                         ctypes.c_size_t(words.nbytes), 3) == 0
    keys, vals = _inputs(kb, cap, 0x3F)
    assert t.insert(np.repeat(keys, 3), np.repeat(vals, 3)) == wc.WC_FLAG_DUPLICATE_KEY and t.size() == cap
    out, found, _ = t.retrieve(keys)
    assert found.all()
    np.testing.assert_array_equal(out, vals)


@pytest.mark.parametrize("kb,W,group", [(4, 8, 1), (4, 8, 4), (8, 4, 2), (4, 16, 2)])
@pytest.mark.parametrize("n", [1, 33, 500_009, 700_001, 3_000_017])
def test_erases_in_strided_chunks(wc, kb, W, group, n):
    """Erased keys are gone, their neighbours stay and the size is exact, from batches that give
    a warp a few keys to batches of several chunks a warp."""
    import torch
    from paper_2009_07914_gb300 import api
    from paper_2009_07914_gb300.table import to_device
    keys, vals = _inputs(kb, 2 * n + 64, n + kb)
    t = wc.SingleValueTable(kb, kb, min_capacity=int(2 * n / 0.85) + 64, window_width=W, seed=SEED)
    t.set_launch(wc.WC_OP_ERASE, group)
    dev = torch.device("cuda", torch.cuda.current_device())
    k, v = to_device(keys, kb, dev), to_device(vals, kb, dev)
    api.wc_insert(t.handle, k[:2 * n], v[:2 * n])
    gone = k[:2 * n:2].contiguous()
    api.wc_erase(t.handle, gone)
    api.wc_erase(t.handle, k[2 * n:])  # never stored
    assert t.size() == n
    out, found = torch.empty_like(k), torch.empty(k.numel(), dtype=torch.uint8, device=dev)
    api.wc_retrieve(t.handle, k, out, found)
    assert not found[:2 * n:2].any() and bool(found[1:2 * n:2].all()) and not found[2 * n:].any()
    assert torch.equal(out[1:2 * n:2], v[1:2 * n:2])
    api.wc_insert(t.handle, gone, gone)
    assert t.size() == 2 * n and t.status() == 0
