"""Open-addressing multi-value tables, one pair or query per thread with walk bits: batch
edges, hot keys that fill windows, erases and appends after them, and the calls after which
the bits may not be trusted -- a snapshot restored, a device view handed out -- against the
multiset oracle; counts split by region against the same counts in small batches."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import wc_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wc():
    from paper_2009_07914_gb300 import build
    build.build()
    import paper_2009_07914_gb300 as m
    return m


def _same(t, o, q):
    offs, _ = t.count_values(q)
    eoffs, _ = o.count_values(q)
    np.testing.assert_array_equal(offs, eoffs)
    vals, _ = t.retrieve_multi(q, offs)
    evals, _ = o.retrieve_multi(q, eoffs)
    np.testing.assert_array_equal(oracle.sorted_segments(vals, offs), oracle.sorted_segments(evals, eoffs))


@pytest.mark.parametrize("kb,W", [(4, 4), (4, 8), (8, 2), (8, 4), (4, 16)])
def test_edges_hot_keys_restore_and_view(wc, kb, W):
    from paper_2009_07914_gb300 import api
    universe = 6_000
    allk = wc_inputs.distinct_u32(0x0A, 2 * universe) if kb == 4 else wc_inputs.distinct_u64(0x0A, 2 * universe)
    for n in (1, 31, 33, 513, 20_011):
        pick = np.minimum(wc_inputs.uniform_u32(n, n) % universe, wc_inputs.uniform_u32(n + 1, n) % universe)
        pick[: n // 8] = 7  # one hot key: its copies fill windows
        keys = allk[pick]
        if n > 100:
            keys[50], keys[51] = 0, 2 ** (8 * kb) - 1
        vals = np.arange(n).astype(keys.dtype)
        t = wc.MultiValueOATable(kb, kb, min_capacity=int(n / 0.9) + 40, window_width=W)
        o = oracle.MultiValue(kb, kb)
        assert t.insert(keys, vals) == o.insert(keys, vals)
        q = allk[:: 1 if n > 100 else 97].copy()
        _same(t, o, q)
        snap = api.wc_table_snapshot(t.handle)
        t.erase(allk[3:universe:5])
        o.erase(allk[3:universe:5])
        t.insert(keys[n // 2:n // 2 + n // 16], vals[n // 2:n // 2 + n // 16])
        o.insert(keys[n // 2:n // 2 + n // 16], vals[n // 2:n // 2 + n // 16])
        _same(t, o, q)
        u = wc.MultiValueOATable(kb, kb, min_capacity=int(n / 0.9) + 40, window_width=W)
        api.wc_table_restore(u.handle, snap)
        o2 = oracle.MultiValue(kb, kb)
        o2.insert(keys, vals)
        _same(u, o2, q)
        api.wc_table_device_view(u.handle)  # from here on user kernels may write slots
        u.insert(keys[:5], vals[:5])
        o2.insert(keys[:5], vals[:5])
        _same(u, o2, q)
        t.clear()
        assert t.size() == 0 and not t.count_values(q)[0].any()


@pytest.mark.parametrize("bucket", [False, True], ids=["open_addressing", "bucket"])
def test_counts_split_by_region(wc, bucket):
    import torch
    from paper_2009_07914_gb300 import api
    n = 3_000_017
    if bucket:
        t = wc.MultiValueTable(4, 4, min_capacity=36_000_000, value_pool_capacity=8 * n)
    else:
        t = wc.MultiValueOATable(4, 4, min_capacity=70_000_000)
    assert t.info["table_bytes"] > 512 << 20
    keys = torch.from_numpy(wc_inputs.distinct_u32(0xC0, n).view(np.int32)).cuda()
    api.wc_insert(t.handle, keys.repeat(3), torch.arange(3 * n, device="cuda", dtype=torch.int32))
    m = t.info["table_bytes"] // 64 + 77
    q = keys.repeat(m // n + 1)[:m].contiguous()
    q[::3] ^= 0x15A5_0000  # mostly keys that were never inserted
    q[::1_000_003] = 0
    a, b = (torch.full((m + 1,), -1, dtype=torch.int64, device="cuda") for _ in range(2))
    total = api.wc_count_values(t.handle, q, a)
    step, at = 1 << 20, 0
    for i in range(0, m, step):
        part = q[i:i + step]
        s = api.wc_count_values(t.handle, part, b[:part.numel() + 1])
        assert torch.equal(a[i:i + part.numel() + 1], b[:part.numel() + 1] + at)
        at += s
    assert total == at == int(a[m])


M64 = (1 << 64) - 1


def _first_two_windows(key, seed, p):
    k = (key ^ seed) & M64
    k ^= k >> 33
    k = (k * 0xFF51AFD7ED558CCD) & M64
    k ^= k >> 33
    k = (k * 0xC4CEB9FE1A85EC53) & M64
    k ^= k >> 33
    w = ((k >> 32) * p) >> 32
    return w, (w + 1 + (((k & 0xFFFFFFFF) * (p - 1)) >> 32)) % p


@pytest.mark.parametrize("W", [8, 16])
def test_recorded_count_sees_slots_that_a_user_kernel_wrote(wc, W):
    """A count is recorded, then the table's slots are handed out and a pair is put into the
    second window of its key without a walk bit (as a user kernel would; written here by a
    copy): the replay and a new count both find it."""
    import ctypes

    import torch
    from paper_2009_07914_gb300 import api
    seed = 0x5EED_C0DE
    t = wc.MultiValueOATable(4, 4, min_capacity=11 * W, window_width=W, seed=seed)
    p = t.info["windows"]
    by_first = {}
    for k in range(1, 5000):
        by_first.setdefault(_first_two_windows(k, seed, p)[0], []).append(k)
    w0, group = max(by_first.items(), key=lambda x: len(x[1]))
    fill, key = group[:W], next(k for k in group[W:] if _first_two_windows(k, seed, p)[1] != w0)
    t.insert(np.array(fill, np.uint32), np.zeros(W, np.uint32))  # the window is full, none walked past it
    q = torch.tensor([key, fill[0]], dtype=torch.int32, device="cuda")
    offs = torch.empty(3, dtype=torch.int64, device="cuda")
    assert api.wc_count_values(t.handle, q, offs) == 1  # the kernels are loaded before the capture
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        api.wc_count_values(t.handle, q, offs, want_total=False)
    g.replay()
    assert offs.tolist() == [0, 0, 1]
    view = api.wc_table_device_view(t.handle)
    word = torch.tensor([5 << 32 | key], dtype=torch.int64, device="cuda")
    slot = view.slots + 8 * W * _first_two_windows(key, seed, p)[1]
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.13")  # the runtime instance libwc.so is linked against
    assert rt.cudaMemcpy(ctypes.c_void_p(slot), ctypes.c_void_p(word.data_ptr()), ctypes.c_size_t(8), 3) == 0
    offs.fill_(-1)
    g.replay()
    assert offs.tolist() == [0, 1, 2]
    assert api.wc_count_values(t.handle, q, offs) == 2 and offs.tolist() == [0, 1, 2]
