"""Bloom filter batches that are split by filter region set and find exactly the bits that
the same keys set and find in batches small enough to stay in input order (which the oracle
checks elsewhere): filters from one region to more than a split takes, odd sizes, sentinels
and a hot key that fills a third of the batch."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wc():
    from paper_2009_07914_gb300 import build
    build.build()
    import paper_2009_07914_gb300 as m
    return m


@pytest.mark.parametrize("kb", [4, 8])
@pytest.mark.parametrize("bits,k", [(1 << 12, 1), (7_000_001, 16), (160_000_000, 7), (1_990_000_000, 8)])
def test_split_batches_equal_small_ones(wc, kb, bits, k):
    import torch
    from paper_2009_07914_gb300 import api
    a, b = (wc.BloomFilterTable(kb, bits=bits, k=k) for _ in range(2))
    n = max((1 << 24) + 33, a.info["table_bytes"] // 4 + 5)
    g = torch.Generator(device="cuda")
    g.manual_seed(bits + kb)
    lo, hi = (-2 ** 31, 2 ** 31) if kb == 4 else (-2 ** 63, 2 ** 63 - 1)
    keys = torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=torch.int32 if kb == 4 else torch.int64)
    keys[::3] = 12345
    keys[1::1_000_003] = 0
    keys[2::1_000_003] = -1
    api.wc_insert(a.handle, keys, None)
    step = 10_000_019
    for i in range(0, n, step):
        api.wc_insert(b.handle, keys[i:i + step], None)
    assert a.size() == b.size() == int(((keys != 0) & (keys != -1)).sum())
    assert a.status(clear=True) == b.status(clear=True) == wc.WC_FLAG_INVALID_KEY
    da, db = api.wc_table_dump_slots(a.handle), api.wc_table_dump_slots(b.handle)
    assert np.array_equal(da, db) and da.any()
    q = torch.randint(lo, hi, (max(n // 2, a.info["table_bytes"] // 32 + 7),), generator=g, device="cuda",
                      dtype=keys.dtype)
    q[::2] = keys[:(q.numel() + 1) // 2]
    fa = torch.full((q.numel(),), 7, dtype=torch.uint8, device="cuda")
    fb = torch.full_like(fa, 7)
    api.wc_contains(a.handle, q, fa)
    for i in range(0, q.numel(), 1_000_003):
        api.wc_contains(b.handle, q[i:i + 1_000_003], fb[i:i + 1_000_003])
    assert torch.equal(fa, fb)
    real = (q[::2] != 0) & (q[::2] != -1)
    assert (fa[::2][real] == 1).all()


@pytest.mark.parametrize("blocks,n", [(31, 900_000_000), (31, (1 << 30) - 1), (64, 1_700_000_000)])
def test_large_batches_into_small_filters(wc, blocks, n):
    """Hundreds of millions of keys of one or two regions (part sizes and unit counts past
    32 bits if they grew with the batch): the same bits and size as a few keys at a time."""
    import torch
    from paper_2009_07914_gb300 import api
    a, b = (wc.BloomFilterTable(4, bits=256 * blocks, k=7) for _ in range(2))
    few = torch.arange(1, 129, device="cuda", dtype=torch.int32) * 7919
    keys = few[:3].repeat((n + 2) // 3)[:n].contiguous()  # three keys again and again, then all of them
    keys[-128:] = few
    api.wc_insert(a.handle, keys, None)
    api.wc_insert(b.handle, few, None)
    assert a.size() == n and b.size() == 128
    assert a.status(clear=True) == b.status(clear=True) == 0
    da, db = api.wc_table_dump_slots(a.handle), api.wc_table_dump_slots(b.handle)
    assert np.array_equal(da, db) and da.any()
    f = torch.zeros(128, dtype=torch.uint8, device="cuda")
    api.wc_contains(a.handle, few, f)
    assert bool((f == 1).all())
