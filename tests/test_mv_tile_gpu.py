"""Bucket multi-value inserts of keys that differ only in high bits (left-aligned codes,
identifiers shifted up): the tile aggregation's table in shared memory spreads them like
any others."""
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


@pytest.mark.parametrize("block", [256, 512])
@pytest.mark.parametrize("shift", [0, 44, 48, 52])
def test_keys_that_differ_in_high_bits(wc, shift, block):
    """The same values as the oracle, in less than four times the time of well mixed keys
    (one chain of a tile's thousand keys would take some twenty times as long)."""
    import torch
    from paper_2009_07914_gb300 import api
    from paper_2009_07914_gb300.table import to_device
    n, u = 1 << 19, 4000
    pick = wc_inputs.uniform_u32(shift + 1, n) % u
    dev = torch.device("cuda", torch.cuda.current_device())
    vals = np.arange(n, dtype=np.uint32)
    ms = []
    for mixed in (True, False):
        allk = wc_inputs.distinct_u64(9, u) if mixed else np.arange(1, u + 1, dtype=np.uint64) << np.uint64(shift)
        keys = allk[pick]
        t = wc.MultiValueTable(8, 4, min_capacity=2 * u, value_pool_capacity=2 * n, window_width=4)
        t.set_launch(wc.WC_OP_INSERT, api.wc_table_get_launch(t.handle, wc.WC_OP_INSERT)["group_size"], block)
        k, v = to_device(keys, 8, dev), to_device(vals, 4, dev)
        best = 1e9
        for _ in range(6):
            api.wc_table_clear(t.handle)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            api.wc_insert(t.handle, k, v)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    o = oracle.MultiValue(8, 4)
    o.insert(keys, vals)
    offs, _ = t.count_values(allk)
    eoffs, _ = o.count_values(allk)
    np.testing.assert_array_equal(offs, eoffs)
    got, _ = t.retrieve_multi(allk, offs)
    exp, _ = o.retrieve_multi(allk, eoffs)
    np.testing.assert_array_equal(oracle.sorted_segments(got, offs), oracle.sorted_segments(exp, eoffs))
    assert ms[1] < 4 * ms[0], ms
