"""The scratch a table's split calls share: its order between streams, and calls that are
recorded into CUDA graphs."""
from __future__ import annotations

import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wc():
    from paper_2009_07914_gb300 import build
    build.build()
    import paper_2009_07914_gb300 as m
    return m


def _keys(n, first=1):
    import torch
    return (torch.arange(first, first + n, device="cuda", dtype=torch.int64) * 0x9E3779B1 % (1 << 32)).to(torch.int32)


def test_streams_that_share_a_handle_are_ordered(wc):
    """The per-thread default stream has one handle for every thread: a split insert of a
    second thread waits for the one that a first thread has pending, though the handles are
    equal (both split into the one scratch of the table)."""
    import torch
    from paper_2009_07914_gb300 import api
    n = 400_000  # split: more than 2^18 pairs, a table above 64 MiB
    t = wc.SingleValueTable(4, 4, min_capacity=9_000_000, window_width=8)
    a, b = _keys(n), _keys(n, n + 1)
    api.wc_insert(t.handle, a, a)  # the scratch exists, the kernels are loaded
    api.wc_table_clear(t.handle)
    torch.cuda.synchronize()
    first_in, done, ev, err = threading.Event(), threading.Event(), {}, []

    def work(name, keys, sleep):
        try:
            s = torch.cuda.ExternalStream(2)  # cudaStreamPerThread
            with torch.cuda.stream(s):
                if sleep:
                    torch.cuda._sleep(600_000_000)  # about 0.3 s
                api.wc_insert(t.handle, keys, keys, stream=2)
                ev[name] = torch.cuda.Event()
                ev[name].record(s)
        except Exception as e:  # pragma: no cover
            err.append(e)
        first_in.set()
        done.wait(60)  # the thread's stream lives as long as the thread

    threads = [threading.Thread(target=work, args=("a", a, True)), threading.Thread(target=work, args=("b", b, False))]
    threads[0].start()
    first_in.wait(60)
    threads[1].start()
    while len(ev) < 2 and not err:
        pass
    if not err:
        ev["b"].synchronize()
        behind = ev["a"].query()
    done.set()
    for th in threads:
        th.join()
    assert not err and behind
    torch.cuda.synchronize()
    out, found = torch.empty_like(a), torch.empty(n, dtype=torch.uint8, device="cuda")
    for keys in (a, b):
        api.wc_retrieve(t.handle, keys, out, found)
        assert torch.equal(out, keys) and bool(found.all())
    assert t.size() == 2 * n


def _record(f):
    import torch
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        f()
    return g


@pytest.mark.parametrize("warm", [True, False])
def test_recorded_insert_keeps_its_scratch(wc, warm):
    """A split insert recorded into a graph replays right after other calls have grown the
    table's scratch (a larger lookup, a larger insert), whether its buffer came from a call
    before the capture or not; a larger one recorded later leaves it its own."""
    import torch
    from paper_2009_07914_gb300 import api
    n = 300_001
    t = wc.SingleValueTable(4, 4, min_capacity=72_000_000, window_width=8)
    assert t.info["table_bytes"] > 512 << 20
    a, b, c = _keys(n), _keys(2 * n, 10_000_000), _keys(9_500_000, 20_000_000)
    if warm:
        api.wc_insert(t.handle, a, a)
    else:
        api.wc_insert(t.handle, a[:100], a[:100])  # the library is loaded, no scratch
    before = api.wc_table_get_info(t.handle)["work_bytes"]
    assert (before > 0) == warm
    g = _record(lambda: api.wc_insert(t.handle, a, a))
    held = api.wc_table_get_info(t.handle)["work_bytes"]
    assert held == before if warm else held > 0  # taken over, or allocated outside the graph
    h = _record(lambda: api.wc_insert(t.handle, b, b))
    api.wc_table_clear(t.handle)
    out, found = torch.empty_like(c), torch.empty(c.numel(), dtype=torch.uint8, device="cuda")
    big = torch.cat([a, c])
    api.wc_insert(t.handle, c, c)
    api.wc_retrieve(t.handle, c, out, found)  # split: one query per 64 bytes
    assert bool(found.all()) and api.wc_table_get_info(t.handle)["work_bytes"] > held
    junk = [torch.full((1 << 22,), 77, dtype=torch.int32, device="cuda") for _ in range(8)]
    for _ in range(2):
        g.replay()
        h.replay()
        torch.cuda.synchronize()
        assert t.size() == c.numel() + 3 * n
        for keys in (a, b, c):
            m = keys.numel()
            api.wc_retrieve(t.handle, keys, out[:m], found[:m])
            assert torch.equal(out[:m], keys) and bool(found[:m].all())
        api.wc_table_clear(t.handle)
        api.wc_insert(t.handle, c, c)
        api.wc_insert(t.handle, big, big)
    assert all(bool((x == 77).all()) for x in junk)


def test_recorded_counting_and_bucket_inserts(wc):
    """Counting and bucket multi-value inserts (always through scratch) recorded without a call
    before them, replayed after larger calls."""
    import torch
    from paper_2009_07914_gb300 import api
    n = 50_003
    a, c = _keys(n), _keys(600_000, 1_000_000)
    t = wc.CountingTable(4, min_capacity=1_500_000)
    m = wc.MultiValueTable(4, 4, min_capacity=1_500_000, value_pool_capacity=8_000_000)
    api.wc_insert(t.handle, a[:1], None)
    api.wc_insert(m.handle, a[:1], a[:1])
    api.wc_table_clear(t.handle)
    api.wc_table_clear(m.handle)
    gt = _record(lambda: api.wc_insert(t.handle, a, None))
    gm = _record(lambda: api.wc_insert(m.handle, a, a))
    api.wc_insert(t.handle, c, None)
    api.wc_insert(m.handle, c, c)
    for _ in range(2):
        gt.replay()
        gm.replay()
    torch.cuda.synchronize()
    out, found = torch.empty_like(a), torch.empty(n, dtype=torch.uint8, device="cuda")
    api.wc_retrieve(t.handle, a, out, found)
    assert bool((out == 2).all()) and bool(found.all())
    offs = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    assert api.wc_count_values(m.handle, a, offs) == 2 * n
    vals = torch.empty(2 * n, dtype=torch.int32, device="cuda")
    api.wc_retrieve_multi(m.handle, a, offs, vals)
    assert torch.equal(vals.view(n, 2), a.view(n, 1).expand(n, 2))
    assert t.size() == n + c.numel()
