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
