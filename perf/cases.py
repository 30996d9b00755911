"""The work this library is used for, as cases that can be timed and compared.

A case is a dict of plain values; `prepare` makes what a program has in hand before the
call (device tensors made from the seed, tables, an executor), `run` makes one pass through
the public calls and returns everything they wrote.  Every pass starts from the same table
contents (it clears the table first, or only reads it), so it can be repeated.

Families:
  sv      clear, insert, retrieve (and, with `erase`, erase every second key and retrieve
          again) on a single-value table: the build-then-query program
  lookup  retrieve alone, from a table built once: the read-mostly program
  count   clear, insert, retrieve on a counting table (k-mer counting)
  set     clear, insert, contains on a hash set;  bloom: the same on a Bloom filter
  mv      clear, insert, count_values, retrieve_multi on a bucket multi-value table;
  mvoa    the same on the open-addressing multi-value table
  exec    one batch of uneven requests on many tables through the batched executor
  host    clear, insert and retrieve through the host-buffer calls (pinned memory)

The order of a multi-value key's values is unspecified, so the values of a key are all its
label (a k-mer's taxon, a row's group): the outputs are then the same whatever the order.
All results are integers and have to be equal, so there are no values in 64-bit floating
point to compare them with (`exact` gives none).
"""
import torch

from paper_2009_07914_gb300 import WC_OPT_OVERFLOW_BITS, WC_OPT_SOA, api, serve
from paper_2009_07914_gb300.table import (BloomFilterTable, CountingTable, HashSetTable, MultiValueOATable,
                                          MultiValueTable, SingleValueTable)

ZIPF_S = 1.1  # exponent of the skewed draws, as in the repository's configurations


def listed():
    return [
        # the smallest requests a served table sees (about 1 k keys): launches and latency
        {"name": "sv32_1k", "family": "sv", "kb": 4, "n": 1000, "queries": 2000, "load": 0.5, "absent": 0.5,
         "bits": False, "soa": False, "erase": True, "slots": 1 << 16},
        # a table that fits in L2: 2^20 pairs at load 0.8, lookups half absent, erase, lookups again
        {"name": "sv32_1m", "family": "sv", "kb": 4, "n": 1 << 20, "queries": 1 << 21, "load": 0.8, "absent": 0.5,
         "bits": False, "soa": False, "erase": True, "slots": 0},
        # the headline workload: 2^27 pairs at load 0.9 with overflow bits, 2^27 lookups, half absent
        {"name": "sv32_128m", "family": "sv", "kb": 4, "n": 1 << 27, "queries": 1 << 27, "load": 0.9, "absent": 0.5,
         "bits": True, "soa": False, "erase": False, "slots": 0},
        # an index that is only read: default options, ragged sizes, nearly every key present
        {"name": "lookup32_50m", "family": "lookup", "kb": 4, "n": 90_000_001, "queries": 50_000_003, "load": 0.8,
         "absent": 0.1, "bits": False, "soa": False, "zipf": False},
        # 8+8-byte pairs and a skewed query stream over the whole set
        {"name": "sv64_zipf_256m", "family": "sv", "kb": 8, "n": 1 << 28, "queries": 1 << 28, "load": 0.9,
         "absent": 0.0, "bits": False, "soa": False, "erase": False, "slots": 0, "zipf": True},
        # k-mer index: 2^28 skewed inserts over 2^24 keys, then every key's values in CSR form
        {"name": "mv_zipf_256m", "family": "mv", "kb": 8, "vb": 4, "n": 1 << 28, "universe": 1 << 24,
         "queries": (1 << 24) + (1 << 22), "zipf": True, "growth": False},
        # uniform multiplicity (a join's build side): 2^26 pairs, 4 per key, open addressing
        {"name": "mvoa_r4_64m", "family": "mvoa", "kb": 4, "vb": 4, "n": 1 << 26, "universe": 1 << 24,
         "queries": 1 << 26, "zipf": False, "growth": False},
        # occurrence counts of a skewed stream, read back for every key
        {"name": "count_zipf_64m", "family": "count", "kb": 4, "n": (1 << 26) + 77, "universe": 1 << 24,
         "queries": 1 << 24, "weights": False},
        # de-duplication: a hash set of 4-byte keys at load 0.9, membership of as many keys, half absent
        {"name": "set32_60m", "family": "set", "kb": 4, "n": 60_000_001, "queries": 60_000_001, "load": 0.9,
         "absent": 0.5, "bits": True},
        # approximate membership at 10 bits per key, k = 7
        {"name": "bloom32_128m", "family": "bloom", "kb": 4, "n": 1 << 27, "queries": 1 << 27, "k": 7,
         "absent": 0.5},
        # 64 tables of uneven size, 128 uneven requests (60 % insert, 35 % retrieve, 5 % erase) in one batch
        {"name": "exec_64_tables", "family": "exec", "tables": 64, "items": 128, "cap_lo": 16, "cap_hi": 26,
         "req_lo": 10, "req_hi": 20, "plan": 5},
        # the same calls on pinned host buffers: copies overlapped with the kernels
        {"name": "host32_32m", "family": "host", "kb": 4, "n": 30_000_001, "queries": 30_000_001, "load": 0.9,
         "absent": 0.5, "bits": True},
    ]


def _log(rng, lo, hi):
    """A whole number spread over [lo, hi] by its logarithm, odd ones among them."""
    return int(min(hi, max(lo, lo * (hi / lo) ** rng.random())))


def draw(rng):
    f = rng.choice(["sv", "sv", "lookup", "mv", "mvoa", "count", "set", "bloom", "exec", "host"])
    kb = rng.choice([4, 8])
    load = round(rng.uniform(0.4, 0.95), 3)
    absent = round(rng.choice([0.0, rng.random(), 0.5]), 3)
    if f in ("sv", "lookup"):
        n = _log(rng, 1000, (1 << 27) if kb == 4 else (1 << 26))
        soa = rng.random() < 0.15
        c = {"family": f, "kb": kb, "n": n, "queries": max(1, int(n * rng.uniform(0.3, 1.5))), "load": load,
             "absent": absent, "bits": not soa and rng.random() < 0.5, "soa": soa, "zipf": rng.random() < 0.3}
        if f == "sv":
            c.update(erase=rng.random() < 0.3, slots=0)
        return c
    if f in ("mv", "mvoa"):
        n = _log(rng, 1000, 1 << 26)
        zipf = f == "mv" and rng.random() < 0.5  # an open-addressing table of a skewed stream walks every copy
        universe = max(1, int(n / rng.choice([1, 2, 4, 8, 16])))
        vb = rng.choice([4, 8]) if f == "mv" else kb
        return {"family": f, "kb": kb, "vb": vb, "n": n, "universe": universe,
                "queries": int(universe * rng.uniform(1.0, 2.0)), "zipf": zipf,
                "growth": f == "mv" and rng.random() < 0.25}
    if f == "count":
        n = _log(rng, 1000, 1 << 27)
        universe = max(1, n // rng.choice([1, 4, 16]))
        return {"family": f, "kb": kb, "n": n, "universe": universe, "queries": universe,
                "weights": rng.random() < 0.4}
    if f == "set":
        n = _log(rng, 1000, 1 << 27)
        return {"family": f, "kb": kb, "n": n, "queries": max(1, int(n * rng.uniform(0.3, 1.5))), "load": load,
                "absent": max(0.1, absent), "bits": rng.random() < 0.5}
    if f == "bloom":
        n = _log(rng, 1000, 1 << 27)
        return {"family": f, "kb": kb, "n": n, "queries": max(1, int(n * rng.uniform(0.3, 1.5))),
                "k": rng.choice([4, 7, 8]), "absent": max(0.1, absent)}
    if f == "exec":
        lo = rng.randint(10, 14)
        return {"family": f, "tables": rng.randint(4, 64), "items": rng.randint(16, 160), "cap_lo": 16,
                "cap_hi": rng.randint(20, 25), "req_lo": lo, "req_hi": rng.randint(lo + 2, 20), "plan": rng.randint(1, 1 << 20)}
    n = _log(rng, 100_000, 1 << 25)
    return {"family": f, "kb": 4, "n": n, "queries": max(1, int(n * rng.uniform(0.3, 1.2))), "load": load,
            "absent": absent, "bits": rng.random() < 0.5}


# ---- inputs -----------------------------------------------------------------------------

_INT = {4: torch.int32, 8: torch.int64}


def _shr(x, s):
    """Logical shift of int64 words."""
    return (x >> s) & ((1 << (64 - s)) - 1)


def _i64(c):
    return c - (1 << 64) if c >= 1 << 63 else c


def _mix32(x):
    """A 32-bit mix (lowbias32) of int64 words below 2^32."""
    m = 0xFFFFFFFF
    x = ((x ^ (x >> 16)) * 0x7FEB352D) & m
    x = ((x ^ (x >> 15)) * 0x846CA68B) & m
    return x ^ (x >> 16)


def _mix64(x):
    """SplitMix64's output function."""
    x = (x ^ _shr(x, 30)) * _i64(0xBF58476D1CE4E5B9)
    x = (x ^ _shr(x, 27)) * _i64(0x94D049BB133111EB)
    return x ^ _shr(x, 31)


def _keys(idx, kb, seed):
    """The distinct keys number idx[i] of a seeded sequence (a bijective mix), never 0 or
    all ones: those two numbers' places are taken by the last two of the sequence."""
    if kb == 4:
        base = int(seed) * 0x632BE5AB & 0xFFFFFFFF
        k = _mix32((idx * 0x9E3779B1 + base) & 0xFFFFFFFF)
        bad = (k == 0) | (k == 0xFFFFFFFF)
        spare = _mix32(((idx + (1 << 31)) * 0x9E3779B1 + base) & 0xFFFFFFFF)
        k = torch.where(bad, spare, k)
        return torch.where(k >= 1 << 31, k - (1 << 32), k).to(torch.int32)
    k = _mix64(idx * _i64(0x9E3779B97F4A7C15) + int(seed) * 0x632BE59BD9B4E019 % (1 << 62))
    return torch.where((k == 0) | (k == -1), k + 2, k)


def _values(idx, vb, seed):
    x = _mix64(idx * _i64(0xD1B54A32D192ED03) + int(seed) + 12345)
    return x.to(torch.int32) if vb == 4 else x


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _zipf(n, universe, seed):
    """n draws from 0..universe-1 with P(rank) falling as rank^-ZIPF_S (bounded Pareto,
    inverse transform)."""
    u = torch.rand(n, generator=_gen(seed), device="cuda", dtype=torch.float64)
    e = 1.0 - ZIPF_S
    x = (u * (float(universe + 1) ** e - 1.0) + 1.0) ** (1.0 / e)
    return x.to(torch.int64).clamp_(1, universe) - 1


def _range(n):
    return torch.arange(n, device="cuda", dtype=torch.int64)


def _query_idx(case, seed):
    """Key numbers to look up: `absent` of them beyond the n stored ones."""
    n, q, gone = case["n"], case["queries"], int(case["queries"] * case["absent"])
    if case.get("zipf"):
        idx = _zipf(q, n, seed + 7)
    elif q - gone <= n:
        idx = (_range(q) * 0x9E3779B1 + int(seed)) % n  # hashed keys: any order is a random one
    else:
        idx = torch.randint(0, n, (q,), generator=_gen(seed + 7), device="cuda")
    if gone:
        out = torch.rand(q, generator=_gen(seed + 8), device="cuda") < case["absent"]
        idx = torch.where(out, n + _range(q), idx)
    return idx


class _State:
    pass


def _sv_table(case):
    opts = (WC_OPT_OVERFLOW_BITS if case["bits"] else 0) | (WC_OPT_SOA if case.get("soa") else 0)
    slots = case.get("slots") or int(case["n"] / case["load"]) + 1
    return SingleValueTable(case["kb"], case["kb"], min_capacity=slots, options=opts)


def prepare(case, seed):
    s = _State()
    s.case, s.family = case, case["family"]
    if s.family == "exec":
        return _prepare_exec(s, case, seed)
    kb, n, q = case["kb"], case["n"], case["queries"]
    if s.family in ("sv", "lookup", "host", "set", "bloom"):
        s.keys = _keys(_range(n), kb, seed)
        s.queries = _keys(_query_idx(case, seed), kb, seed)
        s.found = torch.empty(q, dtype=torch.uint8, device="cuda")
    if s.family in ("sv", "lookup", "host"):
        s.values = _values(_range(n), kb, seed)
        s.out = torch.empty(q, dtype=_INT[kb], device="cuda")
        s.t = _sv_table(case)
        if case.get("erase"):
            s.gone = s.keys[::2].contiguous()
            s.out2, s.found2 = torch.empty_like(s.out), torch.empty_like(s.found)
        if s.family == "lookup":
            api.wc_insert(s.t.handle, s.keys, s.values)
            del s.keys, s.values
        if s.family == "host":
            s.keys, s.values, s.queries, s.out, s.found = (
                x.cpu().pin_memory() for x in (s.keys, s.values, s.queries, s.out, s.found))
    elif s.family == "set":
        s.t = HashSetTable(kb, min_capacity=int(n / case["load"]) + 1,
                           options=WC_OPT_OVERFLOW_BITS if case["bits"] else 0)
    elif s.family == "bloom":
        s.t = BloomFilterTable(kb, bits=10 * n, k=case["k"])
    else:  # repeated keys: count, mv, mvoa
        u = case["universe"]
        if s.family == "count" or case["zipf"]:
            rank = _zipf(n, u, seed)
        else:
            rank = torch.randint(0, u, (n,), generator=_gen(seed), device="cuda")
        s.keys = _keys(rank, kb, seed)
        # every key of the universe in another order, then keys that were never inserted
        qi = _range(q)
        s.queries = _keys(torch.where(qi < u, (qi * 0x9E3779B1 + 1) % u if u > 1 else qi * 0, qi), kb, seed)
        if s.family == "count":
            s.weights = (rank * 0x2545F491 + 3 & 15).to(_INT[kb]) + 1 if case["weights"] else None
            s.t = CountingTable(kb, min_capacity=int(u / 0.9) + 1)
            s.out = torch.empty(q, dtype=_INT[kb], device="cuda")
            s.found = torch.empty(q, dtype=torch.uint8, device="cuda")
        else:
            s.values = _values(rank, case["vb"], seed)  # the key's label
            s.offsets = torch.empty(q + 1, dtype=torch.int64, device="cuda")
            if s.family == "mvoa":
                s.t = MultiValueOATable(kb, kb, min_capacity=int(n / 0.8) + 1)
            elif case["growth"]:
                s.t = MultiValueTable(kb, case["vb"], min_capacity=int(u / 0.8) + 1,
                                      value_pool_capacity=4 * n + 1024, bucket_first_size=1, bucket_growth=1.1)
            else:
                s.t = MultiValueTable(kb, case["vb"], min_capacity=int(u / 0.8) + 1,
                                      value_pool_capacity=n + (n >> 3) + 2 * u)
    return s


class _Executor:
    """Owns an executor handle."""

    def __init__(self, items):
        self.handle = serve.wc_executor_create(torch.cuda.current_device(), 8, max_items=items)

    def __del__(self):
        try:
            serve.wc_executor_destroy(self.handle)
        except Exception:
            pass


def _uniform(g, lo, hi):
    return lo + (hi - lo) * float(torch.rand((), generator=g))


def _exec_plan(case):
    """Capacities and prefills of the tables, and the requests (table, op, first key, n)."""
    g = torch.Generator()
    g.manual_seed(case["plan"])
    caps = [int(2 ** _uniform(g, case["cap_lo"], case["cap_hi"])) for _ in range(case["tables"])]
    fills = [int(c * _uniform(g, 0.05, 0.6)) for c in caps]
    ends, reqs = list(fills), []  # ends: first key number that a table has not seen
    for i in range(case["items"]):
        t = int(_uniform(g, 0, case["tables"])) % case["tables"]
        n = int(2 ** _uniform(g, case["req_lo"], case["req_hi"]))
        u = _uniform(g, 0.0, 1.0)
        room = int(caps[t] * 0.9) - ends[t]
        if u < 0.6 and room > 0:
            n = min(n, room)
            reqs.append((t, 0, ends[t], n))
            ends[t] += n
        elif u < 0.95:
            reqs.append((t, 1, 0, n))
        else:
            reqs.append((t, 2, 0, min(n, fills[t])))
    return caps, fills, ends, reqs


def _prepare_exec(s, case, seed):
    caps, fills, ends, reqs = _exec_plan(case)
    # retrieves name key numbers up to what is stored by then plus as many absent ones;
    # erases come last in the batch and take prefilled keys, which the next pass puts back
    reqs = [r for r in reqs if r[1] != 2] + [r for r in reqs if r[1] == 2]
    s.tables = [SingleValueTable(4, 4, min_capacity=c, window_width=8) for c in caps]
    for i, (t, f) in enumerate(zip(s.tables, fills)):
        api.wc_insert(t.handle, _keys(_range(f), 4, seed + i), _values(_range(f), 4, seed + i))
    total = sum(r[3] for r in reqs if r[1] == 1)
    s.out = torch.empty(max(1, total), dtype=torch.int32, device="cuda")
    s.found = torch.empty(max(1, total), dtype=torch.uint8, device="cuda")
    s.buffers, s.items, at, put_back = [], [], 0, []
    for t, op, first, n in reqs:
        h, sd = s.tables[t].handle, seed + t
        if op == 1:
            qi = (_range(n) * 0x9E3779B1 + at) % (2 * ends[t])
            qi = torch.where(qi < ends[t], qi, qi + (1 << 29))
            # keys that this batch inserts after this request are not asked for
            seen = fills[t] + sum(w[3] for w in s.items if w[0] == t and w[1] == 0)
            qi = torch.where((qi >= seen) & (qi < ends[t]), qi + (1 << 29), qi)
            k, o, f = _keys(qi, 4, sd), s.out[at:at + n], s.found[at:at + n]
            at += n
            s.buffers.append((k, o, f))
            s.items.append((t, 1, serve.work(1, h, k, values_out=o, found_out=f), n))
        else:
            idx = first + _range(n)
            k, v = _keys(idx, 4, sd), _values(idx, 4, sd)
            s.buffers.append((k, v))
            s.items.append((t, op, serve.work(op, h, k, values=v if op == 0 else None), n))
            if op == 2:
                put_back.append((t, 0, serve.work(0, h, k, values=v), n))
    s.items = [w[2] for w in put_back + s.items]
    s.ex = _Executor(len(s.items))
    return s


# ---- one pass ---------------------------------------------------------------------------

def run(s):
    f = s.family
    if f == "exec":
        serve.wc_executor_submit(s.ex.handle, s.items)
        return s.out, s.found
    h = s.t.handle
    if f == "lookup":
        api.wc_retrieve(h, s.queries, s.out, s.found)
        return s.out, s.found
    api.wc_table_clear(h)
    if f == "sv":
        api.wc_insert(h, s.keys, s.values)
        api.wc_retrieve(h, s.queries, s.out, s.found)
        if not s.case["erase"]:
            return s.out, s.found
        api.wc_erase(h, s.gone)
        api.wc_retrieve(h, s.queries, s.out2, s.found2)
        return s.out, s.found, s.out2, s.found2
    if f == "host":
        api.wc_insert_host(h, s.keys, s.values)
        api.wc_retrieve_host(h, s.queries, s.out, s.found)
        torch.cuda.current_stream().synchronize()  # the results are in host memory then
        return s.out, s.found
    if f in ("set", "bloom"):
        api.wc_insert(h, s.keys, None)
        api.wc_contains(h, s.queries, s.found)
        return s.found
    if f == "count":
        api.wc_insert(h, s.keys, s.weights)
        api.wc_retrieve(h, s.queries, s.out, s.found)
        return s.out, s.found
    api.wc_insert(h, s.keys, s.values)
    total = api.wc_count_values(h, s.queries, s.offsets)  # the caller sizes the output by it
    values = torch.empty(total, dtype=s.values.dtype, device="cuda")
    api.wc_retrieve_multi(h, s.queries, s.offsets, values)
    return s.offsets, values


def work(case):
    """Inputs read once, outputs written once, every stored pair's slot written once, and
    for lookups one 32-byte sector per query or the whole table, whichever is less."""
    f = case["family"]
    if f == "exec":
        _, _, _, reqs = _exec_plan(case)
        per = {0: 16, 1: 4 + 5 + 32, 2: 4 + 8}  # pair + slot; query + result + sector; key + slot
        return {"bytes": sum(per[r[1]] * r[3] for r in reqs), "flops": 0}
    kb, n, q = case["kb"], case["n"], case["queries"]

    def reads(slots, width):
        return min(32 * q, slots * width)

    if f in ("sv", "lookup", "host"):
        slots = case.get("slots") or int(n / case["load"])
        look = q * (2 * kb + 1) + reads(slots, 2 * kb)
        put = n * 4 * kb
        more = look + (n // 2) * 3 * kb if case.get("erase") else 0
        return {"bytes": look + more + (0 if f == "lookup" else put), "flops": 0}
    if f == "set":
        return {"bytes": 2 * n * kb + q * (kb + 1) + reads(int(n / case["load"]), kb), "flops": 0}
    if f == "bloom":
        return {"bytes": n * kb + 10 * n // 8 + q * (kb + 1) + reads(10 * n // 256, 32), "flops": 0}
    u = case["universe"]
    if f == "count":
        return {"bytes": n * kb * (2 if case["weights"] else 1) + 2 * u * kb + q * (2 * kb + 1) + reads(u, 2 * kb),
                "flops": 0}
    vb = case["vb"]
    if f == "mv":  # values stored and read back once, a 16-byte key-store slot per key
        return {"bytes": n * (kb + vb) + n * vb * 3 + 2 * 16 * u + q * (2 * kb + 16), "flops": 0}
    return {"bytes": 3 * n * (kb + vb) + n * vb + q * (2 * kb + 16), "flops": 0}


def exact(case, seed):
    return None
