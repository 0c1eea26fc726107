"""Timed cases of the library: what a program that joins tables with it has it do.

Kinds
-----
``join``     tables in, every result row out: load, plan (which builds the
             factors), summarise, desummarise, release.  What an analytical
             query costs from the first call to the last.
``factor``   one table's frequency table (load, build, export), the step a
             system runs ahead of any query.
``summary``  a query planned and summarised over resident factors, with the
             per-group summary read back: optimiser and statistics use.
``rows``     one window of the result rows of a summarised query: how results
             larger than memory are streamed out.
``levels``   the run-length columns of the sorted result in one window.
``batch``    many small counting queries in one CUDA-graph launch.
``serve``    a burst of requests through the native serving runtime.

Key distributions, domains and payload types are those of the repository's
benchmark workloads and generators (uniform and Zipf keys, Poisson dimension
tables, int32 and int64 payloads).  Outputs go into buffers the program keeps,
as large as the result can be or is expected to be, with the number of
entries written beside them; the rest of a buffer stays zero.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2206_10435_gb300 import datagen, gj

DEV = "cuda:0"
PAYLOAD = {"none": 0, "int32": 4, "int64": 8}


def listed():
    return [
        # the smallest join a serving process sees (the lower end of the batch
        # distribution): launches and synchronisations are all of it
        dict(name="join_tiny", kind="join", shape="chain", tables=3, rows=1000, ratio=1, payload="int32",
             host=False, drop=False),
        # the 3-table chain of 10^4 rows per table (10^6 result rows) for a
        # program whose tables and results live in pinned host memory
        dict(name="join_host_chain3", kind="join", shape="chain", tables=3, rows=10000, ratio=10,
             payload="int32", host=True, drop=False),
        # a fact table joined to four dimensions (1.6e8 rows out)
        dict(name="join_star", kind="join", shape="star", tables=5, rows=9999991, ratio=10, payload="int64",
             host=False, drop=False),
        # the two cyclic shapes of the benchmark: the 3-cycle ...
        dict(name="join_triangle", kind="join", shape="triangle", tables=3, rows=400003, ratio=400,
             payload="int64", host=False, drop=False),
        # ... and the 4-cycle
        dict(name="join_square", kind="join", shape="square", tables=4, rows=80000, ratio=80,
             payload="int64", host=False, drop=False),
        # a skewed two-key table of the 5-table chain workload
        dict(name="factor_chain", kind="factor", rows=10000000, keys=2, domain=1000000, zipf=1.1,
             payload="int64"),
        # a fact table whose key needs more than one 64-bit word
        dict(name="factor_wide", kind="factor", rows=30000001, keys=4, domain=1000000, zipf=0.0,
             payload="int64"),
        # the 5-table chain workload, 10^7 rows per table: its summary ...
        dict(name="summary_chain5", kind="summary", tables=5, rows=10000000, domain=1000000, zipf=1.1),
        # ... and one large window of its 1.1e10 result rows
        dict(name="rows_chain5", kind="rows", tables=5, rows=10000000, domain=1000000, zipf=1.1,
             payload="int64", window=100000003),
        # the run-length columns of the same result
        dict(name="levels_chain5", kind="levels", tables=5, rows=10000000, domain=1000000, zipf=1.1,
             window=20000003),
        # counting queries of the batch workload, replayed as one graph
        dict(name="batch_256", kind="batch", queries=256),
        # a burst of the same queries through the serving runtime, up to 2^20
        # rows of each result streamed
        dict(name="serve_192", kind="serve", queries=192, max_rows=1 << 20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["join", "join", "join", "factor", "factor", "summary", "rows", "rows", "levels", "batch",
                       "serve"])
    if kind == "join":
        shape = rng.choice(["chain", "chain", "star", "triangle", "square"])
        c = dict(kind=kind, shape=shape, payload=rng.choice(["none", "int32", "int64"]), host=False, drop=False)
        if shape == "chain":
            k = rng.randint(3, 5)
            rows = _log(rng, 1000, 300000)
            # about 3e7 result rows at most
            top = min(10.0, (3e7 / rows) ** (1.0 / (k - 1)))
            c.update(tables=k, rows=rows, ratio=max(1, int(rng.uniform(1, top))), drop=rng.random() < 0.3)
            if rows <= 30000:
                c["host"] = rng.random() < 0.3
        elif shape == "star":
            c.update(tables=rng.randint(3, 5), rows=_log(rng, 100000, 8000000), ratio=rng.choice([10, 30, 100]))
        elif shape == "triangle":
            c.update(tables=3, rows=_log(rng, 10000, 400000))
            c["ratio"] = max(1, c["rows"] // 1000)
        else:
            c.update(tables=4, rows=_log(rng, 5000, 80000))
            c["ratio"] = max(1, c["rows"] // 1000)
        return c
    if kind == "factor":
        keys = rng.randint(1, 4)
        rows = _log(rng, 1000, 20000000)
        return dict(kind=kind, rows=rows, keys=keys, domain=_log(rng, 1000, 1000000),
                    zipf=rng.choice([0.0, 0.8, 1.1]), payload=rng.choice(["none", "int32", "int64"]))
    if kind in ("summary", "rows", "levels"):
        rows = _log(rng, 10000, 10000000)
        c = dict(kind=kind, tables=rng.randint(3, 5), rows=rows, domain=max(100, int(rows / rng.uniform(5, 20))),
                 zipf=rng.choice([0.0, 0.8, 1.1]))
        if kind == "rows":
            c.update(payload=rng.choice(["none", "int32", "int64"]), window=_log(rng, 30000, 80000000))
        if kind == "levels":
            c["window"] = _log(rng, 30000, 20000000)
        return c
    if kind == "batch":
        return dict(kind=kind, queries=_log(rng, 8, 200))
    return dict(kind=kind, queries=_log(rng, 16, 160), max_rows=1 << rng.choice([16, 20]))


# ------------------------------------------------------------------- inputs

_CDF: dict = {}


def _keys(g, n, domain, zipf):
    """n int32 keys over [0, domain): uniform, or Zipf with the ranks permuted."""
    if zipf == 0.0:
        return torch.randint(0, domain, (n,), generator=g, device=DEV, dtype=torch.int32)
    cdf = _CDF.get((zipf, domain))
    if cdf is None:
        cdf = torch.cumsum(torch.arange(1, domain + 1, device=DEV, dtype=torch.float64) ** -zipf, 0)
        cdf /= cdf[-1].clone()
        _CDF.clear()
        _CDF[(zipf, domain)] = cdf
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    rank = torch.searchsorted(cdf, u, right=True).clamp_(max=domain - 1)
    return torch.randperm(domain, generator=g, device=DEV)[rank].to(torch.int32)


def _payloads(g, n, kind):
    if kind == "none":
        return []
    if kind == "int32":
        return [torch.randint(-2**31, 2**31 - 1, (n,), generator=g, device=DEV, dtype=torch.int32)]
    return [torch.randint(-2**62, 2**62, (n,), generator=g, device=DEV, dtype=torch.int64)]


def _domain(case):
    """Values of a join's shared attributes: rows / ratio."""
    return max(1, case["rows"] // case["ratio"])


def _tables(case, seed):
    """[(attributes, key columns, payload columns)], root first."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    kind, payload = case["kind"], case.get("payload", "none")
    if kind == "factor":
        n = case["rows"]
        return [(list(range(case["keys"])), [_keys(g, n, case["domain"], case["zipf"]) for _ in range(case["keys"])],
                 _payloads(g, n, payload))]
    n = case["rows"]
    if kind in ("summary", "rows", "levels"):
        d, z = case["domain"], case["zipf"]
        return [([i, i + 1], [_keys(g, n, d, z), _keys(g, n, d, z)], _payloads(g, n, payload))
                for i in range(case["tables"])]
    d, k = _domain(case), case["tables"]
    if case["shape"] == "chain":       # end attributes over as many values as rows
        dom = [n] + [d] * (k - 1) + [n]
        return [([i, i + 1], [_keys(g, n, dom[i], 0.0), _keys(g, n, dom[i + 1], 0.0)], _payloads(g, n, payload))
                for i in range(k)]
    if case["shape"] == "star":        # Poisson(2) copies of every dimension key
        out = [(list(range(k - 1)), [_keys(g, n, d, 0.0) for _ in range(k - 1)], _payloads(g, n, payload))]
        for j in range(k - 1):
            reps = torch.poisson(torch.full((d,), 2.0, device=DEV), generator=g).to(torch.int64)
            keys = torch.repeat_interleave(torch.arange(d, device=DEV, dtype=torch.int32), reps)
            keys = keys[torch.randperm(keys.numel(), generator=g, device=DEV)].contiguous()
            out.append(([j], [keys], _payloads(g, keys.numel(), payload)))
        return out
    attrs = [(0, 1), (1, 2), (2, 0)] if case["shape"] == "triangle" else [(0, 1), (1, 2), (2, 3), (3, 0)]
    return [(list(a), [_keys(g, n, d, 0.0), _keys(g, n, d, 0.0)], _payloads(g, n, payload)) for a in attrs]


def _requests(case, seed):
    """Chain queries of the batch distribution, [[(attributes, key columns)]]."""
    return datagen.batch_queries_torch(seed, case["queries"], device=DEV)


def _expected_rows(case):
    """Result rows of a join, on average over the seeds."""
    n, r, k = case["rows"], _matches(case), case["tables"]
    if case["shape"] == "chain":
        return n * r ** (k - 1)
    if case["shape"] == "star":
        return n * 2.0 ** (k - 1)
    return r ** k


def _matches(case):
    """Rows of one table per value of a shared attribute."""
    return case["rows"] / _domain(case)


def _row_bytes(case):
    k, p = case["tables"], PAYLOAD[case.get("payload", "none")]
    kind, shape = case["kind"], case.get("shape", "chain")
    n_vars = {"chain": k + 1, "star": k - 1, "triangle": 3, "square": 4}[shape] if kind == "join" else k + 1
    if case.get("drop"):
        n_vars -= 2
    return 4 * n_vars + p * k


def prepare(case, seed):
    kind = case["kind"]
    ctx = gj.Context(0)
    state = {"case": case, "ctx": ctx}
    if kind in ("batch", "serve"):
        tables = _requests(case, seed)
        ids = [[ctx.load_relation(keys, attrs) for attrs, keys in q] for q in tables]
        if kind == "batch":
            state["batch"] = gj.Batch(ctx, ids)
        else:
            for q in ids:              # the factors are built ahead of the requests
                ctx.query(q).close()
            state.update(ids=ids, arrivals=[0.0] * len(ids),
                         server=gj.NativeServer(ctx, max_rows=case["max_rows"]))
        return state
    tables = _tables(case, seed)
    if kind == "join":
        if case["host"]:
            tables = [(a, [x.cpu().pin_memory() for x in ks], [x.cpu().pin_memory() for x in ps])
                      for a, ks, ps in tables]
        state["out"] = [torch.zeros(_capacity(case), dtype=t, pin_memory=True) if case["host"]
                        else torch.zeros(_capacity(case), dtype=t, device=DEV) for t in _column_types(case)]
        state["tables"] = tables
        return state
    if kind == "factor":
        n, nk = case["rows"], case["keys"]
        state["tables"] = tables
        state["out"] = [torch.zeros(m, dtype=torch.int32, device=DEV) for m in (n, n + 1, nk * n)]
        return state
    ids = [ctx.load_relation(ks, a, ps) for a, ks, ps in tables]
    query = ctx.query(ids)
    state["ids"] = ids
    if kind == "summary":
        query.close()                  # the factors stay
        state["out"] = [[torch.zeros(case["rows"], dtype=torch.int64, device=DEV) for _ in range(3)] for _ in ids]
        return state
    total = query.summarize()
    n = min(case["window"], total)
    row0 = int(np.random.default_rng(seed).integers(0, total - n + 1))
    state.update(query=query, row0=row0, n=n)
    if kind == "rows":
        state["out"] = [torch.zeros(case["window"], dtype=t, device=DEV) for t in _column_types(case)]
    else:
        state["out"] = [[torch.zeros(case["window"], dtype=t, device=DEV)
                         for t in (torch.int32, torch.int64, torch.int64)] for _ in query.var_attr]
    return state


def _capacity(case):
    """Result rows a join's program has room for."""
    return int(1.2 * _expected_rows(case)) + 4096


def _column_types(case):
    n_vars = (_row_bytes(case) - PAYLOAD[case["payload"]] * case["tables"]) // 4
    pay = {"none": [], "int32": [torch.int32], "int64": [torch.int64]}[case["payload"]]
    return [torch.int32] * n_vars + pay * case["tables"]


# --------------------------------------------------------------------- runs

def _call(status, what):
    if status:
        raise gj.GJError(status, what)


def _address(t):
    return ctypes.c_void_p(t.data_ptr())


def run(state):
    return _RUN[state["case"]["kind"]](state)


def _run_join(state):
    ctx, case = state["ctx"], state["case"]
    flags = gj.GJ_REL_HOST if case["host"] else gj.GJ_REL_BORROW
    ids = [ctx.load_relation(ks, a, ps, flags=flags) for a, ks, ps in state["tables"]]
    query = ctx.query(ids, drop_attrs=(0, case["tables"]) if case["drop"] else ())
    total = query.summarize()
    columns = query.desummarize(0, min(total, _capacity(case)), out=state["out"])
    query.close()
    for i in ids:
        ctx.release_relation(i)
    return [total, int(columns[0].shape[0]), state["out"]]


def _run_factor(state):
    ctx, out = state["ctx"], state["out"]
    attrs, keys, pays = state["tables"][0]
    rid = ctx.load_relation(keys, attrs, pays)
    ctx.build_factors(rid)
    groups = ctypes.c_int64()
    _call(gj.lib().gj_factor_export(ctx.h, rid, None, ctypes.byref(groups), *map(_address, out)),
          "gj_factor_export")
    ctx.release_relation(rid)
    return [groups.value, out]


def _run_summary(state):
    query = state["ctx"].query(state["ids"])
    total = query.summarize()
    for j, out in enumerate(state["out"]):
        _call(gj.lib().gj_summary_groups(query.h, j, *map(_address, out)), "gj_summary_groups")
    groups = list(query.n_groups)
    query.close()
    return [total, groups, state["out"]]


def _run_rows(state):
    columns = state["query"].desummarize(state["row0"], state["n"], out=state["out"])
    return [int(columns[0].shape[0]), state["out"]]


def _run_levels(state):
    q, runs = state["query"], []
    for l, out in enumerate(state["out"]):
        n = ctypes.c_uint64()
        _call(gj.lib().gj_level(q.h, l, state["row0"], state["n"], *map(_address, out), state["case"]["window"],
                                ctypes.byref(n)), "gj_level")
        runs.append(n.value)
    return [runs, state["out"]]


def _run_batch(state):
    state["batch"].run()
    return [state["batch"].totals, state["batch"].status]


def _run_serve(state):
    results, _ = state["server"].run(state["ids"], state["arrivals"])
    return [np.array([r[f] for r in results], dtype=np.uint64).view(np.int64)
            for f in ("total", "status", "rows", "hash")]


_RUN = {"join": _run_join, "factor": _run_factor, "summary": _run_summary, "rows": _run_rows,
        "levels": _run_levels, "batch": _run_batch, "serve": _run_serve}


# --------------------------------------------------------------------- work

def _distinct(rows, domain, keys, zipf):
    """About how many distinct key tuples a table holds."""
    cells = float(domain) ** keys
    if zipf == 0.0:
        return cells * -math.expm1(-rows / cells)
    return 0.45 * min(rows, cells)


def _log_mean(lo, hi):
    return (hi - lo) / math.log(hi / lo)


def work(case):
    """Bytes: inputs read once, outputs written once.  The path adds and
    multiplies integers; its operations are counted as none."""
    kind, k = case["kind"], case.get("tables", 1)
    if kind == "join":
        n, p = case["rows"], PAYLOAD[case["payload"]]
        if case["shape"] == "star":
            d = _domain(case)
            inputs = n * (4 * (k - 1) + p) + 2 * d * (k - 1) * (4 + p)
        else:
            inputs = k * n * (8 + p)
        b = inputs + _expected_rows(case) * _row_bytes(case)
    elif kind == "factor":
        n, nk = case["rows"], case["keys"]
        groups = _distinct(n, case["domain"], nk, case["zipf"])
        b = n * (4 * nk + 4 + 2 * PAYLOAD[case["payload"]]) + groups * (4 * nk + 4)
    elif kind == "summary":
        # per group: two keys and a count read, w, mult and off written
        b = k * _distinct(case["rows"], case["domain"], 2, case["zipf"]) * (8 + 4 + 3 * 8)
    elif kind == "rows":
        b = case["window"] * _row_bytes(case)
    elif kind == "levels":
        # runs of (value, frequency, offset); a row starts a run of the last
        # level every eight rows or so, and each level above has half as many
        b = 2 * case["window"] / 8 * 20
    else:
        rows = case["queries"] * 4.5 * _log_mean(10**3, 10**6)
        b = 8 * rows + 12 * case["queries"]
        if kind == "serve":
            # the factors' groups read, the streamed columns written
            b += 0.75 * case["queries"] * case["max_rows"] * 5.5 * 4
    return {"bytes": float(b), "flops": 0.0}


# -------------------------------------------------------------------- exact

def _pad(x, size):
    x = x.reshape(-1)[:size]
    return torch.cat([x, torch.zeros(size - x.numel(), dtype=x.dtype, device=x.device)])


def _sorted_groups(keys):
    """Rows ordered by their key tuple (ties by row): the order, each group's
    first position and its key values."""
    n = keys[0].numel()
    order = torch.arange(n, device=keys[0].device)
    for col in reversed(keys):
        order = order[torch.sort(col[order], stable=True)[1]]
    head = torch.zeros(n, dtype=torch.bool, device=order.device)
    head[0] = True
    for col in keys:
        c = col[order]
        head[1:] |= c[1:] != c[:-1]
    start = torch.nonzero(head).flatten()
    end = torch.cat([start[1:], torch.tensor([n], device=order.device)])
    return order, start, end - start, [col[order[start]] for col in keys]


def _exact_factor(case, seed):
    _, keys, _ = _tables(case, seed)[0]
    order, start, _, key = _sorted_groups(keys)
    n = keys[0].numel()
    start = torch.cat([start, torch.tensor([n], device=order.device)])
    return [start.numel() - 1, [order.to(torch.int32), _pad(start.to(torch.int32), n + 1),
                                _pad(torch.stack(key), len(key) * n)]]


def _join_rowids(tables):
    """Row ids of every result row, in row-id order (relation 0 slowest)."""
    parts, chunk = [], 2000
    sizes = [t[1][0].numel() for t in tables]
    index = []
    held: dict = {}                       # attribute -> (relation, column) that first holds it
    for j, (attrs, keys, _) in enumerate(tables):
        shared = [i for i, a in enumerate(attrs) if a in held] if j else []
        src = [held[attrs[i]] for i in shared]
        word = torch.zeros(sizes[j], dtype=torch.int64, device=DEV)
        for i in shared:
            word = word * 2**31 + keys[i]
        sort, order = torch.sort(word, stable=True)
        index.append((src, sort, order))
        for i, a in enumerate(attrs):
            held.setdefault(a, (j, i))
    chunk = max(chunk, sizes[0] // 40)
    for lo in range(0, sizes[0], chunk):
        rows = [torch.arange(lo, min(lo + chunk, sizes[0]), device=DEV)]
        for j in range(1, len(tables)):
            src, sort, order = index[j]
            want = torch.zeros_like(rows[0])
            for rel, col in src:
                want = want * 2**31 + tables[rel][1][col][rows[rel]]
            first = torch.searchsorted(sort, want)
            count = torch.searchsorted(sort, want, right=True) - first
            at = torch.repeat_interleave(torch.arange(want.numel(), device=DEV), count)
            step = torch.arange(at.numel(), device=DEV) - (torch.cumsum(count, 0) - count)[at]
            rows = [r[at] for r in rows] + [order[first[at] + step]]
        parts.append(rows)
    return [torch.cat([p[j] for p in parts]) for j in range(len(tables))]


def _exact_join(case, seed):
    if _expected_rows(case) > 2e8:
        return None
    tables = _tables(case, seed)
    rows = _join_rowids(tables)
    # the result's key columns: attributes in order of first appearance
    seen, columns = set(), []
    for j, (attrs, keys, _) in enumerate(tables):
        for a, key in zip(attrs, keys):
            if a not in seen:
                seen.add(a)
                if not (case["drop"] and a in (0, case["tables"])):
                    columns.append((j, key))
    order = None
    for j, key in reversed(columns):
        c = key[rows[j]]
        order = torch.sort(c, stable=True)[1] if order is None else order[torch.sort(c[order], stable=True)[1]]
    rows = [r[order] for r in rows]
    out = [key[rows[j]] for j, key in columns]
    out += [p[rows[j]] for j, (_, _, pays) in enumerate(tables) for p in pays]
    n, cap = rows[0].numel(), _capacity(case)
    return [n, min(n, cap), [_pad(c.cpu() if case["host"] else c, cap) for c in out]]


class _Chain:
    """The summary of a chain join in 64-bit integers, and the decoding of
    result rows from it."""

    def __init__(self, case, seed):
        self.tables = _tables(case, seed)
        k, d = case["tables"], case["domain"]
        self.order, self.start, self.count, self.key = zip(*[_sorted_groups(t[1]) for t in self.tables])
        self.w, self.msg = [None] * k, [None] * k
        for j in reversed(range(k)):
            self.w[j] = self.count[j] if j == k - 1 else self.count[j] * self.msg[j + 1][self.key[j][1].long()]
            self.msg[j] = torch.zeros(d, dtype=torch.int64, device=DEV).index_add_(0, self.key[j][0].long(), self.w[j])
        self.incl = [torch.cumsum(w, 0) for w in self.w]
        values = torch.arange(d, device=DEV, dtype=torch.int32)
        self.base = []                    # weight before the first group of each value
        for j in range(k):
            first = torch.searchsorted(self.key[j][0].contiguous(), values)
            before = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), self.incl[j]])
            self.base.append(before[first])
        self.total = int(self.incl[0][-1])

    def groups(self):
        out, down = [], None
        for j, w in enumerate(self.w):
            v = self.key[j][0].long()
            excl = self.incl[j] - w
            mult = w if j == 0 else w * down[v]
            off = excl if j == 0 else excl - self.base[j][v]
            if j + 1 < len(self.w):
                share = self.count[j] if j == 0 else self.count[j] * down[v]
                down = torch.zeros_like(self.msg[j]).index_add_(0, self.key[j][1].long(), share)
            out.append([w, mult, off])
        return out

    def path(self, rows):
        """Groups of result rows, and each row's place within its key path."""
        g, m, rem = [], None, rows
        for j in range(len(self.w)):
            if j == 0:
                at = torch.searchsorted(self.incl[0], rem, right=True)
                rem = rem - (self.incl[0][at] - self.w[0][at])
                m = self.count[0][at]
            else:
                base = self.base[j][self.key[j - 1][1][g[-1]].long()]
                at = torch.searchsorted(self.incl[j], base + rem // m, right=True)
                rem = rem - (self.incl[j][at] - self.w[j][at] - base) * m
                m = m * self.count[j][at]
            g.append(at)
        return g, rem

    def values(self, g):
        return [self.key[0][0][g[0]]] + [self.key[j][1][x] for j, x in enumerate(g)]

    def columns(self, rows):
        g, rem = self.path(rows)
        out, pay = self.values(g), []
        for j in reversed(range(len(g))):
            c = self.count[j][g[j]]
            row = self.order[j][self.start[j][g[j]] + rem % c]
            rem = rem // c
            pay = [p[row] for p in self.tables[j][2]] + pay
        return out + pay


def _window(case, seed, total):
    n = min(case["window"], total)
    return int(np.random.default_rng(seed).integers(0, total - n + 1)), n


def _exact_summary(case, seed):
    c = _Chain(case, seed)
    groups = c.groups()
    return [c.total, [g[0].numel() for g in groups], [[_pad(x, case["rows"]) for x in g] for g in groups]]


def _exact_rows(case, seed):
    c = _Chain(case, seed)
    row0, n = _window(case, seed, c.total)
    parts = [c.columns(torch.arange(lo, min(lo + (1 << 23), row0 + n), device=DEV))
             for lo in range(row0, row0 + n, 1 << 23)]
    return [n, [_pad(torch.cat(p), case["window"]) for p in zip(*parts)]]


def _exact_levels(case, seed):
    c = _Chain(case, seed)
    row0, n = _window(case, seed, c.total)
    lo, hi = max(row0 - 1, 0), min(row0 + n, c.total - 1)
    rows = torch.arange(lo, hi + 1, device=DEV)
    values = c.values(c.path(rows)[0])
    change = torch.zeros(rows.numel(), dtype=torch.bool, device=DEV)
    change[0] = lo == row0                # row 0 of the result starts a run
    runs, out = [], []
    for l, v in enumerate(values):
        change[1:] |= v[1:] != v[:-1]
        starts = rows[change]
        inside = (starts >= row0) & (starts < row0 + n)
        first = starts[inside]
        runs.append(first.numel())
        if first.numel() == 0:
            out.append([_pad(x, case["window"]) for x in (v[:0], first, first)])
            continue
        # the last run ends past the window: the first later row whose
        # prefix differs
        a, b = int(first[-1]), c.total
        prefix = [x[a - lo] for x in values[:l + 1]]
        while b - a > 1:
            m = (a + b) // 2
            here = c.values(c.path(torch.tensor([m], device=DEV))[0])[:l + 1]
            if all(bool(x[0] == p) for x, p in zip(here, prefix)):
                a = m
            else:
                b = m
        end = torch.cat([first[1:], torch.tensor([b], device=DEV)])
        out.append([_pad(x, case["window"]) for x in (v[first - lo], end - first, first)])
    return [runs, out]


def _exact_totals(case, seed):
    """Join size of every request: 64-bit integers wrap, so the same sums in
    floating point tell which sizes reach 2^64 - 1."""
    totals, status = [], []
    for tables in _requests(case, seed):
        msg = None
        for _, (a, b) in reversed(tables):
            d = 10**5 + 1
            a, b = a.long(), b.long()
            w = [torch.ones_like(a), torch.ones(a.shape, dtype=torch.float64, device=DEV)] if msg is None else \
                [m[b] for m in msg]
            msg = [torch.zeros(d, dtype=x.dtype, device=DEV).index_add_(0, a, x) for x in w]
        over = msg[1].sum() >= 2.0**64
        totals.append(torch.where(over, torch.tensor(-1, device=DEV), msg[0].sum()))
        status.append(over.to(torch.int32) * gj.GJ_ERR_OVERFLOW)
    return torch.stack(totals), torch.stack(status)


def _exact_batch(case, seed):
    return list(_exact_totals(case, seed))


def _exact_serve(case, seed):
    total, status = (x.cpu() for x in _exact_totals(case, seed))
    rows = torch.where(status == 0, torch.clamp(total, 0, case["max_rows"]), 0)
    # a size from 2^63 on is negative as a signed word, and streams in full
    rows = torch.where((status == 0) & (total < 0), torch.tensor(case["max_rows"]), rows)
    return [total, status.long(), rows, None]


_EXACT = {"join": _exact_join, "factor": _exact_factor, "summary": _exact_summary, "rows": _exact_rows,
          "levels": _exact_levels, "batch": _exact_batch, "serve": _exact_serve}


def exact(case, seed):
    """What run() returns for these inputs, as torch's integers give it."""
    return _EXACT[case["kind"]](case, seed)
