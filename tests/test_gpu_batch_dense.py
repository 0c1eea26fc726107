"""Batched counting over value accumulators: chunk edges, shared slots owned
by first arrival (ranges above the slots), sums past 2^32 and saturation, and
the sorted path that sparse key ranges keep, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CAP = (1 << 64) - 1


def _spread(q, step, base):
    """Every key value v becomes v * step + base: the same join, wider ranges."""
    rels = [G.Relation(R.name, list(R.attrs), [(k.astype(np.int64) * step + base).astype(np.int32) for k in R.keys])
            for R in q.relations]
    return G.Query(q.name, rels)


def _queries(case):
    if case == "edges":       # rows around the chunk, the slot minimum and one thread row
        rows = [1, 511, 512, 513, 2048, 16383, 16384, 16385, 40000]
        return [G.chain_query(f"e{i}", [n, rows[-1 - i], 700], [50, 2048, 2049, 300], [0.0] * 4, None, 900 + i)
                for i, n in enumerate(rows)]
    if case == "skew":        # ranges above the slots, frequent values owning theirs
        return [G.chain_query(f"s{i}", [30000, 20011, 17000], [9000, 20000, 6000, 9000], [s] * 4, None, 30 + i)
                for i, s in enumerate((0.0, 0.7, 1.5))]
    if case == "big":         # 600^6 = 2^55.4 exact, 600^8 = 2^73.8 saturated, and a dead branch above it
        z = lambda n, v=0: np.full(n, v, np.int32)
        chain = lambda k: [G.Relation(f"R{i}", [i, i + 1], [z(600), z(600)]) for i in range(k)]
        dead = [G.Relation("D", [100, 0], [z(5), z(5, 7)])] + chain(8)
        return [G.Query("exact", chain(6)), G.Query("over", chain(8)), G.Query("dead", dead)]
    if case == "sparse":      # value ranges far above the rows: the sorted path
        return [_spread(G.chain_query(f"w{i}", [3000, 2000, 1000], [40, 30, 200, 50], [0.5] * 4, None, 60 + i),
                        1000003, -2**27) for i in range(3)]
    # a parent with children on both of its columns, and a one-column relation
    rng = np.random.default_rng(5)
    r = lambda n, d: rng.integers(-d, d, n, dtype=np.int32)
    return [G.Query("tree", [G.Relation("P", [0, 1], [r(5000, 300), r(5000, 40)]),
                             G.Relation("A", [0, 2], [r(3000, 300), r(3000, 9)]),
                             G.Relation("B", [1], [r(700, 40)]),
                             G.Relation("C", [1, 3], [r(900, 40), r(900, 5)])])]


@pytest.mark.parametrize("case", ["edges", "skew", "big", "sparse", "tree"])
def test_batch_totals_equal_the_oracle(case):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    ctx = gj.Context(0)
    queries = _queries(case)
    ref = [O.count(q) for q in queries]
    b = gj.Batch(ctx, [gj.load_query(ctx, q) for q in queries])
    for use_graph in (False, True, True):
        b.totals.zero_()
        b.run(use_graph=use_graph)
        torch.cuda.synchronize()
        got = [int(x) for x in b.totals.cpu().numpy().view(np.uint64)]
        assert got == [CAP if r.overflow else r.total for r in ref]
        assert b.status.tolist() == [gj.GJ_ERR_OVERFLOW if r.overflow else gj.GJ_OK for r in ref]
    ctx.close()
