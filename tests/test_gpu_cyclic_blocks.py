"""Blocks of cyclic queries written and placed in one pass: slot tiles (1024) at
their edges, tiles that span more items without slots than are staged, blocks of
several rows, sizes past 2^32 and past 2^64, on one and two cliques and on the
3-cycle, with windows that cut the first and last block, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ring(attrs, m, gap, copies):
    """A cycle whose first attribute takes 0, 1, .., n - 1 in the first relation
    and m values `gap` apart in the last: m blocks, the other items without."""
    rng = np.random.default_rng(m + gap)
    n = max(1, m * gap)
    a = np.arange(n, dtype=np.int32)
    keep = np.repeat((np.arange(m) * gap).astype(np.int32), copies)
    z = lambda k: np.zeros(k, np.int32)
    rels = []
    for i, at in enumerate(attrs):
        if i == 0:
            cols = [a, z(n)]
        elif i == len(attrs) - 1:
            cols = [z(len(keep)), keep]
        else:
            cols = [z(copies), z(copies)]
        rels.append(G.Relation(f"R{i}", list(at), cols,
                               [rng.integers(-2**62, 2**62, len(cols[0]), dtype=np.int64)]))
    return G.Query("ring", rels)


@pytest.mark.parametrize("attrs", [[(0, 1), (1, 2), (2, 0)], [(0, 1), (1, 2), (2, 3), (3, 0)],
                                   [(0, 1), (1, 2), (2, 3), (3, 4), (4, 0)]], ids=["triangle", "square", "pentagon"])
@pytest.mark.parametrize("m,gap,copies", [(1, 1, 1), (1023, 1, 1), (1024, 1, 1), (1025, 3, 1), (700, 9, 2),
                                          (2500, 2, 1), (3, 3000, 3)])
def test_blocks_at_tile_edges(attrs, m, gap, copies):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    q = _ring(attrs, m, gap, copies)
    ref = O.join(q)
    cols = O.columns(q, ref.rowids)
    n = len(ref.rowids)
    ctx = gj.Context(0)
    qq = ctx.query(gj.load_query(ctx, q))
    assert qq.summarize() == n == m * copies ** (len(attrs) - 1)
    for lo, k in ((0, n), (n // 3, n), (1, 1), (n - 1, 5), (max(n // 2 - 3, 0), 1030)):
        if lo >= n:
            continue
        hi = min(lo + k, n)
        got, rids = qq.desummarize(lo, k, rowids=True)
        assert np.array_equal(np.stack([x.cpu().numpy() for x in rids], 1), ref.rowids[lo:hi])
        for x, w in zip(got, cols):
            assert np.array_equal(x.cpu().numpy(), w[lo:hi])
    ctx.close()


@pytest.mark.parametrize("k,rows,total", [(3, 40000, 40000**3), (4, 60000, 60000**4), (4, 70000, None)])
def test_sizes_past_32_and_64_bits(k, rows, total):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    z = np.zeros(rows, np.int32)
    attrs = [(i, (i + 1) % k) for i in range(k)]
    ctx = gj.Context(0)
    qq = ctx.query(gj.load_query(ctx, G.Query("all", [G.Relation(f"R{i}", list(a), [z, z]) for i, a in enumerate(attrs)])))
    if total is None:                    # 70000^4 = 2^64.4
        with pytest.raises(gj.GJError) as e:
            qq.summarize()
        assert e.value.status == gj.GJ_ERR_OVERFLOW
    else:
        assert qq.summarize() == total
    ctx.close()
