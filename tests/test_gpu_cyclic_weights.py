"""Block sizes of cyclic queries from weights of the items and candidates (many
blocks) and from the groups' counts in place (few), on one and two cliques,
with repeated rows, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = {"square": [(0, 1), (1, 2), (2, 3), (3, 0)], "pair": [(0, 1, 2), (0, 1, 3), (2, 3)],
          "diamond": [(0, 1), (1, 2), (2, 0), (2, 3), (3, 0)], "pentagon": [(0, 1), (1, 2), (2, 3), (3, 4), (4, 0)]}


# blocks per item and candidate of the last step: many, few, none
@pytest.mark.parametrize("rows,values", [(150, 9), (600, 45), (300, 250), (40, 40)])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_rows_of_dense_and_sparse_cycles(shape, rows, values):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(rows)
    rels = []
    for i, attrs in enumerate(SHAPES[shape]):
        cols = [rng.integers(0, values, rows, dtype=np.int32) for _ in attrs]
        twice = rng.integers(0, rows, rows // 10)          # groups of several rows
        cols = [np.concatenate([c, c[twice]]) for c in cols]
        rels.append(G.Relation(f"R{i}", list(attrs), cols,
                               [rng.integers(-2**62, 2**62, len(cols[0]), dtype=np.int64)]))
    q = G.Query(shape, rels)
    ref = O.join(q)
    cols = O.columns(q, ref.rowids)
    n = len(ref.rowids)
    ctx = gj.Context(0)
    qq = ctx.query(gj.load_query(ctx, q))
    assert qq.summarize() == n
    for lo, m in ((0, n), (n // 3, 2000), (n - 1, 1)):
        if lo < 0 or lo >= n:
            continue
        hi = min(lo + m, n)
        got, rids = qq.desummarize(lo, m, rowids=True)
        assert np.array_equal(np.stack([x.cpu().numpy() for x in rids], 1), ref.rowids[lo:hi])
        for x, w in zip(got, cols):
            assert np.array_equal(x.cpu().numpy(), w[lo:hi])
    ctx.close()
