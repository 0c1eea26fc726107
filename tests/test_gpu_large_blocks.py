"""Windows over blocks of hundreds of thousands of rows (more emit tiles than a
thread block of the expansion maps one by one), next to blocks of a few rows and
cut at every offset in a tile, for each number of rows per thread, against the
oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rpt", [2, 4, 8])
@pytest.mark.parametrize("hops", [2, 3])
def test_windows_over_large_blocks(hops, rpt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(hops)
    # (key, rows left, rows right): blocks of 7, 830001, 1, 6, 420000, 2, 560340, 11 rows
    blocks = [(1, 7, 1), (2, 3, 276667), (5, 1, 1), (6, 2, 3), (9, 600, 700), (10, 2, 1), (11, 660, 849), (12, 1, 11)]
    left = np.repeat([b[0] for b in blocks], [b[1] for b in blocks]).astype(np.int32)
    right = np.repeat([b[0] for b in blocks], [b[2] for b in blocks]).astype(np.int32)
    left, right = rng.permutation(left), rng.permutation(right)
    rels = [G.Relation("L", [0], [left], [rng.integers(-2**62, 2**62, len(left), dtype=np.int64)]),
            G.Relation("R", [0], [right], [rng.integers(-2**31, 2**31, len(right)).astype(np.int32)])]
    if hops == 3:
        key = np.unique(left)
        rels.append(G.Relation("K", [0], [key], [rng.integers(-2**62, 2**62, len(key), dtype=np.int64)]))
    q = G.Query("large", rels)
    ref = O.join(q)
    cols = O.columns(q, ref.rowids)
    n = len(ref.rowids)
    ctx = gj.Context(0)
    ctx.set_option(gj.GJ_OPT_EMIT_ROWS_PER_THREAD, rpt)
    qq = ctx.query(gj.load_query(ctx, q))
    assert qq.summarize() == n == sum(b[1] * b[2] for b in blocks)
    for lo, m in ((0, n), (1, n), (6, 830003), (7, 600000), (131, n - 300), (300001, 1200003), (900000, 262145)):
        hi = min(lo + m, n)
        got, rids = qq.desummarize(lo, m, rowids=True)
        for j, r in enumerate(rids):
            assert np.array_equal(r.cpu().numpy(), ref.rowids[lo:hi, j])
        for x, w in zip(got, cols):
            assert np.array_equal(x.cpu().numpy(), w[lo:hi])
    ctx.close()
