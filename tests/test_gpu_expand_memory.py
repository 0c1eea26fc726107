"""Device memory of a window's expansion: at most what the levels' frontiers
took one after the other, 64 bytes a row for three relations, also where the
window has a root group per row; and deeper trees, whose levels share arrays,
against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_a_windows_memory(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    n = 1 << 21
    a = torch.arange(n, dtype=torch.int32).cuda()
    torch.cuda.synchronize()
    path = str(tmp_path / "s")
    ctx = gj.Context(0)
    q = ctx.query([ctx.load_relation([a, a], [i, i + 1]) for i in range(3)])
    assert q.summarize() == n
    q.save(path)
    ctx.close()
    # a context whose pool has held the summary's arrays and nothing else
    ctx = gj.Context(0)
    q = gj.Query.load(ctx, path)
    (tmp_path / "s").unlink()
    out = q.alloc_columns(n)
    q.desummarize(0, 1, out=out)               # the kernels are loaded by now
    ctx.pool_usage()
    torch.cuda.synchronize()
    before, _ = torch.cuda.mem_get_info()
    got = q.desummarize(0, n, out=out)
    after, _ = torch.cuda.mem_get_info()
    assert all(torch.equal(c, a) for c in got)
    # and 48 MB of slack: the pool grows by 32 MB at a time
    assert before - after <= 64 * n + (48 << 20)
    ctx.close()


@pytest.mark.parametrize("k", [4, 5, 6, 9])
@pytest.mark.parametrize("shape", ["chain", "star", "mixed"])
def test_deep_trees(shape, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(5 * k)
    rels = []
    for j in range(k):
        n = 60 if j < 2 else int(rng.integers(5, 9))
        r = lambda d: rng.integers(0, d, n, dtype=np.int32)
        shared = [0] if j == 0 else [{"chain": j, "star": 1, "mixed": max(1, j // 2 + 1)}[shape]]
        rels.append(G.Relation(f"T{j}", shared + [j + 1], [r(5), r(5)],
                               [rng.integers(-2**62, 2**62, n, dtype=np.int64)] if j % 2 else []))
    q = G.Query(shape, rels)
    ref = O.join(q)
    cols = O.columns(q, ref.rowids)
    levels = O.gfjs_levels(q, ref.rowids)
    n = len(ref.rowids)
    ctx = gj.Context(0)
    qq = ctx.query(gj.load_query(ctx, q))
    assert qq.summarize() == n > 0
    for lo, m in ((0, n), (n // 3, max(n // 2, 1)), (n - 1, 1)):
        hi = min(lo + m, n)
        got, rids = qq.desummarize(lo, m, rowids=True)
        assert np.array_equal(np.stack([x.cpu().numpy() for x in rids], 1), ref.rowids[lo:hi])
        for x, w in zip(got, cols):
            assert np.array_equal(x.cpu().numpy(), w[lo:hi])
        for l, lv in enumerate(levels):
            off = lv.offset.astype(np.int64)
            keep = (off >= lo) & (off < hi)
            val, freq, at = qq.level(l, lo, m)
            assert np.array_equal(val.cpu().numpy(), lv.value[keep])
            assert np.array_equal(freq.cpu().numpy(), lv.freq[keep].astype(np.int64))
            assert np.array_equal(at.cpu().numpy(), off[keep])
    ctx.close()
