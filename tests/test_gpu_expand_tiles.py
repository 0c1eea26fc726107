"""Window expansion at the edges of its scan's tiles (1024 items): frontiers of
1023, 1024, 1025 and a few tiles' items, windows that cut the first and the
last item, runs of every level and a refused capacity, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", ["chain", "star"])
@pytest.mark.parametrize("groups", [1, 31, 1023, 1024, 1025, 4096, 5000])
def test_windows_and_levels(groups, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(groups)
    a = np.arange(groups, dtype=np.int32) - 7
    b = rng.integers(0, 9, groups, dtype=np.int32)
    r = lambda n, d: rng.integers(0, d, n, dtype=np.int32)
    pay = lambda n: [rng.integers(-2**62, 2**62, n, dtype=np.int64)]
    root = G.Relation("R", [0, 1], [a, b], pay(groups))
    second = G.Relation("S", [1, 2], [r(20, 9), r(20, 4)], pay(20))
    third = G.Relation("T", [2 if shape == "chain" else 1, 3],
                       [r(9, 4 if shape == "chain" else 9), r(9, 3)], pay(9))
    q = G.Query(shape, [root, second, third])
    ref = O.join(q)
    cols = O.columns(q, ref.rowids)
    levels = O.gfjs_levels(q, ref.rowids)
    n = len(ref.rowids)
    ctx = gj.Context(0)
    qq = ctx.query(gj.load_query(ctx, q))
    assert qq.summarize() == n
    cuts = sorted(set([0, 1, n // 3, n // 2, max(n - 1, 0)] + list(rng.integers(0, n + 1, 4))))
    for lo in cuts:
        for m in (1, 5, 1000, n - lo):
            if m < 1 or lo >= n:
                continue
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
    last = len(levels) - 1
    runs = len(levels[last].value)
    if runs > 1:
        with pytest.raises(gj.GJError) as e:
            qq.level(last, 0, n, cap=runs - 1)
        assert e.value.status == gj.GJ_ERR_CAPACITY
    ctx.close()
