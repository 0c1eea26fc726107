"""Factor builds of small relations (one CTA each, one launch): rows at the
edges of its warps, of its two sizes and of its limit, keys of every width up
to and beyond one word, payloads, projected columns, and many relations of one
query, against a stable sort."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    c = gj.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("bits", [(0, 0), (1,), (9, 7), (32,), (20, 31), (32, 30), (11, 12, 13, 14), (32, 32, 32)])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1023, 1024, 1025, 4095, 4096, 4097, 12287, 12288, 12289])
def test_factor_equals_a_stable_sort(ctx, n, bits):
    rng = np.random.default_rng(n * 31 + sum(bits))
    cols = []
    for b in bits:
        lo = -(1 << (b - 1)) if b else 7
        x = rng.integers(lo, lo + (1 << b), n, dtype=np.int64)
        x = np.where(rng.random(n) < 0.5, x[0], x)        # repeated keys
        if b and n > 2:
            x[-2:] = lo, lo + (1 << b) - 1
        cols.append(x.astype(np.int32))
    pays = [rng.integers(-2**31, 2**31 - 1, n, dtype=np.int32), rng.integers(-2**62, 2**62, n, dtype=np.int64)]
    dev = lambda x: torch.from_numpy(x).cuda()
    rid = ctx.load_relation([dev(c) for c in cols], list(range(len(cols))), [dev(p) for p in pays])
    order = list(reversed(range(len(cols))))
    for col_order in (None, order):
        by = cols if col_order is None else [cols[c] for c in col_order]
        perm, gstart, gkey = ctx.factor_export(rid, n, len(cols), col_order)
        ref = np.lexsort(tuple(reversed(by)))
        assert np.array_equal(perm.cpu().numpy().view(np.uint32), ref)
        srt = np.stack([c[ref] for c in cols], 1)
        starts = np.flatnonzero(np.concatenate([[True], (srt[1:] != srt[:-1]).any(1)]))
        assert np.array_equal(gstart.cpu().numpy()[:-1], starts) and int(gstart[-1]) == n
        assert np.array_equal(gkey.cpu().numpy().T, srt[starts])
    q = ctx.query([rid])
    ref = np.lexsort(tuple(reversed(cols)))
    got = q.desummarize(0, q.summarize())
    for a, w in zip(got, [c[ref] for c in cols] + [p[ref] for p in pays]):
        assert np.array_equal(a.cpu().numpy(), w)
    q.close()
    ctx.release_relation(rid)


@pytest.mark.parametrize("rows", [(40, 5000, 13000, 900), (1, 12288, 4096, 4097)])
def test_small_and_large_relations_of_one_query(ctx, rows):
    """A chain whose relations take both builds, with and without its ends
    projected away (their columns are then outside the factor's order)."""
    from paper_2206_10435_gb300 import gj
    doms = [50, max(rows) // 2, max(rows) // 2, 3000, 20]
    q = G.chain_query("mixed", rows, doms, [0.0] * 5, np.int64, sum(rows))
    ids = gj.load_query(ctx, q)
    for drop in ((), (0, 4)):
        ref = O.join(q, drop=drop)
        qq = ctx.query(ids, drop_attrs=drop)
        total = qq.summarize()
        assert total == len(ref.rowids)
        cols, rids = qq.desummarize(0, total, rowids=True)
        assert np.array_equal(np.stack([r.cpu().numpy() for r in rids], 1), ref.rowids)
        for a, w in zip(cols, O.columns(q, ref.rowids, drop=drop)):
            assert np.array_equal(a.cpu().numpy(), w)
        qq.close()
    for i in ids:
        ctx.release_relation(i)
