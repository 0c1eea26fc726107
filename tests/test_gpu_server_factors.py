"""Factors built while a server runs, and just before it: the slots' streams do
not wait on the context's, so a factor has to be complete when it is handed
out.  Tables above the small build's size with repeated keys (their key columns
move to the group count after the group counts are known), with payloads, one
with a key of three words, and an empty one: each request equals the same
request over factors built and waited for beforehand."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _tables(seed):
    rng = np.random.default_rng(seed)
    n = 1 << 18
    i32 = lambda lo, hi, m: rng.integers(lo, hi, m, dtype=np.int64).astype(np.int32)
    pay = lambda m: [rng.integers(-2**62, 2**62, m, dtype=np.int64), i32(-9, 9, m)]
    # the wide table's other columns use all 32 bits: with the separator they
    # make three words; few distinct rows, so that groups hold many
    wide = np.stack([i32(0, 500, 3000)] + [i32(-2**31, 2**31, 3000) for _ in range(4)])
    wide = wide[:, rng.integers(0, 3000, n // 4)]
    return [([i32(0, 300, n), i32(0, 400, n)], [0, 1], pay(n)),
            ([i32(0, 400, n), i32(0, 500, n)], [1, 2], pay(n)),
            (list(wide), [2, 3, 4, 5, 6], pay(n // 4)),
            ([i32(0, 500, 0)], [2], pay(0))]


@pytest.mark.parametrize("ahead", [False, True])
def test_requests_over_fresh_factors(ahead):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    ctx = gj.Context(0, torch.cuda.Stream())
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    chunk, limit = 1 << 14, 3 << 14
    srv = gj.NativeServer(ctx, n_slots=4, chunk_rows=chunk, max_rows=limit)
    for seed in range(6):
        T = _tables(seed)
        cols = [([dev(k) for k in keys], attrs, [dev(p) for p in pays]) for keys, attrs, pays in T]
        torch.cuda.synchronize()

        def load():
            ids = [ctx.load_relation(k, a, p) for k, a, p in cols]
            return ids, [ids[:2], ids[1:3], ids[:3], ids[:2] + ids[3:]]

        ids, queries = load()
        for q in queries:
            ctx.query(q).close()
        torch.cuda.synchronize()
        want, _ = srv.run(queries, np.arange(len(queries)) * 0.05)
        new, queries = load()
        if ahead:
            for q in queries:
                ctx.query(q).close()
        got, _ = srv.run(queries, np.zeros(len(queries)))
        for a, b in zip(want, got):
            assert a["status"] == b["status"] == gj.GJ_OK
            assert (a["total"], a["rows"], a["hash"]) == (b["total"], b["rows"], b["hash"])
        assert [r["total"] > 0 for r in want] == [True, True, True, False]
        for i in ids + new:
            ctx.release_relation(i)
    srv.close()
    ctx.close()
