"""Requests that fail on a device allocation, at every one they make in turn:
the rows reported are those of the chunks that went well, without a hash, and
the next request on the slot is answered."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_10435_gb300 import datagen as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_a_failed_request_reports_the_rows_before_it():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    ctx = gj.Context(0, torch.cuda.Stream())
    q = G.chain_query("f", [900, 700, 800], [40, 30, 30, 40], [0.5] * 4, np.int64, 77)
    total, chunk, chunks = O.count(q).total, 1 << 12, 5
    ids = gj.load_query(ctx, q)
    ctx.query(ids).close()
    limit = chunks * chunk
    assert total > limit

    def serve(fail_at):
        ctx.set_option(gj.GJ_OPT_FAIL_ALLOC_AT, fail_at)
        srv = gj.NativeServer(ctx, n_slots=1, chunk_rows=chunk, max_rows=limit)
        ctx.set_option(gj.GJ_OPT_FAIL_ALLOC_AT, 0)
        res, _ = srv.run([ids, ids], np.zeros(2))
        srv.close()
        return res

    want = serve(0)
    key = lambda r: (r["status"], r["total"], r["rows"], r["hash"])
    assert key(want[0]) == key(want[1]) and want[0]["rows"] == limit and want[0]["hash"] != 0
    seen = set()
    for n in range(1, 200):
        first, second = serve(n)
        assert key(second) == key(want[0]) or first["status"] == gj.GJ_OK
        if first["status"] == gj.GJ_OK:
            assert key(first) == key(want[0])
            break
        assert first["status"] == gj.GJ_ERR_OOM and first["hash"] == 0
        assert first["rows"] % chunk == 0 and first["rows"] < limit
        seen.add(first["rows"])
    assert seen == {i * chunk for i in range(chunks)}
    for i in ids:
        ctx.release_relation(i)
    ctx.close()
