"""Memory that a context keeps between calls: who may hold it, and that it is
given back."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    c = gj.Context(0, torch.cuda.Stream())
    yield c
    c.close()


def _chain(ctx, n):
    """Relations R(0, 1), S(1, 2) of n distinct keys: |Q| = n, and a summary of
    more than 100 bytes a row."""
    a = torch.arange(n, dtype=torch.int32).cuda()
    torch.cuda.synchronize()
    return [ctx.load_relation([a, a], [0, 1]), ctx.load_relation([a, a], [1, 2])]


def test_a_small_summary_does_not_hold_a_large_ones_block(ctx):
    n = 1 << 21
    large, small = _chain(ctx, n), _chain(ctx, 1000)
    big, little = ctx.query(large), ctx.query(small)
    assert big.summarize() == n
    big.close()
    assert little.summarize() == 1000
    held, _ = ctx.pool_usage()
    w, m, o = little.summary_groups(0)
    assert bool((w == 1).all()) and bool((m == 1).all()) and o.tolist() == list(range(1000))
    little.close()
    left, _ = ctx.pool_usage()
    assert held - left <= 8 * MB
    # a large summary after it, and one that takes its block over
    for _ in range(2):
        big = ctx.query(large)
        assert big.summarize() == n
        val, freq, off = big.level(0, n - 5, 5)
        assert val.tolist() == list(range(n - 5, n)) and freq.tolist() == [1] * 5
        big.close()


def test_a_query_on_its_own_stream_gives_its_blocks_back(ctx):
    """Between calls such a query holds its summary and nothing else."""
    n = 1 << 20
    q = ctx.query(_chain(ctx, n))
    q.set_stream(torch.cuda.Stream())
    assert q.summarize() == n
    held, _ = ctx.pool_usage()
    val, freq, off = q.level(2, 0, n)          # a window of all rows
    assert int(val.sum()) == n * (n - 1) // 2
    assert ctx.pool_usage()[0] == held
    q.close()


def test_kept_blocks_serve_another_stream_when_memory_runs_out(ctx):
    """A query with its own stream, on a device that is full but for what the
    context kept from a closed query of the same size."""
    n = 1 << 24
    ids = _chain(ctx, n)
    q = ctx.query(ids)
    assert q.summarize() == n                  # the kernels are loaded by now
    q.close()
    ctx.pool_usage()
    other, first = ctx.query(ids), ctx.query(ids)
    other.set_stream(torch.cuda.Stream())
    assert first.summarize() == n
    first.close()                              # its arrays and scratch are kept
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    filler = torch.empty(max(free - 512 * MB, 1), dtype=torch.int8, device="cuda")
    try:
        assert other.summarize() == n
    finally:
        del filler
        torch.cuda.empty_cache()
    w, m, _ = other.summary_groups(1)
    assert bool((w == 1).all()) and bool((m == 1).all())
    other.close()


def test_idle_blocks_do_not_count_against_a_servers_budget(ctx):
    """A query on its own stream keeps a block from its window; the server's
    budget has room for its requests beside what is in use, but not for that
    block too."""
    from paper_2206_10435_gb300 import gj
    n = 1 << 21
    q = ctx.query(_chain(ctx, n))
    q.set_stream(torch.cuda.Stream())
    assert q.summarize() == n
    ids = _chain(ctx, 20000)
    ctx.query(ids).close()
    ctx.set_option(gj.GJ_OPT_SLOT_ARENA, 32 * MB)
    used, _ = ctx.pool_usage()
    # two slots' arenas, an estimate of about 7 MB a request, and less than the
    # window's 30 bytes a row
    srv = gj.NativeServer(ctx, n_slots=2, hbm_budget=used + 64 * MB + 32 * MB, chunk_rows=1 << 12)
    q.level(2, 0, n)
    res, _ = srv.run([ids] * 4, np.zeros(4))
    assert [(r["status"], r["total"], r["rows"]) for r in res] == [(gj.GJ_OK, 20000, 20000)] * 4
    srv.close()
    q.close()
