"""Links through a table of entries and through one of segments alone, around
the line between them, and the device memory that a summary takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _query(ctx, parent, child):
    """R(0, 1) with a row per entry of parent, S(1, 2) with one per entry of
    child: every row is a group."""
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).cuda()
    ids = [ctx.load_relation([dev(np.arange(len(parent))), dev(parent)], [0, 1]),
           ctx.load_relation([dev(child), dev(np.arange(len(child)))], [1, 2])]
    torch.cuda.synchronize()
    return ctx.query(ids)


@pytest.mark.parametrize("over", [-1, 0, 1, 2000])
@pytest.mark.parametrize("n", [1, 700, 5000])
def test_links_around_the_line(n, over):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(n + over)
    line = 2 * n + 1024                 # entries up to here, then segments
    width = line + over
    child = rng.integers(0, width, n)
    child[0] = 0
    if n > 1:
        child[-1] = width - 1
    child = child - 2**31               # values at the lower end of the type
    parent = rng.choice(np.concatenate([child, [2**31 - 1, child.max() + 1]]), n)
    ctx = gj.Context(0)
    q = _query(ctx, parent, child)
    values, count = np.unique(child, return_counts=True)
    msg = dict(zip(values.tolist(), count.tolist()))
    w = [msg.get(int(p), 0) for p in parent]
    assert q.summarize() == sum(w)
    gw, gm, go = (x.cpu().numpy() for x in q.summary_groups(0))
    assert gw.tolist() == w == gm.tolist() and go.tolist() == (np.cumsum(w) - w).tolist()
    down = dict(zip(*(x.tolist() for x in np.unique(parent, return_counts=True))))
    cw, cm, _ = (x.cpu().numpy().tolist() for x in q.summary_groups(1))
    assert cw == [1] * n and cm == [down.get(v, 0) for v in np.sort(child).tolist()]
    ctx.close()


def test_a_sparse_tables_memory():
    """The table of a separator with four values per group takes no more than
    16 bytes per group (it is of segments alone)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    n = 1 << 21
    rng = np.random.default_rng(3)
    child = rng.integers(0, 8 * n, n)
    child[:2] = 0, 8 * n - 1
    ctx = gj.Context(0)
    q = _query(ctx, rng.choice(child, n), child)
    assert q.n_groups == [n, n]
    # the arrays of the summary (w, off, mult, live groups; segments, messages
    # and links) and the down messages' accumulators, per group
    arrays = n * (44 + 4) + n * (44 + 28) + 20 * n
    torch.cuda.synchronize()
    before, _ = torch.cuda.mem_get_info()
    assert q.summarize() > 0
    after, _ = torch.cuda.mem_get_info()
    # and 48 MB of slack: the pool grows by 32 MB at a time
    assert before - after <= arrays + 16 * 2 * n + (48 << 20)
    ctx.close()
