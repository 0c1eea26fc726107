"""The upward scan at the edges of its two tiles (1024 and 2048 groups; a leaf of
2^20 groups and more takes the larger): every group's weight, multiplicity and
offset of a two-relation join against numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 1023, 1024, 1025, 2049, (1 << 20) - 1, 1 << 20, (1 << 20) + 2047])
@pytest.mark.parametrize("root", [1, 1024, 3001])
def test_groups(leaf, root):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(leaf + root)
    # leaf groups (b, c), all distinct, in segments of uneven size; some values
    # of b without groups, some root groups without a segment
    b = np.sort(rng.integers(0, max(2, leaf // 3), leaf))
    c = np.arange(leaf)
    a, rb = np.arange(root), rng.integers(0, max(2, leaf // 3) + 5, root)
    ctx = gj.Context(0)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).cuda()
    q = ctx.query([ctx.load_relation([dev(a), dev(rb)], [0, 1]), ctx.load_relation([dev(b), dev(c)], [1, 2])])
    total = q.summarize()
    seg = np.bincount(b, minlength=rb.max() + 1)
    w = seg[rb]
    assert total == w.sum()
    gw, gm, go = (x.cpu().numpy() for x in q.summary_groups(0))
    assert np.array_equal(gw, w) and np.array_equal(gm, w) and np.array_equal(go, np.cumsum(w) - w)
    down = np.bincount(rb, minlength=len(seg))
    lw, lm, lo = (x.cpu().numpy() for x in q.summary_groups(1))
    first = np.cumsum(seg) - seg
    assert np.array_equal(lw, np.ones(leaf)) and np.array_equal(lm, down[b]) and np.array_equal(lo, c - first[b])
    ctx.close()
