"""The radix sort behind the factor build at the edges of its tiles (4096 keys):
keys-only words (row id under the key) and (word, row id) pairs, uniform,
skewed and equal digits, one pass to eight, against a stable sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [(3, 4), (10, 14), (20, 20), (32, 31), (32, 32)])
@pytest.mark.parametrize("kind", ["uniform", "skewed", "equal"])
@pytest.mark.parametrize("n", [2, 31, 4095, 4096, 4097, 8192, 50001])
def test_factor_equals_a_stable_sort(n, kind, bits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(n * 7 + sum(bits))
    cols = []
    for b in bits:
        lo = -(1 << (b - 1))
        x = rng.integers(lo, lo + (1 << b), n, dtype=np.int64)
        if kind == "skewed":
            x = np.where(rng.random(n) < 0.7, x[0], x)
        elif kind == "equal":
            x[:] = x[0]
        if kind != "equal" and n > 2:
            x[:2] = lo, lo + (1 << b) - 1      # the column's whole range
        cols.append(x.astype(np.int32))
    ctx = gj.Context(0)
    rid = ctx.load_relation([torch.from_numpy(c).cuda() for c in cols], [0, 1])
    perm, gstart, gkey = ctx.factor_export(rid, n, 2)
    order = np.lexsort((cols[1], cols[0]))
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), order)
    srt = np.stack([c[order] for c in cols], 1)
    starts = np.flatnonzero(np.concatenate([[True], (srt[1:] != srt[:-1]).any(1)]))
    assert np.array_equal(gstart.cpu().numpy()[:-1], starts) and int(gstart[-1]) == n
    assert np.array_equal(gkey.cpu().numpy().T, srt[starts])
    ctx.close()
