"""Runs of equal leading columns around the length from which the row's place is
counted in three parts (64 rows) and around its words of 32 rows, at every
offset in a word, with many equal rows, against a stable sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", [1, 3, 200])
@pytest.mark.parametrize("length", [63, 64, 65, 95, 96, 97, 128, 160, 255])
def test_run_lengths(length, values):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(length * values)
    n = 20011                            # above the small build's size
    runs = []
    while sum(runs) < n:                 # the runs start at every offset
        runs += [length, int(rng.integers(1, 34))]
    lead = np.repeat(rng.choice(2**31 - 1, len(runs), replace=False), runs)[:n].astype(np.int32)
    # every value of the trailing columns' whole words, both ends among them
    some = np.concatenate([[-2**31, 2**31 - 1], rng.integers(-2**31, 2**31, 200)])[:max(values, 2)]
    b, c = (rng.choice(some, n).astype(np.int32) for _ in range(2))
    if values == 1:
        b[2:] = c[2:] = 2**31 - 1        # runs of one key, all bits set
    mix = rng.permutation(n)
    cols = [x[mix] for x in (lead, b, c)]
    ctx = gj.Context(0)
    rid = ctx.load_relation([torch.from_numpy(x).cuda() for x in cols], [0, 1, 2])
    perm, gstart, gkey = ctx.factor_export(rid, n, 3)
    order = np.lexsort((cols[2], cols[1], cols[0]))
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), order)
    srt = np.stack([x[order] for x in cols], axis=1)
    starts = np.flatnonzero(np.concatenate([[True], (srt[1:] != srt[:-1]).any(axis=1)]))
    assert np.array_equal(gstart.cpu().numpy()[:-1], starts) and int(gstart[-1]) == n
    assert np.array_equal(gkey.cpu().numpy().T, srt[starts])
    ctx.close()
