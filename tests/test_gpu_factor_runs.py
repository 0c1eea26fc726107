"""Factor builds of keys wider than one word: rows sorted by the leading
columns, then every run of equal leading columns ordered and cut into groups
by one kernel.  Runs at the kernel's limits (256 rows, tiles of 1280) against
a stable sort, with payloads of every layout; longer runs take another path
and give the same result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lengths(case, n, rng):
    if case == "ones":
        return [1] * n
    if case == "short":
        out = rng.integers(1, 40, n)
    elif case == "limit":
        out = rng.choice([1, 2, 255, 256], n)
    elif case == "long":              # one run over the limit
        out = np.concatenate([rng.integers(1, 100, 20), [257], rng.integers(1, 100, n)])
    else:                             # "straddle": runs of 256 across the tiles' ends
        out = np.tile([1280 - 200, 256, 56], n)
        out = np.concatenate([[x] if x <= 256 else [100] * (x // 100) + ([x % 100] if x % 100 else []) for x in out])
    cut = int(np.searchsorted(np.cumsum(out), n))
    out = list(out[:cut])
    return out + [n - sum(out)]


@pytest.mark.parametrize("payloads", [(), (np.int32,), (np.int64,), (np.int64, np.int32)])
@pytest.mark.parametrize("case", ["ones", "short", "limit", "straddle", "long"])
@pytest.mark.parametrize("n", [1279, 1280, 1281, 1536, 1537, 30011])
def test_runs_equal_a_stable_sort(case, n, payloads):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(n + 7 * len(payloads))
    runs = _lengths(case, n, rng)
    lead = np.repeat(rng.choice(2**31 - 1, len(runs), replace=False).astype(np.int32), runs)
    # two trailing columns of 32 bits; few values, so that full keys repeat
    b = rng.choice(np.array([-2**31, -5, 0, 7, 2**31 - 1], np.int64), n).astype(np.int32)
    c = rng.choice(np.array([-2**31, 1, 2**31 - 1], np.int64), n).astype(np.int32)
    mix = rng.permutation(n)
    cols = [x[mix] for x in (lead, b, c)]
    pays = [rng.integers(np.iinfo(t).min, np.iinfo(t).max, n, dtype=t) for t in payloads]
    ctx = gj.Context(0)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    rid = ctx.load_relation([dev(x) for x in cols], [0, 1, 2], [dev(p) for p in pays])
    perm, gstart, gkey = ctx.factor_export(rid, n, 3)
    order = np.lexsort((cols[2], cols[1], cols[0]))
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), order)
    srt = np.stack([x[order] for x in cols], axis=1)
    starts = np.flatnonzero(np.concatenate([[True], (srt[1:] != srt[:-1]).any(axis=1)]))
    assert np.array_equal(gstart.cpu().numpy()[:-1], starts) and int(gstart[-1]) == n
    assert np.array_equal(gkey.cpu().numpy().T, srt[starts])
    q = ctx.query([rid])
    got = q.desummarize(0, q.summarize())
    for a, w in zip(got, [srt[:, 0], srt[:, 1], srt[:, 2]] + [p[order] for p in pays]):
        assert np.array_equal(a.cpu().numpy(), w)
    ctx.close()
