"""The radix sort behind factor builds above the small build's size (12288
rows), at the edges of its tiles of 4096 keys and past the 4096 tiles up to which
every pass has its own status words: keys-only words and (word, row id) pairs,
one pass to eight, against a stable sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(n, kind, bits):
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
        if kind != "equal":
            x[:2] = lo, lo + (1 << b) - 1      # the column's whole range
        cols.append(x.astype(np.int32))
    dev = [torch.from_numpy(c).cuda() for c in cols]
    ctx = gj.Context(0)
    rid = ctx.load_relation(dev, [0, 1])
    perm, gstart, gkey = ctx.factor_export(rid, n, 2)
    word = (dev[0].long() << 32) + (dev[1].long() + 2**31)     # in key order as signed words
    srt, order = torch.sort(word, stable=True)
    assert torch.equal(perm.long(), order)
    head = torch.ones(n, dtype=torch.bool, device="cuda")
    head[1:] = srt[1:] != srt[:-1]
    starts = head.nonzero().flatten()
    assert torch.equal(gstart[:-1].long(), starts) and int(gstart[-1]) == n
    for c in range(2):
        assert torch.equal(gkey[c], dev[c][order][starts])
    ctx.close()


@pytest.mark.parametrize("bits", [(3, 4), (10, 14), (20, 20), (32, 31), (32, 32)])
@pytest.mark.parametrize("kind", ["uniform", "skewed", "equal"])
@pytest.mark.parametrize("n", [12289, 16383, 16384, 16385, 20480, 20481])
def test_tile_edges(n, kind, bits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _check(n, kind, bits)


@pytest.mark.parametrize("bits", [(10, 14), (20, 20)])
@pytest.mark.parametrize("tiles", [4096, 4097])
def test_status_words_of_many_tiles(tiles, bits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _check(4096 * tiles - (4095 if tiles == 4097 else 0), "uniform", bits)
