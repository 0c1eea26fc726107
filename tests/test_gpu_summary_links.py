"""Links to a child through its table of separator values and through the
search that wider ranges keep: value ranges around the rule's line, parent keys
below, inside and above the child's, several children, and messages past
2^64, with every group's weight, multiplicity and offset against numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _message(keys, weight):
    """{value: sum of the rows' weights} as Python integers."""
    out = {}
    for k, w in zip(keys.tolist(), weight):
        out[k] = out.get(k, 0) + w
    return out


@pytest.mark.parametrize("children", [1, 2, 3, 5])
@pytest.mark.parametrize("over", [-1, 0, 1, 10**6])
def test_groups_of_a_star(children, over):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(children * 7 + (over & 0xff))
    ctx = gj.Context(0)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.int32)).cuda()
    n = 3000
    child, cols = [], []
    for c in range(children):
        # distinct child keys; the parent's groups are its distinct rows
        m = 200 + c
        keys = rng.choice(5000, m, replace=False).astype(np.int64) - 2500
        child.append(keys)
        pk = rng.choice(np.concatenate([keys, [-2**31, 2**31 - 1, keys.min() - 1, keys.max() + 1]]), n)
        cols.append(pk)
    order = np.lexsort(tuple(reversed(cols)))
    srt = np.stack(cols, 1)[order]
    head = np.concatenate([[True], (srt[1:] != srt[:-1]).any(1)])
    groups = srt[head]
    count = np.diff(np.append(np.flatnonzero(head), n))
    G = len(groups)
    # the first child's range is moved to the line of the rule
    line = 4 * (len(child[0]) + G) + 4096
    lo = child[0].min()
    child[0][child[0] == child[0].max()] = lo + line - 1 + over
    ids = [ctx.load_relation([dev(x) for x in cols], list(range(children)))]
    copies = [rng.integers(1, 4, len(k)) for k in child]
    for c, k in enumerate(child):
        rows = np.repeat(k, copies[c])
        ids.append(ctx.load_relation([dev(rows)], [c]))
    q = ctx.query(ids)
    total = q.summarize()
    msg = [_message(k, m.tolist()) for k, m in zip(child, copies)]
    w = [int(c) * int(np.prod([msg[j].get(int(g[j]), 0) for j in range(children)], dtype=object))
         for g, c in zip(groups, count)]
    gw, gm, go = (x.cpu().numpy() for x in q.summary_groups(0))
    assert total == sum(w) and gw.tolist() == w and gm.tolist() == w
    assert go.tolist() == np.concatenate([[0], np.cumsum(w)[:-1]]).tolist()
    for j in range(children):
        down = {}
        for g, c, x in zip(groups, count, w):
            m = msg[j].get(int(g[j]), 0)
            if m:
                down[int(g[j])] = down.get(int(g[j]), 0) + x // m
        ks = np.argsort(child[j], kind="stable")
        want = [int(copies[j][i]) * down.get(int(child[j][i]), 0) for i in ks]
        cw, cm, co = (x.cpu().numpy().tolist() for x in q.summary_groups(j + 1))
        assert cw == copies[j][ks].tolist() and cm == want and co == [0] * len(ks)
    ctx.close()
