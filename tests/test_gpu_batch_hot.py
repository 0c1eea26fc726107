"""Batch counting with frequent separator values a power of two apart: they have
shared-memory slots of their own, so they cost what neighbouring values do."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _batch(ctx, values, n):
    """R(0, 1), S(1, 2), T(2): S's and T's rows take `values` in turn (and once
    the two ends of a range of 2^17); the batch and its count."""
    from paper_2206_10435_gb300 import gj
    ends = np.array([0, (1 << 17) - 1])
    s = np.concatenate([ends, np.resize(values, n)]).astype(np.int32)
    t = np.concatenate([ends, np.resize(values, n // 2 + 1)]).astype(np.int32)
    r = np.concatenate([ends, np.resize(values, 1000)]).astype(np.int32)
    dev = lambda x: torch.from_numpy(x).cuda()
    ids = [ctx.load_relation([dev(np.zeros_like(r)), dev(r)], [0, 1]),
           ctx.load_relation([dev(s), dev(s[::-1].copy())], [1, 2]),
           ctx.load_relation([dev(t)], [2])]
    torch.cuda.synchronize()
    tcount = np.bincount(t, minlength=1 << 17)
    smsg = np.zeros(1 << 17, dtype=object)
    pairs, count = np.unique(np.stack([s, s[::-1]]), axis=1, return_counts=True)
    for (a, b), c in zip(pairs.T.tolist(), count.tolist()):
        smsg[a] += c * int(tcount[b])
    return gj.Batch(ctx, [ids]), sum(int(smsg[x]) for x in r.tolist())


def test_frequent_values_apart():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    n = 1 << 22
    ctx = gj.Context(0)
    us = {}
    for name, values in (("near", [5, 6]), ("apart", [5, 5 + 2048]), ("eight", 4096 * np.arange(8) + 3)):
        b, want = _batch(ctx, np.asarray(values), n)
        times = []
        for _ in range(8):
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            b.run(use_graph=False)
            end.record()
            end.synchronize()
            times.append(start.elapsed_time(end))
        assert int(b.totals[0]) == want and int(b.status[0]) == gj.GJ_OK
        us[name] = min(times)
        b.close()
    # a wide margin: values that share a slot took 15 and 7 times as long
    assert us["apart"] < 3 * us["near"] and us["eight"] < 3 * us["near"], us
    ctx.close()
