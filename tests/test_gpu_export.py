"""Exported arrays (factors, group summaries) at any word-aligned device address,
in pinned host memory and left out one by one: the same words, and nothing
written past them."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["device", "pinned"])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 3, 1000, 40001])
def test_exports(n, shift, where):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(n)
    ctx = gj.Context(0)
    cols = [torch.from_numpy(rng.integers(0, 50, n, dtype=np.int32)).cuda() for _ in range(2)]
    rid = ctx.load_relation(cols, [0, 1])
    q = ctx.query([rid])
    q.summarize()
    want = [t.cpu() for t in ctx.factor_export(rid, n, 2)] + [t.cpu() for t in q.summary_groups(0)]
    G = int(want[1].numel()) - 1

    def room(ref):
        words = ref.numel() * ref.element_size() // 4 + 8
        buf = torch.full((words,), -7, dtype=torch.int32)
        return buf.pin_memory() if where == "pinned" else buf.cuda()

    bufs = [room(t) for t in want]
    # 64-bit arrays keep their own alignment
    ptr = [b.data_ptr() + 4 * (shift if t.element_size() == 4 else shift // 2 * 2) for b, t in zip(bufs, want)]
    P = ctypes.c_void_p
    g = ctypes.c_int64()
    L = gj.lib()
    for left_out in range(4):
        for b in bufs:
            b.fill_(-7)
        torch.cuda.synchronize()
        p = [None if left_out == i % 3 + 1 else P(x) for i, x in enumerate(ptr)]
        assert L.gj_factor_export(ctx.h, rid, None, ctypes.byref(g), *p[:3]) == gj.GJ_OK and g.value == G
        assert L.gj_summary_groups(q.h, 0, *p[3:]) == gj.GJ_OK
        torch.cuda.synchronize()
        for i, (b, t, at) in enumerate(zip(bufs, want, ptr)):
            off = (at - b.data_ptr()) // 4
            ref = t.reshape(-1).view(torch.int32)
            got = b.cpu()
            if left_out == i % 3 + 1:
                assert bool((got == -7).all())
                continue
            assert torch.equal(got[off:off + ref.numel()], ref)
            assert bool((got[:off] == -7).all()) and bool((got[off + ref.numel():] == -7).all())
    ctx.close()
