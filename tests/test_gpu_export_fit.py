"""Exports into device allocations that end where the array ends: copied by the
one kernel; into pinned memory: by the runtime.  (A destination that ends before
the array does is left to the runtime's own check and is not tried here.)"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 1000, 70001])
def test_exact_fit(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_10435_gb300 import gj
    rng = np.random.default_rng(n)
    ctx = gj.Context(0)
    col = torch.from_numpy(rng.integers(0, 90, n, dtype=np.int32)).cuda()
    rid = ctx.load_relation([col], [0])
    perm, gstart, gkey = ctx.factor_export(rid, n, 1)
    L, g = gj.lib(), ctypes.c_int64()
    refs = [perm, gstart, gkey.reshape(-1)]
    cudart = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    ptrs = []
    for r in refs:
        p = ctypes.c_void_p()
        assert cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(4 * r.numel())) == 0
        ptrs.append(p)
    pinned = [torch.zeros(r.numel(), dtype=torch.int32).pin_memory() for r in refs]
    ctx.profile()
    assert L.gj_factor_export(ctx.h, rid, None, ctypes.byref(g), *ptrs) == gj.GJ_OK
    assert ctx.profile()["launches"] == 1
    assert L.gj_factor_export(ctx.h, rid, None, ctypes.byref(g),
                              *[ctypes.c_void_p(p.data_ptr()) for p in pinned]) == gj.GJ_OK
    assert ctx.profile()["launches"] == 0
    for r, p, h in zip(refs, ptrs, pinned):
        got = torch.empty(r.numel(), dtype=torch.int32)
        assert cudart.cudaMemcpy(ctypes.c_void_p(got.data_ptr()), p, ctypes.c_size_t(4 * r.numel()), 2) == 0
        assert torch.equal(got, r.cpu()) and torch.equal(h, r.cpu())
        assert cudart.cudaFree(p) == 0
    ctx.close()
