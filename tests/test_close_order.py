"""The binding's handles on a fake library: a context's queries, batches and
servers are destroyed before it and once each, however they are closed or
collected."""
import ctypes
import gc

import pytest

from paper_2206_10435_gb300 import gj


class FakeLib:
    def __init__(self):
        self.next, self.open, self.log = 0x1000, {}, []

    def __getattr__(self, name):
        kind = name.split("_")[1]
        if name in ("gj_create", "gj_query_create", "gj_batch_create", "gj_server_create"):
            def make(*args):
                out = next(a for a in reversed(args) if hasattr(a, "_obj")) if kind != "create" else args[0]
                self.next += 16
                out._obj.value = self.next
                self.open[self.next] = "ctx" if kind == "create" else kind
                return gj.GJ_OK
            return make
        if name.endswith("destroy"):
            def destroy(h):
                what = self.open.pop(h.value)          # KeyError: destroyed twice
                if what != "ctx":
                    assert "ctx" in self.open.values()  # the handle points into it
                self.log.append(what)
            return destroy
        return lambda *args: gj.GJ_OK


@pytest.fixture()
def lib(monkeypatch):
    fake = FakeLib()
    monkeypatch.setattr(gj, "_lib", fake)
    monkeypatch.setattr("torch.zeros", lambda *a, **k: None)
    return fake


class Stream:
    cuda_stream = 0


def _open():
    ctx = gj.Context(0, Stream())
    return ctx, [ctx.query([1, 2]), gj.Batch(ctx, [[1, 2]]), gj.NativeServer(ctx)]


def test_closed_by_the_context(lib):
    ctx, objs = _open()
    ctx.close()
    assert sorted(lib.log[:3]) == ["batch", "query", "server"] and lib.log[3:] == ["ctx"]
    assert all(o.h is None for o in objs)
    for o in objs + [ctx]:
        o.close()
    assert len(lib.log) == 4


@pytest.mark.parametrize("n", range(3))
def test_collected_in_one_cycle(lib, n):
    ctx, objs = _open()
    objs[n].close()
    cycle = [ctx, objs]
    cycle.append(cycle)
    del ctx, objs, cycle
    gc.collect()
    assert sorted(lib.log[:3]) == ["batch", "query", "server"] and lib.log[3:] == ["ctx"]


def test_dropped_one_by_one(lib):
    ctx, objs = _open()
    for kind in ("query", "batch", "server"):
        objs.pop(0)
        gc.collect()
        assert lib.log[-1] == kind
    ctx.close()
    assert lib.log[-1] == "ctx" and len(lib.log) == 4
