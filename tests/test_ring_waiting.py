"""Rings that wait for the end of a capture to be destroyed: whoever destroys
them may meet another thread at the same list, keeps their storage until the
context is gone, and does not answer for their errors."""
import weakref

import torch

from paper_2609_24456_gb300 import edp


class _Storage:
    pass


class _Lib:
    def __init__(self, status=0, seen=None):
        self.status, self.seen = status, seen

    def edp_destroy(self, ctx):
        if self.seen is not None:
            self.seen.append(ctx)
        return self.status

    def edp_last_error(self, ctx):
        return b""


def _use(monkeypatch, lib, capturing):
    monkeypatch.setattr(edp, "lib", lambda: lib)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", capturing)
    monkeypatch.setattr(edp.Ring, "_waiting", [])


def test_another_thread_takes_the_last(monkeypatch):
    seen = []

    def capturing():  # between the look at the list and the pop
        edp.Ring._waiting.clear()
        return False

    _use(monkeypatch, _Lib(seen=seen), capturing)
    edp.Ring._waiting.append({"ctx": 5})
    edp.Ring._destroy_waiting()
    assert not seen


def test_storage_outlives_the_context(monkeypatch):
    store = _Storage()
    alive = weakref.ref(store)
    seen = []

    class Lib(_Lib):
        def edp_destroy(self, ctx):
            seen.append((ctx, alive() is not None))
            return 0

    _use(monkeypatch, Lib(), lambda: False)
    edp.Ring._waiting.append({"ctx": 5, "obs": store})
    del store
    edp.Ring._destroy_waiting()
    assert seen == [(5, True)]
    assert alive() is None and not edp.Ring._waiting


def test_an_error_does_not_reach_another_ring(monkeypatch):
    seen = []
    _use(monkeypatch, _Lib(status=edp.EDP_ERR_CUDA, seen=seen), lambda: False)
    edp.Ring._waiting.extend([{"ctx": 5}, {"ctx": 6}])
    edp.Ring._destroy_waiting()
    assert sorted(seen) == [5, 6]


def test_nothing_is_destroyed_during_a_capture(monkeypatch):
    seen = []
    _use(monkeypatch, _Lib(seen=seen), lambda: True)
    edp.Ring._waiting.append({"ctx": 5})
    edp.Ring._destroy_waiting()
    assert not seen and len(edp.Ring._waiting) == 1
