"""Batches recorded into a caller's graph, host side (no GPU): what a capture
forbids is not done, and what has no room is refused before it is recorded."""
import pytest

import paper_2607_20211_gb300 as drsf
from tests import fake_cuda

INDEX_MAX = int(0.7 * 8192)   # of a handle built without edges: 2 * 4,096 slots


@pytest.fixture()
def handle(tmp_path_factory):
    h = fake_cuda.Handle(fake_cuda.load(tmp_path_factory.getbasetemp()))
    yield h
    h.close()


def _record(h, call):
    """(status, launches recorded, forbidden calls, recorded copies) of `call` under capture."""
    lib = h.lib
    f0, c0 = lib.fake_forbidden(), lib.fake_recorded_copies()
    lib.fake_launches(b"")
    lib.fake_capture(h.STREAM)
    st = call()
    lib.fake_capture(None)
    return st, lib.fake_launches(b"k_"), lib.fake_forbidden() - f0, lib.fake_recorded_copies() - c0


FORMS = {"plain": lambda h, op, k: h.apply(op, k), "host": lambda h, op, k: h.apply(op, k, host=True),
         "grouped": lambda h, op, k: h.grouped(op, k), "persistent": lambda h, op, k: h.batched(op, k)}


@pytest.mark.parametrize("form", FORMS)
def test_recording_does_nothing_that_a_capture_forbids(handle, form):
    call = FORMS[form]
    for op in (drsf.INSERT, drsf.DELETE):
        assert call(handle, op, 100) == drsf.OK
    for op in (drsf.INSERT, drsf.DELETE):
        st, launches, forbidden, copies = _record(handle, lambda: call(handle, op, 100))
        assert (st, forbidden, copies) == (drsf.OK, 0, 0) and launches > 3
    # plain calls go on as before, and the room is read, not guessed
    assert call(handle, drsf.DELETE, 100) == drsf.OK
    w = handle.lib.fake_waits()
    assert call(handle, drsf.INSERT, 100) == drsf.OK and handle.lib.fake_waits() > w


@pytest.mark.parametrize("form", FORMS)
def test_no_room_refuses_the_recording(handle, form):
    call = FORMS[form]
    assert call(handle, drsf.INSERT, 10) == drsf.OK      # (the persistent kernels' buffers)
    for op in (drsf.INSERT, drsf.DELETE):                # longer than any batch before it
        st, launches, forbidden, copies = _record(handle, lambda: call(handle, op, 4097))
        assert (st, launches, forbidden, copies) == (drsf.ECUDA, 0, 0, 0)
    assert handle.apply(drsf.INSERT, 4000) == drsf.OK
    room = INDEX_MAX - 4010
    st, launches, forbidden, copies = _record(handle, lambda: call(handle, drsf.INSERT, room + 1))
    assert (st, launches, forbidden, copies) == (drsf.ECUDA, 0, 0, 0)
    for op, k in ((drsf.INSERT, room), (drsf.DELETE, 4000)):
        st, launches, forbidden, copies = _record(handle, lambda: call(handle, op, k))
        assert (st, forbidden, copies) == (drsf.OK, 0, 0) and launches > 3


def test_persistent_buffers_are_not_allocated_while_recording(handle):
    st, launches, forbidden, _ = _record(handle, lambda: handle.batched(drsf.INSERT, 10))
    assert (st, launches, forbidden) == (drsf.ECUDA, 0, 0)
    assert handle.batched(drsf.INSERT, 10) == drsf.OK
    st, launches, forbidden, _ = _record(handle, lambda: handle.batched(drsf.INSERT, 10, graphs=257))
    assert (st, launches, forbidden) == (drsf.ECUDA, 0, 0)
