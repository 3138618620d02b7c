"""What drsf_reserve promises, on the host side (no GPU): the calls after it
allocate nothing."""
import pytest

import paper_2607_20211_gb300 as drsf
from tests import fake_cuda


@pytest.fixture()
def handle(tmp_path_factory):
    h = fake_cuda.Handle(fake_cuda.load(tmp_path_factory.getbasetemp()))
    yield h
    h.close()


@pytest.mark.parametrize("size", [1, 5000, 100_000])
def test_calls_after_reserve_allocate_nothing(handle, size):
    lib = handle.lib
    assert lib.drsf_reserve(handle.h, size, handle.STREAM) == drsf.OK
    before = lib.fake_pinned(), lib.fake_held()
    assert lib.drsf_sync(handle.h, handle.STREAM) == drsf.OK
    for k in range(3):
        for op in (drsf.INSERT, drsf.DELETE):
            assert handle.apply(op, min(size, 1000), host=True) == drsf.OK
            assert handle.apply(op, min(size, 1000)) == drsf.OK
            assert lib.drsf_sync(handle.h, handle.STREAM) == drsf.OK
    assert (lib.fake_pinned(), lib.fake_held()) == before


def test_batches_allocate_no_host_memory(handle):
    """Batches that have to read the counters (and rebuild) without drsf_reserve."""
    lib = handle.lib
    p, w = lib.fake_pinned(), lib.fake_waits()
    for k in range(6):
        for op in (drsf.DELETE, drsf.INSERT):
            assert handle.apply(op, 4000) == drsf.OK
    assert lib.fake_waits() > w and lib.fake_pinned() == p
    assert lib.drsf_sync(handle.h, handle.STREAM) == drsf.OK and lib.fake_pinned() == p + 1
