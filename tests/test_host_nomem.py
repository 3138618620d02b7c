"""Growth that runs out of memory (no GPU): the call fails with DRSF_ENOMEM and
the handle is what it was, or, where not even that can be had, says so."""
import numpy as np
import pytest

import paper_2607_20211_gb300 as drsf
from tests import fake_cuda

SMALL = 10
GROWTHS = {   # (form, edges) of a call that grows the handle, and of calls before it
    "buffers": ((drsf.DELETE, 30_000, "plain"), ()),
    "buffers and rebuild": ((drsf.INSERT, 30_000, "plain"), ()),
    "second rebuild": ((drsf.INSERT, 60_000, "plain"), ((drsf.INSERT, 9000, "plain"),)),
    "staging": ((drsf.DELETE, 100_000, "host"), ((drsf.DELETE, SMALL, "host"),)),
    "persistent, first": ((drsf.DELETE, SMALL, "batched"), ()),
    "persistent, more": ((drsf.INSERT, 20_000, "batched"), ((drsf.DELETE, SMALL, "batched"),)),
}


def _call(h, op, k, form):
    if form == "batched":
        return h.batched(op, k, graphs=2 if k <= SMALL else 300)
    return h.apply(op, k, host=form == "host")


def _fresh(lib, before):
    h = fake_cuda.Handle(lib)
    for c in before:
        assert _call(h, *c) == drsf.OK
    return h


@pytest.mark.parametrize("name", GROWTHS)
def test_growth_that_does_not_fit(name, tmp_path_factory):
    lib = fake_cuda.load(tmp_path_factory.getbasetemp())
    call, before = GROWTHS[name]
    h = _fresh(lib, before)
    start = lib.fake_held()
    assert _call(h, *call) == drsf.OK
    grown = lib.fake_held() - start
    h.close()
    assert grown > 0
    refused = went = 0
    for room in np.unique(np.geomspace(1, 3 * grown, 90).astype(np.int64)).tolist() + [0]:
        h = _fresh(lib, before)
        held = lib.fake_held()
        lib.fake_room(room)
        st = _call(h, *call)
        if st == drsf.OK:
            went += 1
            assert lib.fake_held() - held == grown
        else:
            assert st == drsf.ENOMEM and room < 3 * grown
            refused += 1
            assert lib.fake_held() >= held or call[2] == "batched"   # (the offsets' staging is not needed again)
            assert h.apply(call[0], SMALL) == drsf.OK
            lib.fake_room(-1)
            assert _call(h, *call) == drsf.OK
            assert lib.fake_held() - held == grown
        h.close()
    assert refused > 5 and went >= 1


def test_nothing_left_is_reported(tmp_path_factory):
    """An allocator that gives nothing any more, not even what was given back."""
    lib = fake_cuda.load(tmp_path_factory.getbasetemp())
    h = fake_cuda.Handle(lib)
    try:
        lib.fake_room(-1)
        lib.fake_deny(1)
        assert h.apply(drsf.DELETE, 30_000) == drsf.ENOMEM
        lib.fake_deny(0)
        for op, k in ((drsf.DELETE, SMALL), (drsf.INSERT, SMALL), (drsf.DELETE, 30_000)):
            assert h.apply(op, k) == drsf.EPOISONED
    finally:
        h.close()
    assert lib.fake_held() == 0
