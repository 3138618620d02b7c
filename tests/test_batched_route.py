"""Which kernels the batched call runs (CPU): the grid-wide sequence without a
schedule, the persistent per-graph kernels with any, whatever object it is."""
import numpy as np
import pytest
import torch

import paper_2607_20211_gb300 as drsf
from tests import fake_cuda

D = drsf.DEFAULT_CLASSES


class _Recorder:
    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        return lambda *a: self.calls.append((name, a)) or drsf.OK


@pytest.mark.parametrize("args,route", [
    ((), "drsf_apply_grouped"), ((None,), "drsf_apply_grouped"),
    ((D,), "drsf_apply_batched"), ((tuple(list(D)),), "drsf_apply_batched"), ((list(map(list, D)),), "drsf_apply_batched"),
    ((((2 ** 31 - 1, 256, 0),),), "drsf_apply_batched")])
def test_a_schedule_runs_the_persistent_kernels(args, route, monkeypatch):
    lib = _Recorder()
    monkeypatch.setattr(drsf, "_lib", lib)
    monkeypatch.setattr(drsf, "_dev_i32", lambda t, *_: t)
    monkeypatch.setattr(drsf, "_stream_ptr", lambda s: 0)
    f = drsf.DynamicForest.__new__(drsf.DynamicForest)
    f._h, f._stream = 1, None
    f.apply_batched(drsf.INSERT, torch.tensor([[0, 1], [5, 6]], dtype=torch.int32), [0, 5, 9], [0, 1, 2], *args)
    f._h = None
    assert [c[0] for c in lib.calls] == [route]


def test_kernels_of_the_two_calls(tmp_path_factory):
    lib = fake_cuda.load(tmp_path_factory.getbasetemp())
    h = fake_cuda.Handle(lib)
    try:
        h.apply(drsf.INSERT, 10)
        for op in (drsf.INSERT, drsf.DELETE):
            lib.fake_launches(b"")
            assert h.grouped(op, 50) == drsf.OK
            assert lib.fake_launches(b"k_begin") == 1
            assert h.batched(op, 50) == drsf.OK
            assert lib.fake_launches(b"k_bpersist") == 1
    finally:
        h.close()
