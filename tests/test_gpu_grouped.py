"""The batched call through the grid-wide launch sequence: slices checked on the
device, empty slices and graphs, against the oracle."""
import numpy as np
import pytest
import torch

import paper_2607_20211_gb300 as drsf
import workloads
from tests.gpu_util import check_batch, dev_tensor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    drsf.build()


def _union():
    graphs = workloads.batched_graphs(9, seed=51, n_lo=300, n_hi=3000)
    return graphs, workloads.Union(graphs)


@pytest.mark.parametrize("bad", [(0, "next"), (4, "next"), (4, "previous"), (8, "previous"), (3, "empty"), (8, "end")])
def test_an_edge_outside_its_graph_rejects_the_call(bad):
    """One edge of one slice leaves its graph (into the next or the previous
    one, or the slice belongs to an empty neighbour): nothing is applied, the
    error is reported once, and the next call works."""
    graphs, U = _union()
    vo = np.asarray(U.offsets, np.int64)
    f = drsf.DynamicForest(U.n, dev_tensor(workloads.keys_to_edges(U.keys)), dev_tensor(U.parent))
    try:
        slices = [U.shift(i, workloads.insert_batch(g.n, g.keys, 7 + i, i)) for i, g in enumerate(graphs)]
        good = [s.copy() for s in slices]
        k, how = bad
        lo, hi = int(vo[k]), int(vo[k + 1])
        if how == "empty":      # the slice's last edge counted to the next graph
            cnt = [len(s) for s in slices]
            cnt[k], cnt[k + 1] = cnt[k] - 1, cnt[k + 1] + 1
        else:
            cnt = [len(s) for s in slices]
            slices[k][-1, 1] = {"next": hi, "previous": lo - 1, "end": U.n}[how]
        bo = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
        before = f.parent().cpu().numpy()
        f.apply_batched(drsf.INSERT, dev_tensor(np.concatenate(slices)), vo, bo)
        with pytest.raises(drsf.DRSFError) as e:
            f.sync()
        assert e.value.status == drsf.EINVAL
        assert np.array_equal(f.parent().cpu().numpy(), before)
        assert f.num_edges() == len(U.keys)
        bo = np.concatenate([[0], np.cumsum([len(s) for s in good])]).astype(np.int64)
        b = np.concatenate(good)
        f.apply_batched(drsf.INSERT, dev_tensor(b), vo, bo)
        f.sync()
        keys = workloads.apply_keys(U.keys, b, 0)
        assert f.num_edges() == len(keys)
        check_batch(f, U.n, keys, f.parent().cpu().numpy(), drsf.DELETE, b[::2])
    finally:
        f.close()


def test_empty_slices_and_graphs():
    """Graphs without vertices and slices without edges, at both ends and in
    the middle; the result is the plain call's on the union."""
    graphs, U = _union()
    vo = np.asarray(U.offsets, np.int64)
    vo = np.concatenate([vo[:1], vo[:5], vo[4:5], vo[5:], vo[-1:]])     # empty first, after 4, last
    own = np.searchsorted(vo, np.arange(U.n), side="right") - 1
    b = np.concatenate([U.shift(i, workloads.insert_batch(g.n, g.keys, 40, i)) for i, g in enumerate(graphs)
                        if i not in (0, 5)])
    bo = np.searchsorted(own[b[:, 0]], np.arange(len(vo)), side="left").astype(np.int64)
    fs = [drsf.DynamicForest(U.n, dev_tensor(workloads.keys_to_edges(U.keys)), dev_tensor(U.parent)) for _ in range(2)]
    try:
        for op, x in ((drsf.INSERT, b), (drsf.DELETE, b), (drsf.INSERT, b[:0])):
            off = bo if len(x) else np.zeros_like(bo)
            fs[0].apply_batched(op, dev_tensor(x), vo, off)
            fs[1].apply(op, dev_tensor(x))
            assert torch.equal(fs[0].parent(), fs[1].parent())
        fs[0].sync()
    finally:
        for f in fs:
            f.close()
