"""Batches that the caller records into a graph of its own, replayed until the
storage is full, after it moved, and between other calls, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_20211_gb300 as drsf
import workloads
from tests.gpu_util import check_batch, dev_tensor, make_forest

pytestmark = pytest.mark.gpu
I, D = drsf.INSERT, drsf.DELETE
PERSISTENT = ((2 ** 31 - 1, 256, 0, 1),)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    drsf.build()


def _apply(f, form, op, buf, vo=None, bo=None):
    if form == "plain":
        f.apply(op, buf)
    elif form == "grouped":
        f.apply_batched(op, buf, vo, bo)
    else:
        f.apply_batched(op, buf, vo, bo, PERSISTENT)


def _record(f, form, op, buf, vo=None, bo=None):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _apply(f, form, op, buf, vo, bo)
    return g


@pytest.mark.parametrize("form", ["plain", "grouped", "persistent"])
def test_replays_until_the_index_is_full(form):
    """A handle of 100 edges (16,384 index slots, of which an insert may use
    11,468): the third replay of 4,000 fresh edges is skipped and reported,
    a plain call makes room, and the recording, whose storage is gone, is
    skipped and reported from then on."""
    n, b = 5000, 4000
    g = workloads.er_graph(n, 100, seed=3)
    f = make_forest(g)
    keys, par = g.keys, g.parent
    vo, bo = np.array([0, n], np.int64), np.array([0, b], np.int64)
    buf = torch.zeros((b, 2), dtype=torch.int32, device="cuda")   # self-loops: nothing to apply
    try:
        _apply(f, form, I, buf, vo, bo)                           # (buffers)
        graph = _record(f, form, I, buf, vo, bo)
        batches = [workloads.insert_batch(n, g.keys, b, 60 + c) for c in range(4)]
        for c in range(2):
            buf.copy_(dev_tensor(batches[c]))
            graph.replay()
            ref = oracle.apply(n, keys, par, I, batches[c], want_keys=True)
            keys, par = ref.keys, ref.parent
            assert np.array_equal(f.parent().cpu().numpy(), par)
        f.sync()
        buf.copy_(dev_tensor(batches[2]))
        graph.replay()
        graph.replay()
        with pytest.raises(drsf.DRSFError) as e:
            f.sync()
        assert e.value.status == drsf.ENOMEM
        assert f.num_edges() == len(keys)
        assert np.array_equal(f.parent().cpu().numpy(), par)
        assert np.array_equal(workloads.edges_to_keys(f.export_edges().cpu().numpy()), keys)
        keys, par, st = check_batch(f, n, keys, par, I, batches[2])
        assert st["rebuilds"] == 1
        buf.copy_(dev_tensor(batches[3]))
        graph.replay()
        with pytest.raises(drsf.DRSFError) as e:
            f.stats()
        assert e.value.status == drsf.EINVAL
        assert np.array_equal(f.parent().cpu().numpy(), par)
        keys, par, _ = check_batch(f, n, keys, par, D, batches[0][::2])
        _apply(f, form, D, buf[:0], vo, bo * 0)
        graph = _record(f, form, I, buf, vo, bo)
        graph.replay()
        ref = oracle.apply(n, keys, par, I, batches[3], want_keys=True)
        keys, par = ref.keys, ref.parent
        assert np.array_equal(f.parent().cpu().numpy(), par)
        check_batch(f, n, keys, par, D, batches[1])
    finally:
        f.close()


def test_replays_until_the_overflow_list_is_full():
    """65,536 entries: stars whose centres' rows are full, inserted and deleted
    by two recordings."""
    n, b = 40_000, 15_000
    g = workloads.er_graph(n, 60_000, seed=4)
    f = make_forest(g)
    keys, par = g.keys, g.parent
    buf = torch.zeros((b, 2), dtype=torch.int32, device="cuda")
    try:
        graphs = {}
        for op in (I, D):
            f.apply(op, buf)
            graphs[op] = _record(f, "plain", op, buf)
        done = 0
        for c in range(6):
            v = np.arange(200 + c, 200 + c + 2 * b, 2) % n
            e = np.stack([np.full(b, c), np.where(v < 200, v + 300, v)], 1).astype(np.int32)
            buf.copy_(dev_tensor(e))
            graphs[I].replay()
            try:
                f.sync()
            except drsf.DRSFError as err:
                assert err.status == drsf.ENOMEM
                assert np.array_equal(f.parent().cpu().numpy(), par)
                break
            ref = oracle.apply(n, keys, par, I, e, want_keys=True)
            keys, par = ref.keys, ref.parent
            assert np.array_equal(f.parent().cpu().numpy(), par)
            done += 1
        assert 2 <= done < 6
        keys, par, st = check_batch(f, n, keys, par, I, e)     # a plain call makes room
        assert st["rebuilds"] == 1
        check_batch(f, n, keys, par, D, e[::3])
    finally:
        f.close()


@pytest.mark.parametrize("form", ["plain", "grouped"])
def test_a_refused_recording_leaves_the_capture_alone(form):
    """A batch too long for the handle's buffers and one that fits, in one
    capture: the first is refused, the second is in the graph."""
    n, b = 3000, 5000
    g = workloads.er_graph(n, 6000, seed=5)
    f = make_forest(g)
    vo = np.array([0, n], np.int64)
    buf = dev_tensor(workloads.insert_batch(n, g.keys, b, 9))
    try:
        _apply(f, form, I, buf[:100], vo, np.array([0, 100], np.int64))
        f.delete(buf[:100])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            with pytest.raises(drsf.DRSFError) as e:
                _apply(f, form, I, buf, vo, np.array([0, b], np.int64))
            assert e.value.status == drsf.ECUDA
            _apply(f, form, I, buf[:100], vo, np.array([0, 100], np.int64))
        par = f.parent().cpu().numpy()
        graph.replay()
        ref = oracle.apply(n, g.keys, par, I, buf[:100].cpu().numpy(), want_keys=True)
        assert np.array_equal(f.parent().cpu().numpy(), ref.parent)
        f.reserve(b)                                        # longer buffers: the recording is void
        graph.replay()
        with pytest.raises(drsf.DRSFError) as e:
            f.sync()
        assert e.value.status == drsf.EINVAL
        check_batch(f, n, ref.keys, ref.parent, D, buf[:100].cpu().numpy())
    finally:
        f.close()


@pytest.mark.parametrize("form", ["grouped", "persistent"])
def test_offsets_and_host_batches_of_a_recording_are_its_own(form):
    """Two graphs recorded with their own offsets, calls with other offsets
    between the replays; a host batch recorded and its memory reused."""
    graphs = workloads.batched_graphs(5, seed=52, n_lo=300, n_hi=2000)
    U = workloads.Union(graphs)
    vo = np.asarray(U.offsets, np.int64)
    f = drsf.DynamicForest(U.n, dev_tensor(workloads.keys_to_edges(U.keys)), dev_tensor(U.parent))
    keys, par = U.keys, U.parent

    def step(op, e):
        nonlocal keys, par
        ref = oracle.apply(U.n, keys, par, op, e, want_keys=True)
        keys, par = ref.keys, ref.parent
        assert np.array_equal(f.parent().cpu().numpy(), par)

    def batch(sizes, seed):
        per = [U.shift(i, workloads.insert_batch(g.n, g.keys, k, seed + i)) for i, (g, k) in enumerate(zip(graphs, sizes))]
        return np.concatenate(per), np.concatenate([[0], np.cumsum([len(p) for p in per])]).astype(np.int64)

    try:
        e1, b1 = batch([5, 40, 1, 9, 30], 1)
        e2, b2 = batch([50, 4, 21, 1, 3], 100)
        host = np.ascontiguousarray(e2[::-1])
        _apply(f, form, I, dev_tensor(e1), vo, b1)
        step(I, e1)
        dev = dev_tensor(e1)
        g_del = _record(f, form, D, dev, vo, b1)
        g_ins = _record(f, form, I, dev, vo, b1)
        g_host = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g_host):
            f.apply_host(I, host)
        host[:] = 0
        for _ in range(2):
            g_del.replay()
            step(D, e1)
            _apply(f, form, I, dev_tensor(e2), vo, b2)
            step(I, e2)
            g_ins.replay()
            step(I, e1)
            f.apply_host(D, e2)
            step(D, e2)
            g_host.replay()
            step(I, e2)
            _apply(f, form, D, dev_tensor(e2), vo, b2)
            step(D, e2)
        f.sync()
    finally:
        f.close()


def test_static_forest_recorded_before_a_rebuild():
    n = 4000
    g = workloads.er_graph(n, 6000, seed=6)
    f = make_forest(g)
    try:
        f.static_forest()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = f.static_forest()
        graph.replay()
        forest = (out[0] if isinstance(out, (tuple, list)) else out).cpu().numpy()
        assert oracle.check_forest(n, g.keys, forest) == 0
        f.reserve(100_000)
        graph.replay()
        with pytest.raises(drsf.DRSFError) as e:
            f.sync()
        assert e.value.status == drsf.EINVAL
    finally:
        f.close()
