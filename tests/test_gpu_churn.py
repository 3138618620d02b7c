"""Edges that leave and come back: storage given up by a delete is taken again
by later inserts, with every batch equal to the oracle's."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_20211_gb300 as drsf
import workloads
from tests.gpu_util import check_batch, make_forest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    drsf.build()


@pytest.mark.parametrize("n,m,b,cycles", [(40, 60, 30, 40), (3000, 9000, 500, 40), (20_000, 60_000, 6000, 12)])
def test_same_edges_leave_and_come_back(n, m, b, cycles):
    """One batch deleted and inserted again for many cycles, its pairs twice
    in each batch (equal keys race for one index slot), together with fresh
    pairs that take deleted slots of other keys."""
    g = workloads.er_graph(n, m, seed=21)
    f = make_forest(g)
    keys, par = g.keys, g.parent
    rng = np.random.default_rng(5)
    back = workloads.keys_to_edges(rng.permutation(g.keys)[:b])
    old = np.zeros((0, 2), np.int32)
    try:
        for c in range(cycles):
            fresh = workloads.insert_batch(n, keys, b // 4, 100 + c)
            keys, par, _ = check_batch(f, n, keys, par, drsf.DELETE, np.concatenate([back, back[:, ::-1], old]),
                                       labels=c == 0)
            keys, par, _ = check_batch(f, n, keys, par, drsf.INSERT, rng.permutation(
                np.concatenate([back, back[:, ::-1], fresh])), labels=False)
            old = fresh
    finally:
        f.close()


@pytest.mark.parametrize("batched", [False, (), (((2 ** 31 - 1, 512, 0, 2),),), (drsf.DEFAULT_CLASSES,)],
                         ids=["plain", "grouped", "persistent", "persistent-classes"])
def test_window_neither_overflows_nor_rebuilds(batched):
    """A window of returning edges reuses the rows' freed slots: with
    append-only rows 24 cycles of a sixth of the edges would overflow every
    row's slack (a quarter of its degree, at least 4) many times over.  The
    last cycles run against the oracle."""
    g = workloads.er_graph(30_000, 120_000, seed=22)
    f = make_forest(g)
    keys, par = g.keys, g.parent
    rng = np.random.default_rng(6)
    back = workloads.keys_to_edges(rng.permutation(g.keys)[:20_000])
    dev = torch.from_numpy(back).cuda()
    vo = bo = None
    if batched is not False:
        vo, bo = np.array([0, g.n], np.int64), np.array([0, len(back)], np.int64)
    try:
        for c in range(24):
            for op in (drsf.DELETE, drsf.INSERT):
                if batched is not False:
                    f.apply_batched(op, dev, vo, bo, *batched)
                else:
                    f.apply(op, dev)
        st = f.stats()
        assert st["rebuilds"] == 0 and st["overflow"] == 0 and st["edges"] == g.m
        assert np.array_equal(workloads.edges_to_keys(f.export_edges().cpu().numpy()), g.keys)
        par = f.parent().cpu().numpy()
        keys, par, _ = check_batch(f, g.n, keys, par, drsf.DELETE, back)
        keys, par, _ = check_batch(f, g.n, keys, par, drsf.INSERT, back)
    finally:
        f.close()


@pytest.mark.parametrize("flags", [0, drsf.REPL_HS, drsf.REPL_SG], ids=["default", "hs", "sg"])
@pytest.mark.parametrize("b", [1, 513, 2 ** 18 - 1, 2 ** 18, 2 ** 18 + 1])
def test_claim_and_place_around_the_one_launch_limit(b, flags):
    """Inserts around the 2^18 edges up to which one launch claims and places
    them: repeats in both directions, self-loops, edges that exist, rows that
    overflow; the edges go in a second time (all dropped) and out again."""
    n = 60_000
    g = workloads.er_graph(n, n // 2, seed=23)
    rng = np.random.default_rng(b)
    e = rng.integers(0, n, (b, 2)).astype(np.int32)
    e[: b // 4, 0] %= 97                                  # full rows: the overflow list
    q = b // 8
    e[b - q:] = e[:q, ::-1]                               # repeats, turned round
    e[q: q + b // 16, 1] = e[q: q + b // 16, 0]           # self-loops
    e[2 * q: 2 * q + b // 16] = g.edges()[rng.integers(0, g.m, b // 16)]
    e = rng.permutation(e)
    f = make_forest(g, flags=drsf.DETERMINISTIC | flags)
    keys, par = g.keys, g.parent
    try:
        for op in (drsf.INSERT, drsf.INSERT, drsf.DELETE):
            keys, par, _ = check_batch(f, n, keys, par, op, e)
        assert np.array_equal(workloads.edges_to_keys(f.export_edges().cpu().numpy()), keys)
    finally:
        f.close()


@pytest.mark.parametrize("b,detach", [(100, "1"), (5000, "1"), (5000, "0")])
def test_batches_captured_by_the_caller(b, detach, monkeypatch):
    """The caller captures an insert and a delete after the handle has captured
    both shapes itself, runs other batches, and replays its graph on new
    contents of the captured buffer."""
    monkeypatch.setenv("DRSF_DETACH", detach)
    n = 50_000
    g = workloads.er_graph(n, 100_000, seed=31)
    f = make_forest(g)
    keys, par = g.keys, g.parent
    buf = torch.empty((b, 2), dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(b)
    try:
        for c in range(3):
            batch = workloads.insert_batch(n, keys, b, 50 + c)
            for op in (drsf.INSERT, drsf.DELETE):
                keys, par, _ = check_batch(f, n, keys, par, op, batch, labels=False)
        graphs = {}
        for op in (drsf.INSERT, drsf.DELETE):
            graphs[op] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graphs[op]):
                f.apply(op, buf)
        for c in range(3):
            for op in (drsf.INSERT, drsf.DELETE):
                batch = (workloads.insert_batch(n, keys, b, 70 + c) if op == drsf.INSERT
                         else workloads.keys_to_edges(rng.permutation(keys)[:b]))
                buf.copy_(torch.from_numpy(np.ascontiguousarray(batch, np.int32)))
                graphs[op].replay()
                ref = oracle.apply(n, keys, par, op, batch, want_keys=True)
                assert np.array_equal(f.parent().cpu().numpy(), ref.parent)
                keys, par = ref.keys, ref.parent
                keys, par, _ = check_batch(f, n, keys, par, op, batch[:50], labels=False)
    finally:
        f.close()


@pytest.mark.parametrize("batched", [False, (((2 ** 31 - 1, 256, 0, 1),),)], ids=["plain", "persistent"])
@pytest.mark.parametrize("b", [300, 5000, 2 ** 18 + 100])
def test_edges_of_a_full_hub_leave_and_come_back(b, batched):
    """b edges of hubs whose rows are full go to the overflow list, leave and
    come back for many cycles: the list does not grow, and the rows of their
    other ends lose no slots (then, two more edges of each still find one)."""
    hubs, n = 7, b + 100_000
    rng = np.random.default_rng(b)
    ends = np.sort(rng.permutation(np.arange(hubs, n))[:b])
    e = np.stack([np.arange(b) % hubs, ends], 1).astype(np.int32)
    g = workloads.Graph.__new__(workloads.Graph)
    path = np.stack([np.arange(n - 1), np.arange(1, n)], 1)
    g.name, g.n, g.W, g.keys = "hubs", n, 0, workloads.edges_to_keys(path)
    g.parent = np.maximum(np.arange(n) - 1, 0).astype(np.int32)
    f = make_forest(g)
    dev = torch.from_numpy(e).cuda()
    vo, bo = np.array([0, n], np.int64), np.array([0, b], np.int64)
    try:
        st = {}
        for c in range(12):
            for op in (drsf.INSERT, drsf.DELETE):
                if batched is not False:
                    f.apply_batched(op, dev, vo, bo, *batched)
                else:
                    f.apply(op, dev)
                st[op] = f.stats()
            if c == 0:
                most, rebuilds = (st[drsf.INSERT][k] for k in ("overflow", "rebuilds"))   # (room for a batch so long)
            assert st[drsf.INSERT]["overflow"] == most and st[drsf.DELETE]["overflow"] == 0
        assert b - 6 * hubs <= most <= b and f.stats()["rebuilds"] == rebuilds
        keys, par = g.keys, f.parent().cpu().numpy()
        keys, par, st = check_batch(f, n, keys, par, drsf.INSERT, e)
        near = ends[(ends + 5 < n)]
        more = np.stack([near, near + 2], 1)                   # two more for most ends, three at most
        keys, par, st = check_batch(f, n, keys, par, drsf.INSERT, more.astype(np.int32), labels=False)
        assert st["overflow"] == most
        keys, par, st = check_batch(f, n, keys, par, drsf.DELETE, rng.permutation(e))
        assert st["overflow"] == 0
        check_batch(f, n, keys, par, drsf.INSERT, e[::-1], labels=False)
        assert np.array_equal(workloads.edges_to_keys(f.export_edges().cpu().numpy()),
                              np.union1d(keys, workloads.edges_to_keys(e)))
    finally:
        f.close()


def test_removal_at_a_hub_costs_what_it_costs_elsewhere():
    """Half a million edges of one vertex removed from rows and index in less
    than twice the time of as many spread over all vertices (an atomic per edge
    on the hub's row took more than three times as long)."""
    n, b = 1 << 20, 500_000
    rng = np.random.default_rng(2)
    v = np.arange(1, n)
    star = np.stack([np.zeros(n - 1, np.int64), v], 1)
    rest = workloads.keys_to_edges(np.unique(workloads.edges_to_keys(np.stack([v, rng.permutation(v)], 1))))
    rest = rest[rest[:, 0] != rest[:, 1]]
    g = workloads.Graph.__new__(workloads.Graph)
    g.name, g.n, g.W, g.keys = "star", n, 0, np.union1d(workloads.edges_to_keys(star), workloads.edges_to_keys(rest))
    g.parent = np.zeros(n, np.int32)
    f = make_forest(g)
    ms = {}
    try:
        for name, e in (("spread", rest), ("hub", star)):
            d = torch.from_numpy(np.ascontiguousarray(rng.permutation(e)[:b], np.int32)).cuda()
            for _ in range(3):
                f.delete(d)
                f.insert(d)
            f.profile_start(16)
            for _ in range(8):
                f.delete(d)
                f.insert(d)
            ms[name] = f.profile_stop()["delete"]["del_claim"][0]
        assert ms["hub"] < 2 * ms["spread"], ms
    finally:
        f.close()
