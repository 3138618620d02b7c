"""The pieces of cut trees found over all vertices (no top-down search):
depths around the hops of the first step, slices with and without affected
vertices, and pieces around the weight at which the root piece is scanned
instead, against the oracle."""
import numpy as np
import pytest
import torch

import paper_2607_20211_gb300 as drsf
import workloads
from tests.gpu_util import _tiny_graph, check_batch, make_forest, run_trajectory

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    drsf.build()


@pytest.mark.parametrize("depth", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 33])
def test_chains_of_every_depth(depth, monkeypatch):
    """Many chains of one depth under a common root, some cut at each level,
    half of them with a second way back to the root."""
    monkeypatch.setenv("DRSF_DETACH", "0")
    chains = 700
    n = 1 + chains * depth
    edges, parent = [], [0]
    for c in range(chains):
        for k in range(depth):
            v = 1 + c * depth + k
            edges.append((v, 0 if k == 0 else v - 1))
            parent.append(0 if k == 0 else v - 1)
        if c % 2 and depth > 1:
            edges.append((0, 1 + c * depth + depth - 1))
    g = _tiny_graph(n, edges, parent)
    f = make_forest(g)
    cut = np.array([(1 + c * depth + c % depth, parent[1 + c * depth + c % depth]) for c in range(0, chains, 3)],
                   np.int32)
    try:
        keys, par, _ = check_batch(f, n, g.keys, g.parent, drsf.DELETE, cut)
        keys, par, _ = check_batch(f, n, keys, par, drsf.INSERT, cut)
        check_batch(f, n, keys, par, drsf.DELETE, cut[::2])
    finally:
        f.close()


@pytest.mark.parametrize("below", [4095, 4096, 4097, 9000, 30_000])
def test_piece_weights_around_the_swap(below, monkeypatch):
    """A cut below the root detaches `below` vertices of 34,000 (and a second
    tree is cut in small pieces): the piece left out of the scan changes."""
    monkeypatch.setenv("DRSF_DETACH", "0")
    n, m = 34_000, 2000
    rng = np.random.default_rng(below)
    # vertex 0 - children 1 .. n - below - 1; vertex n - below heads a piece of `below` vertices
    h = n - below
    parent = [0] + [0] * (h - 1) + [0] + [h] * (below - 1)
    edges = [(v, parent[v]) for v in range(1, n)]
    edges += [tuple(e) for e in np.stack([rng.integers(1, h, 500), rng.integers(h, n, 500)], 1).tolist()]
    parent += [n] + [n + i // 2 for i in range(m - 1)]      # second tree, binary
    edges += [(n + 1 + i, n + i // 2) for i in range(m - 1)]
    g = _tiny_graph(n + m, edges, parent)
    f = make_forest(g)
    cut = np.array([(h, 0)] + [(n + i, parent[n + i]) for i in range(5, m, 7)], np.int32)
    try:
        keys, par, _ = check_batch(f, n + m, g.keys, g.parent, drsf.DELETE, cut)
        check_batch(f, n + m, keys, par, drsf.INSERT, cut)
    finally:
        f.close()


def test_trajectories_without_the_top_down_search(monkeypatch):
    monkeypatch.setenv("DRSF_DETACH", "0")
    I, D = drsf.INSERT, drsf.DELETE
    run_trajectory(workloads.rmat_graph(16, 16, seed=2), [(I, 1000), (D, 1000), (I, 10_000), (D, 50_000)] * 2, seed=3)
    run_trajectory(workloads.grid_graph(512, 512, seed=3), [(D, 5000), (I, 5000)] * 2, seed=4, tree_frac=0.9, local=64)
    run_trajectory(workloads.er_graph(20_001, 25_000, seed=1), [(I, 2000), (D, 2000)] * 2, seed=5)


@pytest.mark.parametrize("n", [155_000, 156_673, 200_000, 262_144, 262_145, 622_593, 700_001, 778_241, 1_300_000])
def test_list_room_for_every_grid(n):
    """Chains of 40 over all vertices, each cut once, with a batch that tries
    the top-down search first (it gives up: 40 levels) and with one that does
    not: every block lists vertices, whatever the grid and the vertices per
    block (the lists' room is bounded on the host)."""
    parent = np.arange(n) - (np.arange(n) % 40 != 0)
    edges = np.stack([np.arange(n), parent], 1)[parent != np.arange(n)]
    extra = np.stack([np.arange(0, n - 40, 80) + 5, np.arange(0, n - 40, 80) + 37], 1)   # a second way round
    g = _tiny_graph(n, np.concatenate([edges, extra]).tolist(), parent)
    f = make_forest(g)
    cut = edges[edges[:, 0] % 40 == 9].astype(np.int32)
    more = np.concatenate([cut, edges[edges[:, 0] % 40 == 30], edges[edges[:, 0] % 2 == 1]]).astype(np.int32)
    try:
        keys, par, _ = check_batch(f, n, g.keys, g.parent, drsf.DELETE, cut[:32_000])
        check_batch(f, n, keys, par, drsf.DELETE, more)
    finally:
        f.close()


@pytest.mark.parametrize("depth", [1, 2, 15, 16, 17, 18, 19, 33, 1000, 39_999])
def test_hook_paths_around_the_read_only_walk(depth, monkeypatch):
    """Every vertex of a star is cut off at once and hooks to the vertex before
    it: paths of `depth` hooks, around the 16 steps that a walk takes before it
    halves its path, and one of all pieces."""
    monkeypatch.setenv("DRSF_DETACH", "0")
    n = 40_001
    v = np.arange(1, n)
    star = np.stack([np.zeros(n - 1, np.int64), v], 1)
    path = np.stack([v[:-1], v[1:]], 1)
    path = path[(v[:-1] % (depth + 1)) != 0]
    g = _tiny_graph(n, np.concatenate([star, path]).tolist(), [0] * n)
    f = make_forest(g)
    try:
        keys, par, st = check_batch(f, n, g.keys, g.parent, drsf.DELETE, star)
        assert st["tree_cut"] == n - 1
        check_batch(f, n, keys, par, drsf.INSERT, star)
    finally:
        f.close()


@pytest.mark.parametrize("detached,flags", [(2 ** 19 - 1, 0), (2 ** 19, 0), (2 ** 19 + 2049, 0), (2 ** 20 + 1, 0),
                                            (2 ** 20 + 1, drsf.REPL_HS)])
def test_second_reading_around_its_list(detached, flags):
    """2^19 listed rows and more are listed anew before they are read again,
    and a second round is taken from as many that are left (the last two): a
    star cut at every edge, whose vertices keep random edges among them (hubs
    with rows in parts, and edges outside the rows)."""
    n = detached + 1
    rng = np.random.default_rng(detached)
    v = np.arange(1, n)
    star = np.stack([np.zeros(n - 1, np.int64), v], 1)
    e = rng.integers(1, n, (n, 2))
    e[: n // 8, 0] = 1 + e[: n // 8, 0] % 50
    e = np.sort(e[e[:, 0] != e[:, 1]], 1)
    h = len(e) * 7 // 8
    late = rng.permutation(e)[h:]
    keys = np.unique(workloads.edges_to_keys(np.concatenate([star, e[:h]])))
    g = _tiny_graph(n, workloads.keys_to_edges(keys).tolist(), [0] * n)
    f = make_forest(g, flags=drsf.DETERMINISTIC | flags)
    try:
        keys, par, _ = check_batch(f, n, g.keys, g.parent, drsf.INSERT, late.astype(np.int32), labels=False)
        _, _, st = check_batch(f, n, keys, par, drsf.DELETE, star)
        assert st["tree_cut"] == detached
    finally:
        f.close()


@pytest.mark.parametrize("jump", ["sync", "halving", ""])
@pytest.mark.parametrize("sg", [drsf.REPL_SG, drsf.REPL_HS])
def test_top_down_search_before_every_root_search(jump, sg, monkeypatch):
    """Small deletes look top-down first whatever root search the handle has,
    which takes over where the search gives up (a path is too deep for it)."""
    if jump:
        monkeypatch.setenv("DRSF_JUMP", jump)
    n = 30_000
    rng = np.random.default_rng(7)
    flat = np.stack([rng.integers(0, 60, n - 60), np.arange(60, n)], 1)      # 60 hubs with leaves, chords between
    chords = rng.integers(60, n, (3000, 2))
    hubs = np.stack([np.zeros(59, np.int64), np.arange(1, 60)], 1)
    path = np.stack([np.arange(n - 1), np.arange(1, n)], 1)
    for edges, found in ((np.concatenate([hubs, flat, chords[chords[:, 0] != chords[:, 1]]]), True),
                         (np.concatenate([path, chords[np.abs(chords[:, 0] - chords[:, 1]) > 1]]), False)):
        g = _tiny_graph(n, workloads.keys_to_edges(np.unique(workloads.edges_to_keys(edges))).tolist(),
                        None if found else np.maximum(np.arange(n) - 1, 0))
        f = make_forest(g, flags=drsf.DETERMINISTIC | sg)
        keys, par = g.keys, g.parent
        try:
            for c in range(3):
                v = rng.permutation(np.nonzero(par != np.arange(n))[0])[:500]
                cut = np.stack([v, par[v]], 1).astype(np.int32)
                keys, par, st = check_batch(f, n, keys, par, drsf.DELETE, cut)
                if c == 0:
                    assert (st["detach_levels"] > 0) == found and st["detach_levels"] != 0
                keys, par, _ = check_batch(f, n, keys, par, drsf.INSERT, cut)
        finally:
            f.close()
