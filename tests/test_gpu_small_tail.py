"""Batches around the candidate limit of the one-block replacement path
(4,096), with super-forests of every shape, against the oracle."""
import numpy as np
import pytest
import torch

import paper_2607_20211_gb300 as drsf
from tests.gpu_util import _tiny_graph, check_batch, make_forest

pytestmark = pytest.mark.gpu
LIMIT = 4096


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    drsf.build()


def _shape(kind, b, rng):
    """b edges over at most 2 b vertices: all candidates of an insert into an edgeless graph."""
    i = np.arange(b)
    if kind == "star":          # one piece is an end of every candidate
        return np.stack([np.zeros(b, np.int64) + b, i], 1)
    if kind == "path":          # the deepest super-forest
        return np.stack([i, i + 1], 1)
    if kind == "pairs":         # 2 b pieces, b super-trees
        return np.stack([2 * i, 2 * i + 1], 1)
    if kind == "dense":         # many rounds, most candidates inside one component
        e = rng.integers(0, 80, (8 * b, 2))
        e = np.unique(np.sort(e[e[:, 0] != e[:, 1]], 1), axis=0)
        return e[rng.permutation(len(e))[:b]]
    e = rng.integers(0, b, (3 * b, 2))
    e = np.unique(np.sort(e[e[:, 0] != e[:, 1]], 1), axis=0)
    return e[rng.permutation(len(e))[:b]]


@pytest.mark.parametrize("b", [1, 2, 33, 1023, 1024, 1025, 2049, LIMIT - 1, LIMIT, LIMIT + 1, 3 * LIMIT])
@pytest.mark.parametrize("kind", ["star", "path", "pairs", "dense", "random"])
def test_insert_shapes(kind, b):
    """An insert whose every edge is a candidate, the same edges deleted
    (one tree edge in three kept) and inserted again, ids permuted."""
    rng = np.random.default_rng(b)
    e = _shape(kind, b, rng)
    n = 2 * b + 100
    e = rng.permutation(n)[e].astype(np.int32)
    g = _tiny_graph(n, [], list(range(n)))
    f = make_forest(g)
    try:
        keys, par, _ = check_batch(f, n, g.keys, g.parent, drsf.INSERT, e)
        keys, par, _ = check_batch(f, n, keys, par, drsf.DELETE, e[np.arange(len(e)) % 3 != 0])
        check_batch(f, n, keys, par, drsf.INSERT, e)
    finally:
        f.close()


@pytest.mark.parametrize("flags", [drsf.REPL_SG, drsf.REPL_HS])
@pytest.mark.parametrize("cuts", [5, 700, 1500, 2800])
def test_delete_candidates(flags, cuts):
    """Deletes whose detached pieces keep several cross edges each: a path
    with chords, cut in many places; both replacement variants."""
    n = 9000
    rng = np.random.default_rng(cuts)
    chords = rng.integers(0, n, (2 * cuts, 2))
    chords = chords[np.abs(chords[:, 0] - chords[:, 1]) > 1]
    edges = [(i, i + 1) for i in range(n - 1)] + [tuple(c) for c in chords.tolist()]
    g = _tiny_graph(n, edges, [max(i - 1, 0) for i in range(n)])
    f = make_forest(g, flags=drsf.DETERMINISTIC | flags)
    at = np.sort(rng.permutation(n - 1)[:cuts])
    b = np.stack([at, at + 1], 1).astype(np.int32)
    try:
        keys, par, _ = check_batch(f, n, g.keys, g.parent, drsf.DELETE, b)
        keys, par, _ = check_batch(f, n, keys, par, drsf.INSERT, b)
        check_batch(f, n, keys, par, drsf.DELETE, b)
    finally:
        f.close()


@pytest.mark.parametrize("cross", [0, 1, 200, 300, 2047, 2048, 2049, 3000, 4096, 4097, 9000])
def test_large_batches_with_few_candidates(cross):
    """Batches above 64K edges (the replacement kernel's form with less shared
    memory) most of whose edges lie inside one tree: candidate counts around
    both forms' limits, inserted and deleted again."""
    core, b = 30_000, 70_000
    n = core + 10_000
    rng = np.random.default_rng(cross)
    inner = rng.integers(0, core, (2 * b, 2))
    inner = inner[np.abs(inner[:, 0] - inner[:, 1]) > 1][:b]
    outer = np.stack([rng.integers(0, core, cross), core + rng.permutation(n - core)[:cross]], 1)
    g = _tiny_graph(n, [(i, i + 1) for i in range(core - 1)], [max(i - 1, 0) for i in range(core)] + list(range(core, n)))
    f = make_forest(g)
    e = rng.permutation(np.concatenate([inner, outer])).astype(np.int32)
    try:
        keys, par, st = check_batch(f, n, g.keys, g.parent, drsf.INSERT, e)
        assert st["replacement"] == cross
        keys, par, _ = check_batch(f, n, keys, par, drsf.DELETE, e)
        check_batch(f, n, keys, par, drsf.INSERT, e)
    finally:
        f.close()


@pytest.mark.parametrize("b", [20, 33, 34, 60, 500, 2047, 2048, 2049, LIMIT - 1, LIMIT])
@pytest.mark.parametrize("shape", ["rising", "falling", "comb"])
def test_deep_super_forests_take_logarithmic_rounds(shape, b):
    """Super-forests deeper than the levels that the orientation takes one by
    one, with hook chains of all pieces (keys that rise along a path): ranked,
    in as many rounds as the tour's length has binary digits."""
    n = 2 * b + 100
    i = np.arange(b)
    d = b // 3
    e = np.stack([np.where(i < d, i, i % max(d, 1)), i + 1], 1) if shape == "comb" else np.stack([i, i + 1], 1)
    e = (n - 1 - e if shape == "falling" else e).astype(np.int32)
    g = _tiny_graph(n, [], list(range(n)))
    f = make_forest(g)
    try:
        keys, par, st = check_batch(f, n, g.keys, g.parent, drsf.INSERT, e)
        depth = d if shape == "comb" else b
        assert (st["rank_rounds"] > 0) == (depth > 32)
        assert st["rank_rounds"] <= (2 * b).bit_length() and st["hook_rounds"] <= b.bit_length()
        keys, par, _ = check_batch(f, n, keys, par, drsf.DELETE, e[np.arange(b) % 5 != 0])
        check_batch(f, n, keys, par, drsf.INSERT, e)
    finally:
        f.close()


@pytest.mark.parametrize("flags", [0, drsf.REPL_SG])
@pytest.mark.parametrize("trees,b", [(2, 30_000), (16, 30_000), (17, 300_000), (100, 100_000), (1000, 400_000)])
def test_parallel_edges_between_few_trees(trees, b, flags):
    """Inserts whose every edge joins two of a few trees: minima and resets of
    few components by all candidates, over several rounds on the grid."""
    n = 200_000
    v = np.arange(n)
    star = np.stack([v % trees, v], 1)[trees:]
    g = _tiny_graph(n, star.tolist(), v % trees)
    rng = np.random.default_rng(trees)
    e = rng.integers(0, n, (b, 2))
    e = e[(e[:, 0] % trees) != (e[:, 1] % trees)].astype(np.int32)
    f = make_forest(g, flags=drsf.DETERMINISTIC | flags)
    try:
        keys, par, st = check_batch(f, n, g.keys, g.parent, drsf.INSERT, e)
        assert st["replacement"] == trees - 1
        keys, par, _ = check_batch(f, n, keys, par, drsf.DELETE, e)
        check_batch(f, n, keys, par, drsf.INSERT, e[: b // 2])
    finally:
        f.close()
