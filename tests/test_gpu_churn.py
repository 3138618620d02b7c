"""Edges that leave and come back: storage given up by a delete is taken again
by later inserts, with every batch equal to the oracle's."""
import numpy as np
import pytest
import torch

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
