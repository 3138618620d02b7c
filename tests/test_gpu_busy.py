"""Deletes whose first hooking round is taken from the rows, on a device that
other streams keep busy: blocks of the replacement kernel that start late read
the same counts as the ones that have finished."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_20211_gb300 as drsf
from tests.gpu_util import _tiny_graph, dev_tensor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    drsf.build()


@pytest.mark.parametrize("flags", [0, drsf.REPL_HS, drsf.REPL_SG], ids=["default", "hs", "sg"])
@pytest.mark.parametrize("cuts", [60, 100, 130, 200, 260, 900, 2100, 3000, 5000])
def test_late_blocks_take_the_same_branch(cuts, flags, monkeypatch):
    """Edges that the scan chose and candidates left, together around 256 and
    4,096 (where the replacement kernel changes its form): a path with a
    sparse set of chords, so that the default is the hooking variant, on four
    handles with streams of their own beside a stream of plain kernels."""
    monkeypatch.setenv("DRSF_DETACH", "0")
    n, handles, cycles = 200_000, 4, 3
    rng = np.random.default_rng(cuts)
    lo = rng.integers(0, n - 400, 12_000)
    chords = np.stack([lo, lo + rng.integers(2, 400, len(lo))], 1)
    edges = np.concatenate([np.stack([np.arange(n - 1), np.arange(1, n)], 1), chords])
    g = _tiny_graph(n, edges.tolist(), np.maximum(np.arange(n) - 1, 0))
    at = np.sort(rng.permutation(n - 1)[:cuts])
    batch = np.stack([at, at + 1], 1).astype(np.int32)
    own = [drsf.OwnStream(0) for _ in range(handles)]
    fs, outs = [], [[] for _ in range(handles)]
    busy, a = torch.cuda.Stream(), torch.randn(1536, 1536, device="cuda")
    try:
        for o in own:
            with torch.cuda.stream(o.torch):
                fs.append(drsf.DynamicForest(n, dev_tensor(g.edges()), dev_tensor(g.parent),
                                             flags=drsf.DETERMINISTIC | flags, stream=o.torch))
        dev = dev_tensor(batch)
        torch.cuda.synchronize()
        for _ in range(cycles):
            for op in (drsf.DELETE, drsf.INSERT):
                with torch.cuda.stream(busy):
                    for _ in range(4):
                        a = a @ a * 1e-3
                for f, o, out in zip(fs, own, outs):
                    with torch.cuda.stream(o.torch):
                        f.apply(op, dev)
                        out.append(f.parent())
        torch.cuda.synchronize()
        for f in fs:
            f.sync()
        keys, par = g.keys, g.parent
        for k in range(2 * cycles):
            ref = oracle.apply(n, keys, par, drsf.INSERT if k & 1 else drsf.DELETE, batch, want_keys=True)
            keys, par = ref.keys, ref.parent
            for out in outs:
                assert np.array_equal(out[k].cpu().numpy(), par), k
    finally:
        for f in fs:
            f.close()
        for o in own:
            o.close()
