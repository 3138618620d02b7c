"""The work that programs have this framework do, as cases that can be timed.

Almost every case is one step of a sliding window over an evolving graph: one
insert batch (fresh edges, and edges that come back) followed by one delete
batch (the last step's fresh edges, tree edges of long standing and non-tree
edges), with the forest read after each batch.  Two batches P and Q take
turns: a step inserts the one that is absent and deletes the one that is
present, so the graph, the number of tree edges that a delete cuts and the
number of trees that an insert joins stay the same however many steps are
taken.  The tree edges of P are the replacement edges that deleting Q brings
in, and the other way round; `prepare` finds them by running the window for a
few steps, as a program that has been running for a while would have.

Graphs: R-MAT (0.57, 0.19, 0.19, 0.05, ids permuted), Erdos-Renyi, road-like
grids (each 4-neighbour edge with p = 0.6, plus 0.1% shortcuts) and many small
graphs side by side; the initial forest is a BFS forest from the smallest
vertex of each component.  Results are whole numbers and a function of the
inputs alone (minimum-key replacement edges), so they are compared exactly,
and there is no 64-bit value to measure them against.
"""
import math

import numpy as np
import torch

import paper_2607_20211_gb300 as drsf

GRID_KEEP, GRID_SHORTCUTS, GRID_LOCAL = 0.6, 0.001, 64
MASK = 0xFFFFFFFF
WARM_STEPS = 8        # steps of the window that prepare runs (even)


def listed():
    return [
        # A tenant of a serving loop sends its smallest request: launches and
        # latency are all there is to it.
        {"name": "rmat14-b100", "graph": "rmat", "n": 16384, "m": 16384 * 16, "batch": 100, "fresh": 0.5, "cut": 0.25,
         "call": "apply", "labels": False},
        # The small plain configuration: a sparse random graph with many
        # components, whose labels the program reads after each step.
        {"name": "er20k-b2000", "graph": "er", "n": 20000, "m": 25000, "batch": 2000, "fresh": 0.25, "cut": 0.45,
         "call": "apply", "labels": True},
        # A middle-sized tenant with a ragged number of vertices and an odd
        # batch, connectivity read after each step.
        {"name": "rmat200k-b3001", "graph": "rmat", "n": 200003, "m": 200003 * 13, "batch": 3001, "fresh": 0.5,
         "cut": 0.25, "call": "apply", "labels": True},
        # Batches that arrive in host memory, with the counters and the forest
        # read back to the host after each batch.
        {"name": "rmat20-b10k-host", "graph": "rmat", "n": 1 << 20, "m": 16 << 20, "batch": 10000, "fresh": 0.5,
         "cut": 0.25, "call": "host", "labels": False},
        # The largest batches: a sixteenth of the graph's edges each way.
        {"name": "rmat20-b1m", "graph": "rmat", "n": 1 << 20, "m": 16 << 20, "batch": 1000000, "fresh": 0.5,
         "cut": 0.25, "call": "apply", "labels": False},
        # Few edges at a time on a large graph.
        {"name": "rmat22-b100", "graph": "rmat", "n": 1 << 22, "m": 16 << 22, "batch": 100, "fresh": 0.5, "cut": 0.25,
         "call": "apply", "labels": False},
        {"name": "rmat22-b10k", "graph": "rmat", "n": 1 << 22, "m": 16 << 22, "batch": 10000, "fresh": 0.5,
         "cut": 0.25, "call": "apply", "labels": False},
        # The benchmark's workload: 100K-edge batches on R-MAT scale 22.
        {"name": "rmat22-b100k", "graph": "rmat", "n": 1 << 22, "m": 16 << 22, "batch": 100000, "fresh": 0.5,
         "cut": 0.25, "call": "apply", "labels": False},
        # Deep trees: a road-like network, deletes that are mostly tree edges.
        {"name": "grid4096-b100k", "graph": "grid", "n": 4096 * 4096, "m": 20150000, "batch": 100000, "fresh": 0.1,
         "cut": 0.9, "call": "apply", "labels": False},
        # Many independent graphs kept as one union and updated together, by
        # the plain call on the union ...
        {"name": "many256-union", "graph": "many", "graphs": 256, "lo": 1000, "hi": 256000, "share": 0.025,
         "fresh": 0.4, "cut": 0.4, "call": "apply", "labels": False},
        # ... and by the batched call (one group of blocks for each graph).
        {"name": "many128-batched", "graph": "many", "graphs": 128, "lo": 1000, "hi": 65536, "share": 0.025,
         "fresh": 0.4, "cut": 0.4, "call": "batched", "labels": False},
        # A tenant that is not resident is admitted: its handle is built from
        # edge list and forest, takes one insert and one delete batch, is
        # read and closed again.
        {"name": "rmat18-admit", "graph": "rmat", "n": 1 << 18, "m": 16 << 18, "batch": 5000, "fresh": 0.5,
         "cut": 0.25, "call": "admit", "labels": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rmat", "rmat", "rmat", "rmat", "er", "er", "grid", "many", "batched", "admit"])
    call = rng.choice(["apply", "apply", "apply", "host"])
    labels = rng.random() < 0.25
    if kind in ("many", "batched"):
        small = kind == "batched"
        return {"graph": "many", "graphs": _log(rng, 16, 128 if small else 200), "lo": 1000,
                "hi": _log(rng, 8000, 65536 if small else 200000), "share": round(rng.uniform(0.005, 0.025), 5),
                "fresh": 0.4, "cut": 0.4, "call": "batched" if small else "apply", "labels": labels}
    if kind == "grid":
        w, h = _log(rng, 100, 3000), _log(rng, 100, 3000)
        n, m = w * h, int(w * h * (2 * GRID_KEEP + GRID_SHORTCUTS))
        return {"graph": "grid", "n": n, "width": w, "m": m, "batch": _log(rng, 100, min(100000, m // 30)),
                "fresh": 0.1, "cut": 0.9, "call": call, "labels": labels}
    if kind == "er":
        n = _log(rng, 5000, 1000000)
        m = int(n * rng.uniform(1.25, 8.0))
        return {"graph": "er", "n": n, "m": m, "batch": _log(rng, 100, min(300000, m // 12)), "fresh": 0.25,
                "cut": 0.45, "call": call, "labels": labels}
    admit = kind == "admit"
    n = _log(rng, 16384, 1 << (18 if admit else 22))
    m = int(n * rng.uniform(4.0, 16.0))
    return {"graph": "rmat", "n": n, "m": m, "batch": _log(rng, 100, min(500000, m // 16)), "fresh": 0.5,
            "cut": 0.25, "call": "admit" if admit else call, "labels": labels or admit}


# ------------------------------------------------------------------ inputs

def _rand(g, *size):
    return torch.rand(*size, device="cuda", generator=g)


def _keys(u, v):
    """Edge keys (smaller id << 32 | larger id), loops dropped, sorted, each once."""
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    return torch.unique(((lo << 32) | hi)[lo != hi])


def _er(g, n, m):
    return _keys(*(torch.randint(0, n, (2, m), device="cuda", generator=g)))


def _rmat(g, n, m):
    scale = max(1, (n - 1).bit_length())
    m = int(m * ((1 << scale) / n) ** 2)   # pairs with an end >= n are dropped below
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(scale):
        r = _rand(g, m)
        u = (u << 1) | (r >= 0.76)
        v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    perm = torch.randperm(1 << scale, device="cuda", generator=g)
    u, v = perm[u], perm[v]
    keep = (u < n) & (v < n)
    return _keys(u[keep], v[keep])


def _grid(g, w, h):
    n = w * h
    i = torch.arange(n, device="cuda")
    right = i[((i % w) < w - 1) & (_rand(g, n) < GRID_KEEP)]
    down = i[(i < n - w) & (_rand(g, n) < GRID_KEEP)]
    far = torch.randint(0, n, (2, int(round(GRID_SHORTCUTS * n))), device="cuda", generator=g)
    return _keys(torch.cat([right, down, far[0]]), torch.cat([right + 1, down + w, far[1]]))


def _graph(case, g):
    """(vertex offsets of the graphs, width of the grid or 0, edge keys)"""
    if case["graph"] == "many":
        vo, keys = [0], []
        for i in range(case["graphs"]):   # sizes log-uniform, average degrees uniform in [4, 16], in no order
            at, deg = (i * 0.6180339887) % 1, (i * 0.7548776662) % 1
            n = int(case["lo"] * (case["hi"] / case["lo"]) ** at)
            k = (_rmat if i & 1 else _er)(g, n, int(n * (2 + 6 * deg)))
            keys.append(k + ((vo[-1] << 32) | vo[-1]))
            vo.append(vo[-1] + n)
        return vo, 0, torch.cat(keys)
    n = case["n"]
    if case["graph"] == "grid":
        w = case.get("width", math.isqrt(n))
        return [0, n], w, _grid(g, w, n // w)
    return [0, n], 0, (_er if case["graph"] == "er" else _rmat)(g, n, case["m"])


def _bfs_forest(n, keys):
    """BFS forest from each component's smallest vertex; a vertex's parent is its smallest neighbour one level up."""
    u, v = keys >> 32, keys & MASK
    lab = torch.arange(n, device="cuda")
    a, b = u, v
    while a.numel():
        la, lb = lab[a], lab[b]
        lab.scatter_reduce_(0, torch.maximum(la, lb), torch.minimum(la, lb), "amin")
        while True:
            up = lab[lab]
            if torch.equal(up, lab):
                break
            lab = up
        open_ = lab[a] != lab[b]
        a, b = a[open_], b[open_]
    parent = torch.full((n,), n, dtype=torch.int64, device="cuda")
    depth = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    i = torch.arange(n, device="cuda")
    roots = lab == i
    parent[roots], depth[roots] = i[roots], 0
    level = 0
    while u.numel():
        du, dv = depth[u], depth[v]
        open_ = (du < 0) | (dv < 0)
        u, v, du, dv = u[open_], v[open_], du[open_], dv[open_]
        fu, fv = (du == level) & (dv < 0), (dv == level) & (du < 0)
        child, up = torch.cat([v[fu], u[fv]]), torch.cat([u[fu], v[fv]])
        parent.scatter_reduce_(0, child, up, "amin")
        depth[child] = level + 1
        level += 1
    return parent.int()


def _absent(keys, some):
    """Which of some are not among the sorted keys."""
    if not keys.numel():
        return torch.ones_like(some, dtype=torch.bool)
    at = torch.searchsorted(keys, some).clamp(max=keys.numel() - 1)
    return keys[at] != some


def _fresh(case, g, vo, width, keys, count):
    """Two disjoint lists of about count[i] new pairs inside graph i."""
    of = torch.repeat_interleave(torch.arange(len(count), device="cuda"), (2.3 * count).long() + 4)
    base, size = vo[of], vo[of + 1] - vo[of]
    k = of.numel()
    u = (_rand(g, k).double() * size).long()
    if width:
        x = (u % width + torch.randint(-GRID_LOCAL, GRID_LOCAL + 1, (k,), device="cuda", generator=g))
        y = (u // width + torch.randint(-GRID_LOCAL, GRID_LOCAL + 1, (k,), device="cuda", generator=g))
        v = y.clamp(0, int(vo[-1]) // width - 1) * width + x.clamp(0, width - 1)
    else:
        v = (_rand(g, k).double() * size).long()
    pairs = _keys(base + u, base + v)
    pairs = pairs[_absent(keys, pairs)]
    of = torch.searchsorted(vo, pairs >> 32, right=True) - 1
    have = torch.bincount(of, minlength=len(count)).clamp(min=1)
    take = (count / have)[of]
    r = _rand(g, pairs.numel())
    return pairs[r < take], pairs[(r >= take) & (r < 2 * take)]


def _in_tree(parent, keys):
    u, v = keys >> 32, keys & MASK
    return (parent[u] == v) | (parent[v] == u)


def _new_tree_edges(p0, p1):
    """Keys of the tree edges of p1 that p0 does not have."""
    i = torch.arange(p0.numel(), device="cuda")
    q = p1.long()
    m = (q != i) & (p0 != p1) & (p0[q] != i)
    return _keys(i[m], q[m])


def _pick(g, keys, vo, count):
    """About count[i] of the keys inside graph i."""
    of = torch.searchsorted(vo, keys >> 32, right=True) - 1
    have = torch.bincount(of, minlength=len(count)).clamp(min=1)
    return keys[_rand(g, keys.numel()) < (count / have)[of]]


def _batch(g, keys, vo, repeats=True):
    """int32 [b, 2] in random order and orientation, a few pairs twice; grouped by graph, with the groups' offsets."""
    if repeats:
        keys = torch.cat([keys, keys[torch.randperm(keys.numel(), device="cuda", generator=g)[:keys.numel() // 256]]])
    keys = keys[torch.randperm(keys.numel(), device="cuda", generator=g)]
    of = torch.searchsorted(vo, keys >> 32, right=True) - 1
    if len(vo) > 2:
        of, at = torch.sort(of, stable=True)
        keys = keys[at]
    u, v = keys >> 32, keys & MASK
    flip = _rand(g, keys.numel()) < 0.5
    e = torch.stack([torch.where(flip, v, u), torch.where(flip, u, v)], 1).int().contiguous()
    bo = torch.zeros(len(vo), dtype=torch.int64)
    bo[1:] = torch.bincount(of, minlength=len(vo) - 1).cumsum(0).cpu()
    return e, bo.numpy()


def _edges(keys):
    return torch.stack([keys >> 32, keys & MASK], 1).int().contiguous()


# --------------------------------------------------------------- the cases

def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    vo_list, width, keys = _graph(case, g)
    n, vo = vo_list[-1], torch.tensor(vo_list, device="cuda")
    graphs = len(vo_list) - 1
    if "batch" in case:
        size = torch.full((1,), float(case["batch"]), device="cuda")
    else:   # between a fifth and nine fifths of the mean share of each graph's edges
        per = torch.bincount(torch.searchsorted(vo, keys >> 32, right=True) - 1, minlength=graphs)
        size = (_rand(g, graphs) * 1.6 + 0.2) * case["share"] * per
    x0, x1 = _fresh(case, g, vo, width, keys, case["fresh"] * size)
    present = torch.unique(torch.cat([keys, x1]))
    parent = _bfs_forest(n, present)
    cut = _pick(g, keys[_in_tree(parent, keys)], vo, case["cut"] * size)
    f = drsf.DynamicForest(n, _edges(present), parent)

    # the window, a few steps: what the tree edges deleted in one step are
    # replaced by is what the next one deletes
    fresh, gone = (x0, x1), cut[:0]
    for k in range(WARM_STEPS):
        new, old = fresh[k & 1], fresh[1 - (k & 1)]
        f.insert(_edges(torch.cat([gone, new])))
        p0 = f.parent()
        back = gone[_in_tree(p0, gone)]
        f.delete(_edges(torch.cat([cut, old])))
        p1 = f.parent()
        got = _new_tree_edges(p0, p1)
        got = got[_absent(torch.sort(torch.cat([new, back])).values, got)]
        gone, cut = cut, torch.cat([got, back])
    still = keys[~(_in_tree(p0, keys) | _in_tree(p1, keys))]
    still = still[_absent(torch.sort(torch.cat([cut, gone])).values, still)]
    rest = [(1 - case["fresh"]) * size - torch.bincount(torch.searchsorted(vo, s >> 32, right=True) - 1,
                                                        minlength=graphs) for s in (cut, gone)]
    plain = _pick(g, still, vo, sum(r.clamp(min=0) for r in rest))
    side = _rand(g, plain.numel()) < 0.5
    (p, po), (q, qo) = (_batch(g, torch.cat([a, b, c]), vo)
                        for a, b, c in ((cut, plain[side], x1), (gone, plain[~side], x0)))
    f.delete(_edges(plain[~side]))    # now P is present and Q is absent
    f.sync()
    state = {"call": case["call"], "labels": case["labels"], "turn": 0, "batches": (q, p), "offsets": (qo, po),
             "vo": np.asarray(vo_list, np.int64), "n": n}
    if case["call"] == "admit":
        state["edges"], state["parent"] = f.export_edges().clone(), f.parent()
        state["edges"] = _edges(torch.sort((state["edges"][:, 0].long() << 32) | state["edges"][:, 1].long()).values)
        f.close()
    else:
        state["forest"] = f
    if case["call"] == "host":
        state["batches"] = tuple(b.cpu().pin_memory() for b in state["batches"])
    return state


def run(state):
    k = state["turn"]
    call = state["call"]
    (put, take), (po, to) = ((state["batches"][i] for i in (k, 1 - k)), (state["offsets"][i] for i in (k, 1 - k)))
    if call == "admit":
        with drsf.DynamicForest(state["n"], state["edges"], state["parent"]) as f:
            f.insert(put)
            f.delete(take)
            return {"parent": f.parent(), "labels": f.labels()}
    f = state["forest"]
    state["turn"] = 1 - k
    out = {}
    if call == "host":
        for op, name, b in ((drsf.INSERT, "insert", put), (drsf.DELETE, "delete", take)):
            f.apply_host(op, b)
            s = f.stats()
            out[name] = f.parent().cpu()
            out[name + "_counts"] = np.array([s["applied"], s["dropped"], s["tree_cut"], s["replacement"], s["edges"]])
    elif call == "batched":
        f.apply_batched(drsf.INSERT, put, state["vo"], po)
        out["insert"] = f.parent()
        f.apply_batched(drsf.DELETE, take, state["vo"], to)
        out["delete"] = f.parent()
    else:
        f.insert(put)
        out["insert"] = f.parent()
        f.delete(take)
        out["delete"] = f.parent()
    if state["labels"]:
        out["labels"] = f.labels()
    return out


def work(case):
    """Bytes that any implementation moves: each batch read (8 bytes an edge), one entry of an edge index (16) and two row
    entries (8) for each of its edges, the forest read and written once for each batch; an admitted tenant's edge list
    too, with its index and row entries."""
    if case["graph"] == "many":
        n = case["graphs"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        m = 5 * n
        batch = case["share"] * m
    else:
        n, m, batch = case["n"], case["m"], case["batch"]
    moved = 2 * (32 * batch + 8 * n) + (4 * n if case["labels"] else 0)
    if case["call"] == "admit":
        moved += 32 * m + 4 * n
    return {"bytes": float(moved), "flops": 0.0}


def tolerance(case):
    return "exact"
