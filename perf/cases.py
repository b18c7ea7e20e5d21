"""Performance cases of the K-Best graph edit distance library.

Each case is a batch of graph pairs that goes through a public entry point of the binding
(paper_2605_00830_gb300/fastged.py): fastged_batch_ex on host graphs (the whole call: flatten,
upload, kernels, download), a device-resident plan that is run and read back, or
fastged_cross for a distance matrix. The shapes are those of the repository's workloads
(paper_2605_00830_gb300/workloads.py) and of its tests; every graph is drawn from the seed.

A case is a dict:
  entry     "batch", "plan" or "cross"
  shape     "tiny" (ER, 5-8 vertices), "molecule" (tree + rings), "dense" (ER), "large" (BA and
            an edited copy), "sweep" (a pair of G(n, 0.4)), "mix" (70 % molecule, 25 % dense,
            5 % large, as the serving stream)
  pairs     graph pairs; n_lo, n_hi: vertices per graph
  K         beam width; per_pair_k: each pair draws 32, 128 or 512 instead
  cost      "unit", "setting1" or "setting2"; variant, vertex_order: the call's options
  rows, cols    the two sides of a distance matrix (entry "cross")
"""
import math

import numpy as np

from paper_2605_00830_gb300 import fastged as F
from paper_2605_00830_gb300 import workloads as W

COSTS = {"unit": W.UNIT_COSTS, "setting1": W.SETTING1_COSTS, "setting2": W.SETTING2_COSTS}
SERVED_K = (32, 128, 512)


def _case(name, entry, shape, pairs, n_lo, n_hi, K, cost="setting1", **more):
    c = {"name": name, "entry": entry, "shape": shape, "pairs": pairs, "n_lo": n_lo,
         "n_hi": n_hi, "K": K, "cost": cost, "per_pair_k": False, "variant": 0,
         "vertex_order": 0, "rows": 0, "cols": 0}
    c.update(more)
    return c


def listed():
    return [
        # one query of an interactive user: a single molecule pair from host memory
        _case("single_query", "batch", "molecule", 1, 24, 30, 100),
        # the plain method's small random graphs, a resident batch: launch and latency bound
        _case("tiny_plan", "plan", "tiny", 200, 5, 8, 16, "unit"),
        # the headline workload: a resident batch of molecule pairs
        _case("molecule_plan", "plan", "molecule", 20000, 10, 40, 100),
        # the same pairs in a user's hands: host graphs in, costs and maps out, the paper's
        # second cost setting
        _case("molecule_setting2", "batch", "molecule", 5003, 10, 40, 100, "setting2"),
        # what a server batches: molecule queries, each with its own K
        _case("molecule_served", "batch", "molecule", 4096, 10, 40, 512, per_pair_k=True),
        # nearest-neighbour classification: one GED matrix of test against training graphs
        _case("knn_matrix", "cross", "molecule", 0, 10, 40, 20, rows=61, cols=256),
        # the search's two options together: completing every last-level successor, and
        # branching by descending degree
        _case("molecule_options", "batch", "molecule", 1001, 10, 40, 100, variant=1,
              vertex_order=1),
        # dense random graphs of 50-200 vertices
        _case("dense_plan", "plan", "dense", 1024, 50, 200, 256, "unit"),
        # large sparse graphs and their edited copies
        _case("large_plan", "plan", "large", 64, 500, 1000, 1024, "unit"),
        # a slice of the serving stream as one batch: three shapes, per-query K
        _case("serving_mix", "batch", "mix", 400, 10, 1000, 512, per_pair_k=True),
        # the paper's K sweep: small graphs, a beam of 100,000
        _case("wide_beam", "plan", "molecule", 16, 18, 22, 100000),
        # the paper's graph-size sweep: one dense pair, K = 5,000
        _case("size_sweep", "batch", "sweep", 1, 200, 200, 5000),
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.randrange(9)
    entry = rng.choice(["batch", "plan"])
    cost = rng.choice(["unit", "setting1", "setting2"])
    if kind == 0:
        return _drawn(entry, "tiny", _log(rng, 1, 2000), 5, 8, _log(rng, 1, 64), cost)
    if kind == 1:
        lo = rng.randint(2, 20)
        return _drawn(entry, "molecule", _log(rng, 1, 20000), lo, rng.randint(lo + 5, 40),
                      _log(rng, 8, 128), cost)
    if kind == 2:
        return _drawn(entry, "molecule", _log(rng, 1, 3000), 10, rng.randint(30, 60),
                      _log(rng, 130, 2000), cost)
    if kind == 3:
        return _drawn("batch", "molecule", _log(rng, 50, 5000), 10, 40, 512, "setting1",
                      per_pair_k=True)
    if kind == 4:
        return _drawn("batch", "molecule", _log(rng, 10, 2000), 10, 40, _log(rng, 16, 128),
                      cost, variant=rng.randint(0, 1), vertex_order=rng.randint(0, 1))
    if kind == 5:
        lo = rng.randint(40, 80)
        return _drawn(entry, "dense", _log(rng, 1, 600), lo, rng.randint(lo + 20, 250),
                      _log(rng, 16, 512), cost)
    if kind == 6:
        lo = rng.randint(260, 600)
        return _drawn(entry, "large", _log(rng, 1, 24), lo, rng.randint(lo + 10, 1000),
                      _log(rng, 32, 1024), rng.choice(["unit", "setting1"]))
    if kind == 7:
        return _drawn("plan", "molecule", _log(rng, 1, 16), 18, rng.randint(20, 24),
                      _log(rng, 2000, 100000), "setting1")
    n = rng.randint(30, 200)
    return _drawn(entry, "sweep", rng.randint(1, 3), n, n, _log(rng, 500, 5000), "setting1")


def _drawn(*args, **more):
    c = _case("", *args, **more)
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------------------

_ZIPF_CDF = np.cumsum(np.arange(1, 11) ** -1.2 / (np.arange(1, 11) ** -1.2).sum())


def _sizes(case, count, lo, hi):
    """Vertices of `count` graphs, uniform on [lo, hi]. They follow from the case alone (and
    everything else from the seed), so that the outputs of every seed have the same lengths."""
    return np.random.default_rng([case["pairs"], case["n_lo"], case["n_hi"], count]).integers(
        lo, hi + 1, count)


def _molecules(rng, n):
    """Molecule-like graphs of n[k] vertices, as workloads.molecule_like draws them (a random recursive tree and
    up to three ring edges, Zipf vertex labels, edge labels 0/1/2 at 70/25/5 %), all at once."""
    count = len(n)
    first = np.concatenate([[0], np.cumsum(n)])
    lab = np.minimum(np.searchsorted(_ZIPF_CDF, rng.random(first[-1]), side="right"), 9)
    g = np.repeat(np.arange(count), n)
    t = np.arange(first[-1]) - first[g]
    par = np.floor(rng.random(first[-1]) * t).astype(np.int64)
    tree = t > 0
    # tree edges first, then ring candidates in drawing order; a repeated key is dropped
    tries = 8
    cg = np.repeat(np.arange(count), tries)
    ca, cb = (np.floor(rng.random(count * tries) * n[cg]).astype(np.int64) for _ in range(2))
    ok = ca != cb
    key = np.concatenate([(g[tree] << 20) | (par[tree] << 10) | t[tree],
                          (cg[ok] << 20) | (np.minimum(ca, cb)[ok] << 10) | np.maximum(ca, cb)[ok]])
    _, idx = np.unique(key, return_index=True)
    ring = np.sort(idx[idx >= tree.sum()])
    rg = key[ring] >> 20
    rank = np.arange(len(ring)) - np.searchsorted(rg, rg, side="left")
    extra = rng.integers(0, 4, count)
    key = np.sort(np.concatenate([key[:tree.sum()], key[ring[rank < extra[rg]]]]))
    eg = key >> 20
    edges = np.stack([(key >> 10) & 1023, key & 1023], axis=1).astype(np.int32)
    el = np.minimum(np.searchsorted([0.70, 0.95, 1.0], rng.random(len(key)), side="right"), 2)
    cut = np.searchsorted(eg, np.arange(count + 1))
    lab, el = lab.astype(np.int32), el.astype(np.int32)
    return [W.Graph(int(n[k]), lab[first[k]:first[k + 1]], edges[cut[k]:cut[k + 1]],
                    el[cut[k]:cut[k + 1]]) for k in range(count)]


def _er(rng, n, p, labels):
    n = int(n)
    a, b = np.triu_indices(n, 1)
    on = rng.random(len(a)) < p
    return W.Graph(n, rng.integers(0, labels, n).astype(np.int32),
                   np.stack([a[on], b[on]], axis=1).astype(np.int32))


def _large(rng, n):
    """A BA graph (m = 3) and its copy after 2-10 % of edits, as the large workload's pairs."""
    st = W.Stream(int(rng.integers(1 << 62)))
    g1 = W.barabasi_albert(st, int(n), 3, 16)
    return [g1, W.perturb(st, g1, float(rng.uniform(0.02, 0.1)), 16)]


def _inputs(case, seed):
    """(graphs, pairs, per-pair K or None) of a case."""
    rng = np.random.default_rng([seed, 77])
    lo, hi, P = case["n_lo"], case["n_hi"], case["pairs"]
    if case["entry"] == "cross":
        graphs = _molecules(rng, _sizes(case, case["rows"] + case["cols"], lo, hi))
        r, c = np.meshgrid(np.arange(case["rows"]), np.arange(case["cols"]), indexing="ij")
        return graphs, np.stack([r.ravel(), c.ravel() + case["rows"]], axis=1), None
    def sparse_to_dense(n):
        return _er(rng, n, rng.uniform(0.05, 0.5), 8)

    if case["shape"] == "tiny":
        graphs = [_er(rng, n, 0.35, 4) for n in _sizes(case, 2 * P, lo, hi)]
    elif case["shape"] == "molecule":
        graphs = _molecules(rng, _sizes(case, 2 * P, lo, hi))
    elif case["shape"] == "dense":
        graphs = [sparse_to_dense(n) for n in _sizes(case, 2 * P, lo, hi)]
    elif case["shape"] == "large":
        graphs = [g for n in _sizes(case, P, lo, hi) for g in _large(rng, n)]
    elif case["shape"] == "sweep":
        graphs = [_er(rng, lo, 0.4, 4) for _ in range(2 * P)]
    else:
        # the stream's shares, the shapes spread over the batch
        mol = iter(_molecules(rng, _sizes(case, 2 * P, 10, 40)))
        er, ba = _sizes(case, 2 * P, 50, 200), _sizes(case, P, 500, 1000)
        graphs = []
        for p in range(P):
            if p % 20 == 7:
                graphs += _large(rng, ba[p])
            elif p % 4 == 1:
                graphs += [sparse_to_dense(er[2 * p]), sparse_to_dense(er[2 * p + 1])]
            else:
                graphs += [next(mol), next(mol)]
    pairs = np.arange(2 * P, dtype=np.int32).reshape(-1, 2)
    kpp = rng.choice(SERVED_K, P).astype(np.int32) if case["per_pair_k"] else None
    return graphs, pairs, kpp


class _State:
    """A user's handle, graphs in the C layout, plan and output arrays."""

    def __init__(self, case, seed):
        graphs, pairs, kpp = _inputs(case, seed)
        self.case, self.K, self.plan = case, case["K"], 0
        self.ged = F.FastGED(COSTS[case["cost"]])
        self.opt = F.make_options(k_per_pair=kpp, variant=case["variant"],
                                  vertex_order=case["vertex_order"])
        if case["entry"] == "cross":
            self.graphs = graphs
            self.rows = np.arange(case["rows"])
            self.cols = np.arange(case["rows"], case["rows"] + case["cols"])
            return
        self.mm = F.Marshalled(graphs, pairs)
        self.out = (np.zeros(self.mm.n_pairs, np.int32),
                    np.zeros(int(self.mm.map_off[-1]), np.int32),
                    np.zeros(self.mm.n_pairs, np.int64))
        if case["entry"] == "plan":
            self.plan = F.fastged_plan_create(self.ged.h, self.mm, self.K, self.opt)

    def __del__(self):
        try:
            if self.plan:
                F.fastged_plan_destroy(self.plan)
            self.ged.close()
        except Exception:
            pass


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    if state.case["entry"] == "cross":
        return F.fastged_cross(state.ged.h, state.graphs, state.rows, state.cols, state.K)
    cost, maps, nev = state.out
    if state.plan:
        F.fastged_plan_run(state.plan)
        F.fastged_plan_read(state.plan, cost, maps, nev)
    else:
        F.fastged_batch_ex(state.ged.h, state.mm, state.K, state.opt, cost, maps, nev)
    return {"cost": cost, "map": maps, "n_evals": nev}


# ---- what a pass cannot do without ------------------------------------------------------

def _pair_work(shape, lo, hi, K):
    """(input and output bytes, successors) of one pair of mean size."""
    n = (lo + hi) / 2.0
    if shape == "molecule":
        m, edge_bytes = n + 0.5, 12
    elif shape == "large":
        m, edge_bytes = 3.0 * n, 8
    else:
        m, edge_bytes = {"tiny": 0.35, "dense": 0.275, "sweep": 0.4}[shape] * n * (n - 1) / 2, 8
    width, succ = 1.0, 0.0
    for i in range(int(n)):
        level = width * max(n - i * min(1.0, (n - 1) / n) + 1, 1)
        succ += level
        width = min(K, level)
    return 2 * (4 * n + edge_bytes * m) + 8 + 4 * n + 12, succ


def work(case):
    """bytes: labels and edges of both graphs, the pair, its cost, map and count. flops: one
    integer operation per successor, whose PED the method's n_evals counts."""
    Ks = SERVED_K if case["per_pair_k"] else (case["K"],)
    parts = [(1.0, case["shape"], case["n_lo"], case["n_hi"])]
    if case["shape"] == "mix":
        parts = [(0.7, "molecule", 10, 40), (0.25, "dense", 50, 200), (0.05, "large", 500, 1000)]
    b = s = 0.0
    for share, shape, lo, hi in parts:
        for K in Ks:
            pb, ps = _pair_work(shape, lo, hi, K)
            b += share * pb / len(Ks)
            s += share * ps / len(Ks)
    if case["entry"] == "cross":
        # the graphs once each, a cost per entry
        P, n = case["rows"] * case["cols"], case["rows"] + case["cols"]
        mean = (case["n_lo"] + case["n_hi"]) / 2.0
        return {"bytes": n * (4 * mean + 12 * (mean + 0.5)) + 4 * P, "flops": P * s}
    return {"bytes": case["pairs"] * b, "flops": case["pairs"] * s}


# ---- the results from plain numpy -------------------------------------------------------

def _dense_form(g):
    adj = np.zeros((g.n + 1, g.n + 1), np.int64)   # a last row and column without neighbours
    lab = np.zeros((g.n + 1, g.n + 1), np.int64)
    a, b = g.edges[:, 0], g.edges[:, 1]
    adj[a, b] = adj[b, a] = 1
    if g.elabel is not None:
        lab[a, b] = lab[b, a] = g.elabel
    return adj, lab


def _solve(g1, g2, cost, K, variant, by_degree):
    """(cost, map, evaluations) of Algorithm 1 for one pair: levels of (PED, parent slot,
    child) triples, the deletion last, the K least kept in that order."""
    vsub, vdel, vins, esub, edel, eins = cost
    A1, L1 = _dense_form(g1)
    A2, L2 = _dense_form(g2)
    n1, n2, m2 = g1.n, g2.n, len(g2.edges)
    order = np.arange(n1)
    if by_degree:
        order = np.argsort(-A1[:n1, :n1].sum(1), kind="stable")
    maps = np.full((1, 0), n2)
    ped = np.zeros(1, np.int64)
    used = np.zeros((1, n2 + 1), np.int64)
    nev = 0

    def complete(p, us):
        inside = np.einsum("su,uv,sv->s", us, A2, us) // 2
        return p + vins * (n2 - us[:, :n2].sum(1)) + eins * (m2 - inside)

    for i, v in enumerate(order):
        prior = [(t, order[t]) for t in range(i) if A1[v, order[t]]]
        hit = np.zeros((len(ped), n2 + 1), np.int64)
        other = np.zeros((len(ped), n2 + 1), np.int64)
        for t, x in prior:
            row = A2[maps[:, t]]
            hit += row
            other += row * (L2[maps[:, t]] != L1[v, x])
        C = np.concatenate([(g2.vlabel != g1.vlabel[v]) * vsub, [vdel]])
        d = ped[:, None] + C + eins * (used @ A2 - hit) + edel * (len(prior) - hit) + esub * other
        slot, child = np.nonzero(1 - used * (np.arange(n2 + 1) < n2))
        d = d[slot, child]
        nev += len(d)
        if variant == 1 and i == n1 - 1:
            nxt = used[slot]
            nxt[np.arange(len(d)), child] |= child < n2
            total = complete(d, nxt)
            nev += len(d)
            best = np.lexsort((np.arange(len(d)), d, total))[0]
            m = np.append(maps[slot[best]], child[best])
            return total[best], m, nev, order
        keep = np.argsort(d, kind="stable")[:K]
        slot, child, ped = slot[keep], child[keep], d[keep]
        maps = np.concatenate([maps[slot], child[:, None]], axis=1)
        used = used[slot]
        used[np.arange(len(ped)), child] |= child < n2
    total = complete(ped, used)
    best = int(np.argmin(total))
    return total[best], maps[best], nev + len(ped), order


def exact(case, seed):
    if case["shape"] not in ("tiny", "molecule") or case["entry"] == "cross":
        return None
    if work(case)["flops"] > 6e6 or case["pairs"] > 300:
        return None
    graphs, pairs, kpp = _inputs(case, seed)
    costs, maps, nevs = [], [], []
    for p, (a, b) in enumerate(pairs):
        c, m, n, order = _solve(graphs[a], graphs[b], COSTS[case["cost"]],
                                int(kpp[p]) if kpp is not None else case["K"],
                                case["variant"], case["vertex_order"])
        out = np.zeros(len(m), np.int64)
        out[order] = np.where(m == graphs[b].n, -1, m)
        costs.append(c)
        maps.append(out)
        nevs.append(n)
    return {"cost": np.array(costs), "map": np.concatenate(maps), "n_evals": np.array(nevs)}
