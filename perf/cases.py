"""Performance cases of libtw: the calls that a user of the library makes, each through its Python entry points.

A case is a dict of plain values.  ``prepare`` makes the graphs (or samples) and the context that a program holds
before the call, ``run`` makes the call once, ``work`` says what the call cannot do without, ``exact`` gives the
floating-point outputs from plain numpy in 64 bits, and ``draw`` gives further cases of the same ranges.

Graphs.  The seed of a single-graph case relabels the vertices of one graph of the family: the level sizes (and so the
work) stay those of the case, the sets, the searches and the pairs are others.  Batches are drawn anew from the seed.

Outputs.  Orderings and tree decompositions are computed (the calls ask for them) but not returned: which of several
equally good orderings comes back depends on the order in which the GPU's threads reach the table, so two runs of the
same call differ.  What is returned is exact and the same in every run: answers, level sizes, level fingerprints and the
counters of sets and pairs.
"""
import math

import numpy as np

from paper_1709_09990_gb300 import graphgen as gg
from paper_1709_09990_gb300 import learned, native

_N_PARAMS = 32 * 12 + 32 + 32 + 1


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest call a user makes: the exact treewidth, ordering and decomposition of a 20-vertex graph
        # (32-bit sets, three decide runs of a few thousand sets per level).
        {"name": "solve_gnp20", "call": "solve", "family": "gnp", "n": 20, "par": 0.3, "graph": 0},
        # A sparse graph of ordinary size whose lower bound is its treewidth: one decide run, 64-bit sets, levels of
        # about 10^5 sets.
        {"name": "solve_pktree34", "call": "solve", "family": "pktree", "n": 34, "par": 8, "graph": 8},
        # A dense graph: the sweep makes 13 decide runs of small levels before the first yes.
        {"name": "solve_gnp44", "call": "solve", "family": "gnp", "n": 44, "par": 0.5, "graph": 4},
        # The geometric graph that the library's benchmark quotes: 79 M sets, levels of up to 5.9 M sets.
        {"name": "solve_rgg40", "call": "solve", "family": "rgg", "n": 40, "par": 0.25, "graph": 0},
        # More than 64 vertices: 128-bit sets and a sweep of many short runs.
        {"name": "solve_gnp70", "call": "solve", "family": "gnp", "n": 70, "par": 0.8, "graph": 110},
        # One decide run with its level fingerprints (a caller that checks the wavefront), 32-bit sets, levels of
        # millions of sets.
        {"name": "decide_rgg25", "call": "decide", "family": "rgg", "n": 25, "par": 0.25, "graph": 12, "dk": 0},
        # The wavefront of the partial 10-tree up to level 10 (567 M sets): tables and lists far larger than the L2.
        {"name": "level10_pktree60", "call": "level", "family": "pktree", "n": 60, "par": 10, "graph": 0, "k": 10,
         "level": 10},
        # A few dozen small graphs in one call.
        {"name": "batch_64", "call": "batch", "count": 64, "n_lo": 12, "n_hi": 24},
        # Hundreds of graphs of uneven size in one call: the batch workload's families and sizes, without the sparse
        # large graphs that take seconds each.
        {"name": "batch_512", "call": "batch", "count": 512, "n_lo": 16, "n_hi": 48},
        # The learned starting bound in use: features, proposals, and the certified batched solve from them.
        {"name": "learned_256", "call": "learned", "count": 256, "n_lo": 24, "n_hi": 48},
        # Features (degree statistics, MMD+, min-degree and min-fill widths) of a set of graphs.
        {"name": "features_512", "call": "features", "count": 512, "n_lo": 30, "n_hi": 56},
        # Training of the starting-bound network: 60 epochs over 2000 samples.
        {"name": "train_2000", "call": "train", "count": 2000, "epochs": 60, "minibatch": 256},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gnp", "gnp", "pktree", "pktree", "rgg", "rgg", "wide", "wide", "decide", "decide", "level",
                       "batch", "batch", "learned", "features", "train"])
    graph = rng.randrange(1000)
    if kind == "gnp":
        n = rng.randint(14, 46)
        return {"call": "solve", "family": "gnp", "n": n, "par": round(rng.uniform(_p_lo(n), 0.5), 3), "graph": graph}
    if kind == "pktree":
        k = rng.randint(3, 12)
        return {"call": "solve", "family": "pktree", "n": rng.randint(max(14, k + 2), 32), "par": k, "graph": graph}
    if kind == "rgg":
        return {"call": "solve", "family": "rgg", "n": rng.randint(16, 30), "par": round(rng.uniform(0.25, 0.4), 3),
                "graph": graph}
    if kind == "wide":
        return {"call": "solve", "family": "gnp", "n": rng.randint(65, 128), "par": round(rng.uniform(0.78, 0.95), 3),
                "graph": graph}
    if kind == "decide":
        # a run that answers yes (k = tw), or the last one that answers no
        family = rng.choice(["gnp", "rgg"])
        n = rng.randint(18, 36) if family == "gnp" else rng.randint(18, 28)
        par = round(rng.uniform(_p_lo(n), 0.5) if family == "gnp" else rng.uniform(0.25, 0.4), 3)
        return {"call": "decide", "family": family, "n": n, "par": par, "graph": graph, "dk": rng.choice([0, -1])}
    if kind == "level":
        return {"call": "level", "family": "pktree", "n": rng.randint(52, 64), "par": 10, "graph": graph, "k": 10,
                "level": rng.randint(6, 8)}
    if kind == "batch":
        lo = rng.randint(12, 20)
        return {"call": "batch", "count": _log_int(rng, 16, 400), "n_lo": lo, "n_hi": rng.randint(lo + 4, 46)}
    if kind == "learned":
        lo = rng.randint(16, 28)
        return {"call": "learned", "count": _log_int(rng, 24, 200), "n_lo": lo, "n_hi": rng.randint(lo + 6, 46)}
    if kind == "features":
        lo = rng.randint(12, 40)
        return {"call": "features", "count": _log_int(rng, 16, 600), "n_lo": lo, "n_hi": rng.randint(lo + 4, 100)}
    return {"call": "train", "count": _log_int(rng, 200, 2000), "epochs": rng.randint(10, 60),
            "minibatch": rng.choice([64, 100, 128, 256])}


# ----------------------------------------------------------------- the inputs
def _p_lo(n):
    """Least edge probability drawn for G(n, p): sparser graphs of that size have levels of 10^8 sets and more."""
    return 0.15 + 0.25 * min(1.0, max(0.0, (n - 16) / 30.0))


def _graph(case):
    n, graph = case["n"], case["graph"]
    if case["family"] == "gnp":
        return gg.gnp(n, case["par"], graph)
    if case["family"] == "rgg":
        return gg.rgg(n, case["par"], graph)
    return gg.partial_ktree(n, case["par"], graph)


def _batch(case, seed, count=None):
    """Graphs of the batch workload's two families in turn, n uniform in the case's range: G(n, p), and partial
    k-trees with k in [3, 12] and at most 30 vertices."""
    lo, hi = case["n_lo"], case["n_hi"]
    out = []
    for j in range(case["count"] if count is None else count):
        rng = gg.Rng((seed << 20) + j)
        if j % 2 == 0:
            n = rng.randint(lo, hi)
            p = _p_lo(n) + (0.5 - _p_lo(n)) * rng.uniform()
            out.append(gg.gnp(n, p, 0, rng=rng))
        else:
            n = rng.randint(min(lo, 30), min(hi, 30))
            k = rng.randint(3, min(12, n - 2))
            out.append(gg.partial_ktree(n, k, 0, rng=rng))
    return out


def _feature_graphs(case, seed):
    """As _batch, but both families over the whole range of n (features cost the same whatever the treewidth)."""
    lo, hi = case["n_lo"], case["n_hi"]
    return [gg.mixed_graph((seed << 20) + j, lo, hi, True) if j % 4 else
            gg.partial_ktree(max(lo, 8), 3 + j % 5, (seed << 20) + j) for j in range(case["count"])]


def _samples(case, seed):
    """Feature vectors and targets shaped like those of labelled graphs: n in [12, 40], edge density in [0.1, 0.5], the
    degree statistics that go with them, and a target tw/n that grows with the density."""
    r = np.random.default_rng(seed)
    B = case["count"]
    n = r.integers(12, 41, B).astype(np.float64)
    d = r.uniform(0.1, 0.5, B)
    sd = np.sqrt(d * (1 - d) / n)
    x = np.zeros((B, 12))
    x[:, 0] = n / 64
    x[:, 1] = d
    x[:, 2] = np.clip(d - 2 * sd, 0, 1)
    x[:, 3] = np.clip(d + 2 * sd, 0, 1)
    x[:, 4] = d * (n - 1) / n
    x[:, 5] = sd
    x[:, 6] = np.clip(1.25 - 2.5 * d, 0, 1)
    x[:, 7] = 1 - x[:, 6]
    x[:, 10] = np.clip(1.1 * d + 0.05 * r.standard_normal(B), 0, 1)
    x[:, 11] = np.clip(x[:, 10] + 0.08 + 0.03 * r.standard_normal(B), 0, 1)
    y = 0.6 * x[:, 10] + 0.4 * x[:, 11] + 0.01 * r.standard_normal(B)
    perm = np.stack([r.permutation(B) for _ in range(case["epochs"])]).astype(np.int32)
    return x.astype(np.float32), y.astype(np.float32), perm, learned.init_params(seed)


def _fit(x, y, seed):
    """A small network for the starting bound, fitted in numpy (a program has one from an earlier training)."""
    p = learned.init_params(seed).astype(np.float64)
    x, y = x.astype(np.float64), y.astype(np.float64)
    m, v = np.zeros_like(p), np.zeros_like(p)
    for t in range(1, 301):
        g = _grad(p, x, y)[1]
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p -= 1e-2 * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return p.astype(np.float32)


def prepare(case, seed):
    call = case["call"]
    if call in ("solve", "decide", "level"):
        adj = gg.relabel(_graph(case), seed)
        rows = gg.to_rows_u64(adj)
        state = {"case": case, "rows": rows, "n": len(adj)}
        state["ctx"] = native.Context(fingerprints=call != "solve")
        if call == "decide":
            with native.Context() as c:
                state["k"] = max(0, c.solve(rows, n=len(adj), want_order=False)["tw"] + case["dk"])
        return state
    ctx = native.Context()
    if call == "batch":
        return {"case": case, "ctx": ctx, "graphs": _batch(case, seed)}
    if call == "learned":
        old = _batch(case, seed + 7919, 64)  # graphs solved earlier, which the network was fitted to
        n = np.array([len(a) for a in old], np.float64)
        y = ctx.solve_batch(old, want_orders=False)["tw"] / n
        graphs = _batch(case, seed)
        return {"case": case, "ctx": ctx, "graphs": graphs, "params": _fit(ctx.features(old), y, seed),
                "n": np.array([len(a) for a in graphs], np.int32)}
    if call == "features":
        return {"case": case, "ctx": ctx, "graphs": _feature_graphs(case, seed)}
    x, y, perm, params = _samples(case, seed)
    return {"case": case, "ctx": ctx, "x": x, "y": y, "perm": perm, "params": params}


# ------------------------------------------------------------------- the call
def _u64(values):
    return np.array(values, np.uint64).view(np.int64)


def _counters(stats):
    return {"levels": _u64(stats["level_size"]),
            "sets": stats["states_expanded"], "candidates": stats["candidates"], "pairs": stats["generated"]}


def _levels(stats):
    return {**_counters(stats), "fp_sum": _u64(stats["fp_sum"]), "fp_xor": _u64(stats["fp_xor"])}


def run(state):
    case, ctx = state["case"], state["ctx"]
    call = case["call"]
    if call == "solve":
        r = ctx.solve(state["rows"], n=state["n"], want_order=True, want_td=True)
        return {"tw": r["tw"], **_counters(r["stats"])}
    if call == "decide":
        r = ctx.decide(state["rows"], n=state["n"], k=state["k"], want_order=True)
        return {"yes": r["yes"], **_levels(r["stats"])}
    if call == "level":
        r = ctx.decide_level(state["rows"], n=state["n"], k=case["k"], level=case["level"], count_only=True)
        return {"count": r["count"], **_levels(r["stats"])}
    if call == "batch":
        r = ctx.solve_batch(state["graphs"], want_orders=True)
        return {"tw": r["tw"], "status": r["per_graph_status"]}
    if call == "learned":
        x = ctx.features(state["graphs"])
        hint = learned.propose(ctx, state["params"], x, state["n"], offset=-0.5)
        r = ctx.solve_batch(state["graphs"], k_hint=hint, want_orders=True)
        return {"x": x, "hint": hint, "tw": r["tw"], "status": r["per_graph_status"]}
    if call == "features":
        return {"x": ctx.features(state["graphs"])}
    params = state["params"].copy()
    loss = ctx.mlp_train(params, state["x"], state["y"], case["minibatch"], state["perm"], lr=3e-3)
    return {"params": params, "loss": loss}


# ------------------------------------------------------------------- the work
def work(case):
    """Bytes: every set of the wavefront written and read once (its key and, written only, its last vertex), and the
    rows of the graphs; for the network, the samples and orders.  Operations: the network's multiply-adds (the searches
    are integer work)."""
    call = case["call"]
    if call == "train":
        B, E = case["count"], case["epochs"]
        return {"bytes": B * 52 + B * E * 4 + 3 * _N_PARAMS * 4, "flops": 6 * _N_PARAMS * B * E}
    if call == "features":
        n = (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": case["count"] * (n * 8 * math.ceil(n / 64) + 48), "flops": 0}
    state = prepare(case, 1)
    if call in ("solve", "decide", "level"):
        n = state["n"]
        sets = run(state)["sets"]
        w = 4 if n <= 32 else 8 if n <= 64 else 16
        return {"bytes": sets * (2 * w + 1) + n * 8 * math.ceil(n / 64), "flops": 0}
    r = state["ctx"].solve_batch(state["graphs"])
    rows = sum(len(a) for a in state["graphs"])
    return {"bytes": r["stats"]["states_expanded"] * 17 + rows * 8, "flops": 0}


# ------------------------------------------------------- 64-bit reference values
def _grad(p, x, y):
    """Loss terms (yhat - y)^2 and the gradient of their mean for the 12-32-1 ReLU network."""
    W1, b1, W2, b2 = p[:384].reshape(32, 12), p[384:416], p[416:448], p[448]
    z = x @ W1.T + b1
    h = np.maximum(z, 0)
    diff = h @ W2 + b2 - y
    g = 2 * diff / len(y)
    dz = (g[:, None] * W2) * (z > 0)
    return diff * diff, np.concatenate([(dz.T @ x).ravel(), dz.sum(0), g @ h, [g.sum()]])


def _features64(adj):
    n = len(adj)
    deg = [a.bit_count() for a in adj]
    s, s2 = sum(deg), sum(d * d for d in deg)
    hist = [0, 0, 0, 0]
    for d in deg:
        hist[min(3, 4 * d // n)] += 1

    def bits(a):
        while a:
            b = a & -a
            yield b.bit_length() - 1
            a ^= b

    # MMD+: contract a vertex of least degree into its neighbour of least degree
    rows, alive, mmd_plus = list(adj), (1 << n) - 1, 0
    while alive.bit_count() >= 2:
        v = min(bits(alive), key=lambda u: (rows[u] & alive).bit_count())
        nv = rows[v] & alive
        mmd_plus = max(mmd_plus, nv.bit_count())
        if nv:
            u = min(bits(nv), key=lambda t: (rows[t] & alive).bit_count())
            rows[u] |= nv & ~(1 << u)
            for t in bits(nv & ~(1 << u)):
                rows[t] |= 1 << u
        alive &= ~(1 << v)

    def width(cost):
        rows, alive, most = list(adj), (1 << n) - 1, 0
        while alive:
            v = min(bits(alive), key=lambda u: cost(rows, rows[u] & alive))
            nv = rows[v] & alive
            most = max(most, nv.bit_count())
            for t in bits(nv):
                rows[t] |= nv & ~(1 << t)
            alive &= ~(1 << v)
        return most

    by_degree = width(lambda rows, nu: nu.bit_count())
    by_fill = width(lambda rows, nu: sum((nu & ~rows[a] & ~(1 << a)).bit_count() for a in bits(nu)))
    return [n / 64, s / (n * (n - 1)), min(deg) / n, max(deg) / n, s / (n * n), math.sqrt(n * s2 - s * s) / (n * n),
            *(h / n for h in hist), mmd_plus / n, (by_degree + by_fill) / (2 * n)]


def exact(case, seed):
    call = case["call"]
    if call == "features":
        return {"x": np.array([_features64(a) for a in _feature_graphs(case, seed)], np.float64)}
    if call == "learned":
        x = np.array([_features64(a) for a in _batch(case, seed)], np.float64)
        return {"x": x, "hint": None, "tw": None, "status": None}
    if call != "train":
        return None  # whole numbers only
    x, y, perm, params = _samples(case, seed)
    x, y, p = x.astype(np.float64), y.astype(np.float64), params.astype(np.float64)
    m, v, t, loss = np.zeros_like(p), np.zeros_like(p), 0, []
    for order in perm:
        total = 0.0
        for at in range(0, len(order), case["minibatch"]):
            idx = order[at: at + case["minibatch"]]
            sq, g = _grad(p, x[idx], y[idx])
            total += sq.sum()
            t += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 3e-3 * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        loss.append(total / len(order))
    return {"params": p, "loss": np.array(loss)}
