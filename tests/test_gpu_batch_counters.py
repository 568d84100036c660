"""The totals of a batched call count every decide run once, whichever kernels a
graph passes through: runs that a kernel gave up because they outgrew it, and that
the next one makes again, are not counted twice."""
import numpy as np
import pytest

from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu

KEYS = ("states_expanded", "candidates", "generated", "decide_runs")


def _graphs():
    # runs of a few sets up to levels of 13 M: graphs that stay in the persistent
    # kernel, that leave it (above 2^12 sets), and that leave the level-synchronous
    # one too (above 2^21 sets a level)
    small = [gg.mixed_graph(4000 + j, 10, 30, j % 2 == 0) for j in range(24)]
    return small + [gg.gnp(44, 0.3, 1), gg.path(70), gg.gnp(40, 0.45, 2)]


def _sum(stats):
    return {key: sum(s[key] for s in stats) for key in KEYS}


@pytest.mark.parametrize("cfg", [{}, {"batch_kernel": 1}, {"batch_arena_states": 4096}, {"batch_arena_states": 1 << 19}],
                         ids=["default", "level_synchronous", "small_arena", "large_arena"])
def test_totals_are_those_of_the_graphs_runs(cfg):
    graphs = _graphs()
    with context() as one, context(**cfg) as batch:
        single = [one.solve(a, want_order=False) for a in graphs]
        tw = np.array([r["tw"] for r in single])
        got = batch.solve_batch(graphs)
        assert got["tw"].tolist() == tw.tolist()
        assert {key: got["stats"][key] for key in KEYS} == _sum([r["stats"] for r in single])
        # one run per graph; k = tw (yes) and below it (no)
        for dk in (0, 1):
            ks = np.maximum(tw - dk, 0).astype(np.int32)
            runs = [one.decide(a, k=int(k))["stats"] for a, k in zip(graphs, ks)]
            res = batch.decide_batch(graphs, ks)
            assert res["status"] == 0
            assert {key: res["stats"][key] for key in KEYS} == _sum(runs)


@pytest.mark.parametrize("cfg", [{}, {"batch_kernel": 1}], ids=["default", "level_synchronous"])
def test_totals_with_proposed_bounds(cfg):
    # proposals below tw: the runs from there (or from the lower bound) up to tw
    graphs = _graphs()
    with context() as one, context(**cfg) as batch:
        tw = [one.solve(a, want_order=False)["tw"] for a in graphs]
        lb = [int(max(one.bounds(a)[:2])) for a in graphs]
        runs = [one.decide(a, k=k)["stats"] for a, t, b in zip(graphs, tw, lb) for k in range(max(t - 1, b), t + 1)]
        got = batch.solve_batch(graphs, k_hint=np.array(tw, np.float32) - 1)
        assert got["tw"].tolist() == tw
        assert {key: got["stats"][key] for key in KEYS} == _sum(runs)
