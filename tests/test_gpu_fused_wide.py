"""The fused solve on graphs of more than 64 vertices (128-bit sets), on graphs
of different widths through one context (its tables move when the width does),
and the runs that stop because a smaller k has answered."""
import pytest

import oracle
from oracle import bounds
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


def _check(adj, sol, tw):
    assert sol["tw"] == tw
    order = sol["order"].tolist()
    assert sorted(order) == list(range(len(adj)))
    assert oracle.width_q(adj, order) == tw
    assert oracle.verify_td(adj, sol["td_parent"], sol["td_bags"]) == tw


WIDE = {"gnp70": gg.gnp(70, 0.8, 110), "gnp80": gg.gnp(80, 0.9, 120), "path70": gg.path(70), "path128": gg.path(128),
        "k66": gg.complete(66), "gnp128": gg.gnp(128, 0.96, 168)}


@pytest.mark.parametrize("name", list(WIDE))
def test_wide_fused_solve(name):
    adj = WIDE[name]
    lb = max(bounds.mmd(adj), bounds.mmd_plus(adj))
    ref = oracle.solve(adj, k_start=lb, want_order=False)
    exp = oracle.decide(adj, ref["tw"])
    with context(fingerprints=True) as fused, context(fused_states=-1) as loop:
        a = fused.solve(adj, want_td=True)
        b = loop.solve(adj, want_td=True)
    _check(adj, a, ref["tw"])
    for key in ("level_size", "fp_sum", "fp_xor"):
        assert a["stats"][key] == exp[key], key
    for key in ("states_expanded", "candidates", "generated", "decide_runs", "level_size"):
        assert a["stats"][key] == b["stats"][key], key
    assert a["stats"]["kernel_launches"] <= 3 + a["stats"]["levels"]  # (a fingerprint launch per level)


def test_widths_in_turn():
    graphs = [gg.workload_gnp20(), gg.gnp(70, 0.8, 110), gg.gnp(44, 0.5, 4), gg.gnp(80, 0.9, 120), gg.path(9)]
    tws = [oracle.solve(a, k_start=max(bounds.mmd(a), bounds.mmd_plus(a)), want_order=False)["tw"] for a in graphs]
    with context() as c:
        for _ in range(2):
            for adj, tw in zip(graphs, tws):
                _check(adj, c.solve(adj, want_td=True), tw)


@pytest.mark.parametrize("seed", range(4))
def test_runs_above_the_answer_stop(seed):
    # tw is the lower bound: the runs k+1 and k+2, far larger, stop with the
    # first yes; the counters are the first run's alone
    adj = gg.relabel(gg.partial_ktree(28, 4, 921), seed)
    with context(fingerprints=True) as fused, context(fused_states=-1, fingerprints=True) as loop:
        a = [fused.solve(adj, want_td=True) for _ in range(3)]
        b = loop.solve(adj, want_td=True)
    for r in a:
        _check(adj, r, b["tw"])
        for key in ("states_expanded", "generated", "decide_runs", "level_size", "fp_sum", "fp_xor"):
            assert r["stats"][key] == b["stats"][key], key
