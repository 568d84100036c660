"""Graphs of up to 64 and of more vertices in turn through one context, with the
default arena (the tables of both widths lie at the same place) and with given
ones (they do not), after runs that gave up and with one and three groups."""
import pytest

import oracle
from oracle import bounds
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu

GRAPHS = [gg.gnp(70, 0.8, 110), gg.workload_gnp20(), gg.gnp(44, 0.5, 4), gg.path(128), gg.path(9)]


@pytest.mark.parametrize("states", [0, 700, 1 << 14])
def test_widths_in_turn_find_empty_tables(states):
    refs = []
    for adj in GRAPHS:
        lb = max(bounds.mmd(adj), bounds.mmd_plus(adj))
        tw = oracle.solve(adj, k_start=lb, want_order=False)["tw"]
        refs.append((tw, oracle.decide(adj, tw)))
    with context(fused_states=states, fingerprints=True) as c:
        for turn in range(3):
            for adj, (tw, exp) in list(zip(GRAPHS, refs))[:: -1 if turn == 1 else 1]:
                one = c.decide(adj, k=tw)  # (one group)
                three = c.solve(adj)
                assert one["yes"] and three["tw"] == tw
                for st in (one["stats"], three["stats"]):
                    for key in ("level_size", "fp_sum", "fp_xor"):
                        assert st[key] == exp[key], (key, turn, len(adj))


@pytest.mark.parametrize("adj", [gg.path(128), gg.path(70), gg.gnp(70, 0.8, 110), gg.workload_gnp20()],
                         ids=["path128", "path70", "gnp70", "gnp20"])
def test_launches_do_not_grow_with_the_levels(adj):
    # the bounds, the fused launch and one launch for all level fingerprints
    with context(fingerprints=True) as c:
        for _ in range(2):
            assert c.solve(adj, want_td=True)["stats"]["kernel_launches"] <= 3
