"""The level-synchronous batched kernel searches graphs of up to 32 vertices on
32-bit sets and larger ones on 64-bit sets, in one launch: level sizes and
fingerprints around the change of width, and orderings, against the oracle."""
import numpy as np
import pytest

import oracle
from oracle import bounds
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


def _graphs():
    return [gg.gnp(n, 0.65, 900 + n) for n in (30, 31, 32, 33, 34, 48)] + [gg.complete(32), gg.path(32), gg.path(33),
                                                                         gg.workload_gnp20()]


@pytest.mark.parametrize("batch_kernel,arena", [(1, 0), (0, 4096)], ids=["level_synchronous", "persistent"])
def test_widths_in_one_batch(batch_kernel, arena):
    graphs = _graphs()
    tws = [oracle.solve(a, k_start=max(bounds.mmd(a), bounds.mmd_plus(a)), want_order=False)["tw"] for a in graphs]
    with context(batch_kernel=batch_kernel, batch_arena_states=arena) as ctx:
        for dk in (0, -1):
            ks = np.array([max(0, tw + dk) for tw in tws], np.int32)
            res = ctx.decide_batch(graphs, ks)
            assert res["status"] == 0
            for g, adj in enumerate(graphs):
                exp = oracle.decide(adj, int(ks[g]))
                L = len(exp["level_size"])
                assert bool(res["yes"][g]) == exp["yes"], g
                assert [int(x) for x in res["level_size"][g][:L]] == exp["level_size"], g
                assert [int(x) for x in res["fp_sum"][g][:L]] == exp["fp_sum"], g
                assert [int(x) for x in res["fp_xor"][g][:L]] == exp["fp_xor"], g
        sol = ctx.solve_batch(graphs)
    assert sol["tw"].tolist() == tws
    pos = 0
    for g, adj in enumerate(graphs):
        order = sol["orders"][pos: pos + len(adj)].tolist()
        assert oracle.width_elim(adj, order) == tws[g]
        pos += len(adj)
