"""The fused solve's buffer under a tight memory cap, for graphs of more than 64
vertices: it counts against the cap like the context's other buffers, and gives way
to the level loop of a graph that outgrew it, so the cap holds and the answers are
those without the fused launch.  (For smaller graphs a context holds it besides.)"""
import pytest

import oracle
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu

MB = 1 << 20
# (levels of 0.7 to 1.4 M sets: more than the fused arena holds)
GRAPHS = {"n70": gg.gnp(70, 0.55, 1), "n66": gg.gnp(66, 0.55, 2), "n36": gg.partial_ktree(36, 8, 3)}
BESIDES_MB = {"n70": 0, "n66": 0, "n36": 139}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("cap_mb", [176, 200])
def test_outgrown_graph_under_a_cap(name, cap_mb):
    torch = pytest.importorskip("torch")
    adj = GRAPHS[name]
    with context(fused_states=-1) as warm:  # (every kernel loaded before memory is looked at)
        warm.solve(adj)
    with context(mem_cap_bytes=cap_mb * MB, fused_states=-1) as loop:
        b = loop.solve(adj, want_td=True)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with context(mem_cap_bytes=cap_mb * MB) as c:
        a = c.solve(adj, want_td=True)
        held = free - torch.cuda.mem_get_info()[0]
        # small solves go on through the same context, before and after
        small = [c.solve(gg.workload_gnp20(), want_td=True) for _ in range(2)]
        again = c.solve(adj, want_td=True)
    for r in (a, again):
        assert r["tw"] == b["tw"]
        assert oracle.width_elim(adj, r["order"].tolist()) == b["tw"]
        assert oracle.verify_td(adj, r["td_parent"], r["td_bags"]) == b["tw"]
        for key in ("level_size", "states_expanded", "generated", "decide_runs"):
            assert r["stats"][key] == b["stats"][key], key
    assert [s["tw"] for s in small] == [8, 8]
    # (the context's small fixed buffers, rounded up by the driver)
    assert held <= (cap_mb + BESIDES_MB[name] + 16) * MB, held // MB
