"""The table is probed in 32-byte sectors and new sets are staged per warp:
level sets must stay exact where sectors overflow (high loads, one- and
few-sector probe limits, which re-run levels with larger tables), where states
have more candidates than one queue pass takes (16), and where a warp's stage
fills several times, for all three state widths."""
import math

import pytest

import oracle
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu

GRAPHS = {"u32": (gg.workload_gnp20(), 8), "u64": (gg.gnp(44, 0.5, 4), 31), "u128": (gg.gnp(80, 0.9, 120), 73)}


@pytest.fixture(scope="module")
def expected():
    return {name: oracle.decide(adj, k) for name, (adj, k) in GRAPHS.items()}


@pytest.mark.parametrize("fused", [0, -1])
@pytest.mark.parametrize("probes,load", [(1, 90), (4, 90), (9, 75), (256, 90)])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_full_sectors(expected, name, probes, load, fused):
    adj, k = GRAPHS[name]
    with context(fingerprints=True, max_probes=probes, table_load_pct=load, fused_states=fused) as c:
        got = c.decide(adj, k=k)["stats"]
    for key in ("level_size", "fp_sum", "fp_xor"):
        assert got[key] == expected[name][key], key


@pytest.mark.parametrize("n", [15, 16, 17, 18, 21])
def test_many_candidates(n):
    # no edges: the empty set alone has n candidates, and level i holds C(n, i) sets
    with context() as c:
        got = c.decide([0] * n, k=0)["stats"]
    assert got["level_size"] == [math.comb(n, i) for i in range(n)]


@pytest.mark.parametrize("n", [33, 66, 70, 128])
def test_many_candidates_wide(n):
    # a star: the centre never passes at k = 1; the levels are stopped early
    with context() as c:
        got = c.decide_level(gg.star(n), 1, 3, count_only=True)
    assert got["stats"]["level_size"][:4] == [math.comb(n - 1, i) for i in range(4)]
