"""The level-synchronous batch under a memory cap that its graphs exceed together
but not alone: every graph is answered, with the levels of its own run, and the
device memory held during the call keeps to the cap."""
import threading

import numpy as np
import pytest

import oracle
from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _graphs():
    # sixteen relabelled copies of two graphs whose runs keep 7.7 and 2.8 M sets
    # (12 B each), and small ones between them
    out = []
    for j in range(8):
        out += [gg.relabel(gg.partial_ktree(36, 8, 3), j), gg.workload_gnp20(), gg.relabel(gg.gnp(44, 0.42, 1), j)]
    return out


class _Lowest:
    """Least free device memory while the block runs."""

    def __enter__(self):
        import torch
        self.look = lambda: torch.cuda.mem_get_info()[0]
        torch.cuda.synchronize()
        self.first = self.least = self.look()
        self.stop = False
        self.thread = threading.Thread(target=self._run)
        self.thread.start()
        return self

    def _run(self):
        while not self.stop:
            self.least = min(self.least, self.look())

    def __exit__(self, *exc):
        self.stop = True
        self.thread.join()


@pytest.mark.parametrize("cap_mb", [96, 512])
@pytest.mark.parametrize("batch_kernel", [0, 1], ids=["persistent", "level_synchronous"])
def test_graphs_that_exceed_the_cap_together(batch_kernel, cap_mb):
    pytest.importorskip("torch")
    graphs = _graphs()
    with context() as one:
        # (each graph's own solve: ties of the lower bound go by index, so relabelled
        # copies may start their sweeps at different k)
        single = [one.solve(a, want_order=False) for a in graphs]
        tw = [r["tw"] for r in single]
        levels = [one.decide(a, k=t)["stats"]["level_size"] for a, t in zip(graphs[:3], tw)] * 8
    with context(batch_kernel=batch_kernel) as free:
        ref = free.decide_batch(graphs, np.array(tw, np.int32))
    with context(batch_kernel=batch_kernel, mem_cap_bytes=cap_mb * MB) as c:
        with _Lowest() as mem:
            res = c.decide_batch(graphs, np.array(tw, np.int32))
        sol = c.solve_batch(graphs)
    assert res["status"] == 0 and res["yes"].tolist() == [1] * len(graphs)
    for g in range(len(graphs)):
        assert res["level_size"][g][: len(levels[g])].tolist() == levels[g], g
    for key in ("level_size", "fp_sum", "fp_xor"):
        assert np.array_equal(res[key], ref[key]), key
    for key in ("states_expanded", "candidates", "generated", "decide_runs"):
        assert res["stats"][key] == ref["stats"][key], key
    assert sol["status"] == 0 and sol["tw"].tolist() == tw
    assert sol["stats"]["states_expanded"] == sum(r["stats"]["states_expanded"] for r in single)
    pos = 0
    for adj, t in zip(graphs, tw):
        assert oracle.width_elim(adj, sol["orders"][pos: pos + len(adj)].tolist()) == t
        pos += len(adj)
    # (all runs at once keep more than 1 GB; one alone 130 MB with the table, the
    # lists and, while it moves, a second arena)
    used = (mem.first - mem.least) // MB
    assert used <= max(cap_mb, 288) + 32, used
    assert res["stats"]["expand_launches"] > ref["stats"]["expand_launches"]


@pytest.mark.parametrize("cap_mb", [0, 8])
def test_small_graphs_in_the_persistent_kernel(cap_mb):
    # one graph of 16 vertices among larger ones (its runs may hold 2^16 sets, the
    # others' 2^12), and a batch of them under a cap that leaves a block 2^12:
    # graphs that outgrow that go on in the level-synchronous kernel
    mixed = [gg.gnp(16, 0.3, 1)] + [gg.mixed_graph(9100 + j, 17, 28, j % 2 == 0) for j in range(30)]
    small = [gg.gnp(16, 0.15 + 0.01 * j, 60 + j) for j in range(40)]
    with context(mem_cap_bytes=cap_mb * MB) as c:
        for graphs in (mixed, small):
            exp = [oracle.solve(a, want_order=False)["tw"] for a in graphs]
            res = c.solve_batch(graphs)
            assert res["status"] == 0 and res["tw"].tolist() == exp
            pos = 0
            for adj, t in zip(graphs, exp):
                assert oracle.width_elim(adj, res["orders"][pos: pos + len(adj)].tolist()) == t
                pos += len(adj)
