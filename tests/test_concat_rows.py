"""The batched row layout against the per-graph one, over every form that a
graph may have: lists and tuples of ints, numpy rows, more than 64 vertices,
and rows that are no 64-bit words (their other bits are cut off)."""
import numpy as np
import pytest

from paper_1709_09990_gb300 import graphgen as gg

FORMS = {
    "empty": [],
    "lists": [gg.path(5), [0], gg.complete(64), gg.gnp(33, 0.4, 1)],
    "wide": [gg.path(65), gg.path(3), gg.gnp(128, 0.5, 2)],
    "no vertices": [[], gg.path(4)],
    "tuples": [tuple(gg.path(6)), gg.path(2)],
    "numpy": [np.array(gg.path(6), np.uint64), [np.uint64(2), 1]],
    "cut off": [[-1, 3], [1 << 70, 5], gg.path(3)],
}


@pytest.mark.parametrize("form", list(FORMS))
def test_concat_rows(form):
    graphs = FORMS[form]
    rows, ns, offs = gg.concat_rows_u64(graphs)
    assert rows.dtype == np.uint64 and ns.dtype == np.int32 and offs.dtype == np.int64
    assert ns.tolist() == [len(g) for g in graphs] and len(offs) == len(graphs)
    at = 0
    for g, adj in enumerate(graphs):
        each = gg.to_rows_u64(adj).reshape(-1)
        assert offs[g] == at
        assert rows[at: at + len(each)].tolist() == each.tolist()
        at += len(each)
    assert len(rows) == at
