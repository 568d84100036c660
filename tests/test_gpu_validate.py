"""Graphs that are refused: a loop, an edge without its mirror (above or below
the diagonal), a bit past the last vertex; at the edges of the row words."""
import numpy as np
import pytest

from paper_1709_09990_gb300 import graphgen as gg
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 128])
def test_refused_graphs(n):
    from paper_1709_09990_gb300 import native
    good = gg.to_rows_u64(gg.gnp(n, 0.4, n))

    def flipped(*bits):
        rows = good.copy()
        for r, c in bits:
            rows[r, c // 64] ^= np.uint64(1 << (c % 64))
        return rows

    W = good.shape[1]
    bad = [flipped((0, 0)), flipped((n - 1, n - 1))]
    if n > 1:
        bad += [flipped((0, n - 1)), flipped((n - 1, 0))]
    if n > 3:
        # as many bits above the diagonal as below, but not each other's mirrors
        a = [(0, 2), (3, 1)] if not (int(good[0, 0]) >> 2) & 1 and not (int(good[3, 0]) >> 1) & 1 else None
        bad += [flipped(*a)] if a else []
    if n < 64 * W:
        bad += [flipped((0, n)), flipped((n - 1, 64 * W - 1))]
    with context() as ctx:
        ctx.bounds(good)
        assert ctx.features([[int(r[0]) | (int(r[-1]) << 64 if W > 1 else 0) for r in good]]).shape == (1, 12)
        for rows in bad:
            with pytest.raises(native.TwError) as e:
                ctx.bounds(rows)
            assert e.value.status == native.TW_ERR_INVALID
