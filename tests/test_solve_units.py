"""The triangular solve's DAG does not grow as the leaf clusters shrink: its
units are half a tile, whatever the leaf size (no GPU)."""
import numpy as np
import pytest

from test_schedule_hazards import SOLVE, _check, _trees, lib  # noqa: F401


@pytest.mark.parametrize("n,tile", [(6, 64), (5, 32)])
def test_edges_do_not_grow_with_smaller_leaves(lib, n, tile):  # noqa: F811
    edges = {}
    for leaf in (2, 4, 8, tile // 2):
        st, rep = _check(lib, _trees(n, leaf), SOLVE, rank_cap=64, tile=tile)
        assert st == 0 and rep[3] == 0, rep
        edges[leaf] = int(rep[9])
    # clusters of at most half a tile lie between a quarter and a half tile at
    # every leaf size: the same units, the same edges up to where leaves end early
    assert max(edges.values()) <= 1.5 * edges[tile // 2], edges
