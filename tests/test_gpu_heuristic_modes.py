"""The heuristic kernel at the edges of its three ways to keep distances and
list flags (all in shared memory, flags in shared memory, all in global
memory), against the oracle's Dijkstra: shortest distances are whole numbers,
so they are equal or wrong."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def op():
    import paper_2411_16667_gb300 as pkg
    pkg.build()
    from paper_2411_16667_gb300 import opmos
    if opmos.opmos_device_count() == 0:
        pytest.fail("no CUDA device visible to the library")
    return opmos


# 44,332 nodes are the most whose distances fit; 753,664 the most whose flags do
@pytest.mark.parametrize("rows,cols,d", [(1, 1, 1), (1, 2, 2), (31, 1, 1), (33, 65, 3), (211, 210, 2), (212, 211, 2),
                                         (868, 868, 1), (869, 869, 1)])
def test_heuristic_of_every_mode(op, rows, cols, d):
    g = synth.small_grid(rows + cols, rows, cols, d, 0, 9)
    goal = (rows // 2) * cols + cols // 3
    got = op.opmos_heur(op.opmos_graph.from_synth(g), goal).copy()
    assert np.array_equal(got, oracle.heuristic(g, goal))


def test_unreachable_nodes_and_many_arcs_into_one(op):
    """A goal every other node has an arc to (one node's arcs take many rounds
    of its lanes), and nodes nothing leads to it from."""
    n = 3000
    arcs = [(u, 0, (1 + u % 7,)) for u in range(1, n - 5)] + [(0, n - 1, (3,)), (n - 2, n - 1, (2,))]
    g = synth.from_arcs(n, arcs)
    got = op.opmos_heur(op.opmos_graph.from_synth(g), 0).copy()
    assert np.array_equal(got, oracle.heuristic(g, 0))
    assert (got[0, n - 5:] == 0xFFFFFFFF).all()
