"""The heuristic by a cluster of blocks (graphs whose distances do not fit one
SM, while there are SMs to spare) and the ways around it, against the oracle's
Dijkstra: shortest distances are whole numbers, so they are equal or wrong."""
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


# the fewest nodes, numbers of nodes that leave blocks one short, the most
# objectives, and both sides of the most nodes whose distances fit 8 blocks
@pytest.mark.parametrize("rows,cols,d", [(44_333, 1, 1), (211, 215, 16), (311, 307, 3), (496, 497, 2), (497, 497, 2)])
def test_sizes(op, rows, cols, d):
    g = synth.small_grid(rows + cols, rows, cols, d, 0, 9)
    goal = (rows // 2) * cols + cols // 3
    got = op.opmos_heur(op.opmos_graph.from_synth(g), goal).copy()
    assert np.array_equal(got, oracle.heuristic(g, goal))


def test_lists_longer_than_their_shared_part(op):
    """Every node has an arc to the goal, half of them below the first threshold."""
    n = 60_001
    arcs = [(u, 0, (1 + 40 * (u % 2), 1 + u % 50)) for u in range(1, n - 3)] + [(n - 2, n - 1, (2, 2))]
    g = synth.from_arcs(n, arcs)
    got = op.opmos_heur(op.opmos_graph.from_synth(g), 0).copy()
    assert np.array_equal(got, oracle.heuristic(g, 0))
    assert (got[:, n - 3:] == 0xFFFFFFFF).all()


def test_one_cluster_a_pair_or_one_block(op):
    """A batch has more pairs than there are clusters: its heuristics come from
    single blocks, a query's own from clusters, and the searches agree."""
    g = synth.small_grid(5, 212, 211, 2, 0, 9)
    dg = op.opmos_graph.from_synth(g)
    goals = np.arange(300, 360, dtype=np.uint32)
    starts = (goals - 2).astype(np.uint32)
    for (status, r), s, t in zip(op.opmos_solve_batch(dg, starts, goals), starts, goals):
        assert status == op.OK and np.array_equal(r.costs, op.opmos_solve(dg, int(s), int(t)).costs)
