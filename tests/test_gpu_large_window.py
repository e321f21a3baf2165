"""Searches whose window is large enough for several champions a node, and
batches whose results come down in several stretches: fronts and paths equal the
oracle's fronts and those of the queries solved alone."""
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


# both sides of the window; one objective to as many as there are (weights of
# one objective, then of all others: two objectives use both); equal costs
@pytest.mark.parametrize("d,cmax", [(1, 9), (2, 9), (2, 2), (3, 40), (4, 1), (5, 5), (8, 3), (16, 2)])
@pytest.mark.parametrize("window", [131071, 131072])
def test_several_champions(op, d, cmax, window):
    g = synth.small_grid(7 * d + cmax, 9 if d > 4 else 14, 8 if d > 4 else 13, d, 0, cmax)
    r = op.opmos_solve(op.opmos_graph.from_synth(g), 0, g.n - 1, window=window, mem_budget_bytes=4 << 30)
    exp = oracle.solve(g, 0, g.n - 1)
    assert np.array_equal(r.costs, exp.costs)
    for c, (nodes, arcs) in zip(r.costs, r.paths):
        assert nodes[0] == 0 and nodes[-1] == g.n - 1
        assert np.array_equal(g.cost[:, arcs.astype(np.int64)].sum(axis=1), c)


# the last pool is longer than two stretches of 8 MiB
@pytest.mark.parametrize("queries,side,d", [(1, 6, 2), (7, 12, 3), (600, 26, 3)])
def test_batch_results_equal_those_solved_alone(op, queries, side, d):
    g = synth.small_grid(side, side, side, d, 1, 30)
    dg = op.opmos_graph.from_synth(g)
    pairs = [(i % 3, g.n - 1 - i % 5) for i in range(queries)]
    alone = {p: op.opmos_solve(dg, *p) for p in set(pairs)}
    words = 0
    batch = op.opmos_solve_batch(dg, [p[0] for p in pairs], [p[1] for p in pairs])
    for (status, r), p in zip(batch, pairs):
        assert status == op.OK
        assert np.array_equal(r.costs, alone[p].costs)
        assert np.array_equal(r.paths.offsets[1:] > r.paths.offsets[:-1], np.ones(len(r.costs), bool))
        for c, (nodes, arcs) in zip(r.costs, r.paths):
            assert nodes[0] == p[0] and nodes[-1] == p[1]
            assert np.array_equal(g.cost[:, arcs.astype(np.int64)].sum(axis=1), c)
        words += r.costs.size + 2 * r.paths.nodes.size
    assert queries < 600 or words > 2 * (2 << 20)
