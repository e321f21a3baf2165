"""The test against P goes through the index of P (tiles whose minima do not
dominate are passed over) at every number of objectives: on a large front it
takes less than half the comparisons of every label with every solution.
Without the index it takes three quarters and more of them."""
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


@pytest.mark.parametrize("seed,rows,cols,d,cmax", [(114, 7, 7, 16, 2), (3, 8, 7, 14, 3)])
def test_many_objectives_use_the_index(op, seed, rows, cols, d, cmax):
    g = synth.small_grid(seed, rows, cols, d, 0, cmax)
    r = op.opmos_solve(op.opmos_graph.from_synth(g), 0, g.n - 1, window=1024)
    assert np.array_equal(r.costs, oracle.solve(g, 0, g.n - 1).costs)
    assert 2 * r.stats["p_cmp"] < r.stats["inserted"] * len(r.costs)
