"""The oracle's tests on byte columns (nine objectives or more, every cost met
below 256) against its tests on the labels themselves: costs times 300 do not fit
a byte and change nothing else, so front, paths and counters must be the same.
Also the turn from one to the other in the middle of a run, and brute force."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from pins import brute_front, check_front


def _scaled(g, by):
    return dataclasses.replace(g, cost=g.cost * np.uint32(by))


def _same(g, by=300):
    a, b = oracle.solve(g, 0, g.n - 1), oracle.solve(_scaled(g, by), 0, g.n - 1)
    assert np.array_equal(a.costs * np.uint32(by), b.costs)
    assert len(a.paths) == len(b.paths)
    for (n0, e0), (n1, e1) in zip(a.paths, b.paths):
        assert np.array_equal(n0, n1) and np.array_equal(e0, e1)
    a.stats.pop("ns"), b.stats.pop("ns")
    assert a.stats == b.stats
    return a


# lists below, at and above the 16 labels of a block; costs of 0 (equal vectors),
# pruned labels, the fewest and the most objectives
@pytest.mark.parametrize("seed,rows,cols,d,cmin,cmax", [
    (1, 1, 3, 9, 0, 2), (2, 3, 3, 9, 0, 1), (3, 4, 4, 16, 0, 2), (4, 5, 4, 9, 0, 3), (5, 5, 5, 10, 0, 1), (6, 4, 5, 12, 1, 9)])
def test_byte_columns_change_nothing(seed, rows, cols, d, cmin, cmax):
    g = synth.small_grid(seed, rows, cols, d, cmin, cmax)
    res = _same(g)
    check_front(g, 0, g.n - 1, res.costs, res.paths)


@pytest.mark.parametrize("seed", range(6))
def test_byte_columns_against_brute_force(seed):
    g = synth.random_digraph(seed, 6 + seed % 3, 9 + seed, p=0.4, cmax=3)
    res = oracle.solve(g, 0, g.n - 1)
    assert [tuple(int(x) for x in r) for r in res.costs] == brute_front(g, 0, g.n - 1)


def test_a_cost_beyond_a_byte_met_late():
    """Path costs pass 255 after several expansions: the search starts over on
    the labels themselves."""
    g = synth.small_grid(8, 5, 5, 9, 40, 90)
    res = _same(g, by=7)
    assert res.costs.max() > 255


def test_large_front_of_sixteen_objectives():
    """17,539 solutions: 3 s on byte columns, 50 s without."""
    g = synth.small_grid(114, 7, 7, 16, 0, 2)
    res = oracle.solve(g, 0, g.n - 1)
    assert len(res.costs) == 17539 and res.stats["labels"] == 171986
    assert res.stats["ns"] < 30e9
