"""Merges split into parts when the list of parts is too short for what every
node asks for: searches of many objectives whose fronts are large. The parts
grow until they fit, so no node with much to compare is left to one warp."""
import hashlib
import os

import numpy as np
import pytest

import oracle
import synth
from pins import check_front_sampled

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def op():
    import paper_2411_16667_gb300 as pkg
    pkg.build()
    from paper_2411_16667_gb300 import opmos
    if opmos.opmos_device_count() == 0:
        pytest.fail("no CUDA device visible to the library")
    return opmos


@pytest.fixture(scope="module")
def grid16():
    g = synth.small_grid(114, 7, 7, 16, 0, 2)
    return g, oracle.solve(g, 0, g.n - 1)


def _no_long_merge_by_one_warp(stats):
    """Per step, the longest merge by one warp takes less time than the longest
    part of a split one: what is split is what has more to compare. (Left out of
    the list it takes all its parts' time: 5 to 30 times as much, measured.)"""
    part, whole = stats["longest_task_ns"][:2]
    assert whole < part


@pytest.mark.parametrize("window", [64, 1024, 16384, 131072])
def test_few_nodes_many_parts(op, grid16, window):
    """50 nodes, frontiers of up to 17,539 labels: every node has more parts to
    do than the places a node would get alike."""
    g, exp = grid16
    r = op.opmos_solve(op.opmos_graph.from_synth(g), 0, g.n - 1, window=window)
    assert np.array_equal(r.costs, exp.costs)
    check_front_sampled(g, 0, g.n - 1, r.costs, r.paths, nrows=200, npaths=200)
    _no_long_merge_by_one_warp(r.stats)


@pytest.mark.parametrize("window", [1024, 4096])
def test_more_asked_for_than_places(op, window):
    """1,153 nodes that ask for up to 128 parts each: more than the list holds."""
    path = os.path.join(os.path.dirname(__file__), "golden", "routes.digests")
    name, _, s, t, count, _, _, digest = next(
        line.split() for line in open(path) if line.startswith("route6x8x24-d12"))
    g, q = synth.time_route(int(name.split("-s")[-1]), 6, 8, 24, 12)
    assert q[0] == (int(s), int(t))
    r = op.opmos_solve(op.opmos_graph.from_synth(g), int(s), int(t), window=window)
    assert len(r.costs) == int(count)
    assert hashlib.sha256(np.ascontiguousarray(r.costs, dtype="<u4").tobytes()).hexdigest()[:16] == digest
    _no_long_merge_by_one_warp(r.stats)
