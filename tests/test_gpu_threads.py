"""Calls from several threads: each launches kernels that the others launch for
graphs of other sizes."""
import threading

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


def _star(n):
    """Every node has an arc to node 0: a heuristic of two rounds."""
    return synth.from_arcs(n, [(u, 0, (1 + u % 7,)) for u in range(1, n)])


# one kernel (distances in shared memory) with 180 KB and with 16 or 31 KB
@pytest.mark.parametrize("small", [9, 3600])
def test_heuristics_of_two_sizes_side_by_side(op, small):
    """opmos_heuristic_noalloc in one thread beside opmos_heuristic in another:
    only calls of the first have to be kept from overlapping."""
    import torch
    gl, gs = _star(40_000), _star(small)
    L, S = op.opmos_graph.from_synth(gl), op.opmos_graph.from_synth(gs)
    exp_l, exp_s = oracle.heuristic(gl, 0), oracle.heuristic(gs, 0)
    out = torch.empty((1, L.n), dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    failed = []
    stop = threading.Event()

    def small_ones():
        try:
            while not stop.is_set():
                h = op.opmos_heur(S, 0)
            assert np.array_equal(h.copy(), exp_s)
        except Exception as e:  # noqa: BLE001 -- reported by the test
            failed.append(e)

    t = threading.Thread(target=small_ones)
    t.start()
    try:
        for _ in range(5_000):
            op.opmos_heuristic_noalloc(L, 0, 1, out.data_ptr(), stream.cuda_stream)
            if failed:
                break
    finally:
        stop.set()
        t.join()
    assert not failed
    assert np.array_equal(out.cpu().numpy().view(np.uint32), exp_l)
