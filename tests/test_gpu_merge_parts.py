"""Merges split into as many parts as a search makes: 1 to 128 warps side by side.
A part is a share of the candidates (whole groups of 32, or 4 to 16 lanes of one)
times a range of what they are compared with -- the frontier, the node's
candidates, P. The result must be the host's merge whatever the split; searches
whose nodes take all 128 parts, P among what is divided, must give the oracle's
front."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_kernels import _antichain, _reference

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def op():
    import paper_2411_16667_gb300 as pkg
    pkg.build()
    from paper_2411_16667_gb300 import opmos
    if opmos.opmos_device_count() == 0:
        pytest.fail("no CUDA device visible to the library")
    return opmos


# parts: shares only (1 to 8), then 2 to 16 ranges; candidates: one group of 32, two,
# some that leave a part's lanes empty, many in slots and lists; frontiers of fewer
# entries than ranges, and of several rounds a range
@pytest.mark.parametrize("parts", [1, 2, 4, 8, 16, 32, 64, 128])
@pytest.mark.parametrize("d,nf,nc,slots,lists", [
    (3, 0, 20, 32, 32), (2, 5, 32, 32, 1), (3, 300, 7, 128, 32), (5, 4000, 30, 128, 8), (4, 200, 33, 32, 32),
    (8, 90, 64, 128, 32), (3, 3000, 1000, 128, 32), (12, 60, 500, 64, 8), (16, 700, 100, 45, 8), (1, 1, 40, 60, 8),
    # removed entries: frontiers of one round of the compaction, one more, many; one candidate alone
    (3, 256, 40, 128, 32), (3, 257, 40, 128, 32), (4, 255, 9, 128, 32), (3, 3000, 1, 128, 32), (5, 2500, 3, 60, 8)])
def test_any_number_of_parts(op, parts, d, nf, nc, slots, lists):
    rng = np.random.default_rng(parts + 1000 * nf + nc + d)
    hi = 40 if nf < 400 else 400
    front = _antichain(rng, nf, d, hi) if nf else np.zeros((0, d), np.uint32)
    nf = len(front)
    cand = rng.integers(0, hi, size=(nc, d)).astype(np.uint32)
    if nf:  # some equal entries of the frontier, some just worse, some just better
        third = nc // 3
        pick = front[rng.integers(0, nf, size=third)].astype(np.int64)
        cand[:third] = np.maximum(pick + rng.integers(-1, 2, size=(third, 1)), 0)
    cand[-2:] = cand[0]  # equal candidates: the smallest arc wins
    arc = rng.permutation(10 * nc)[:nc].astype(np.uint32)
    costs, origin = op.opmos_test_merge(front, cand, arc, parts, slots, lists)
    got = sorted((tuple(int(v) for v in c), int(o)) for c, o in zip(costs, origin))
    assert got == _reference(front, cand, arc)


def test_parts_beyond_the_most(op):
    front, cand = np.zeros((0, 2), np.uint32), np.ones((3, 2), np.uint32)
    with pytest.raises(op.OpmosError) as e:
        op.opmos_test_merge(front, cand, np.arange(3), 129)
    assert e.value.code == op.ERR_INVALID_ARG


def test_lists_of_parts_that_fill_in_a_batch(op):
    """43 nodes of a batched query ask for up to 5,504 parts; its list holds 2,048."""
    g = synth.small_grid(3, 7, 6, 14, 0, 2)
    goals = [g.n - 1, g.n - 2]
    exp = {t: oracle.solve(g, 0, t).costs for t in goals}
    out = op.opmos_solve_batch(op.opmos_graph.from_synth(g), [0] * 4, goals * 2, window=1024,
                               mem_budget_bytes=16 << 30, alone_labels=1 << 40)
    for (status, r), t in zip(out, goals * 2):
        assert status == op.OK and np.array_equal(r.costs, exp[t])
