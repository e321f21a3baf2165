"""Counters of opmos_stats are whole numbers of 64 bits: a block adds to words of 32
in shared memory, and what a step adds beyond them is not lost (times and
comparisons of a long step; one phase longer than 4.3 s)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def op():
    import paper_2411_16667_gb300 as pkg
    pkg.build()
    from paper_2411_16667_gb300 import opmos
    if opmos.opmos_device_count() == 0:
        pytest.fail("no CUDA device visible to the library")
    return opmos


@pytest.mark.parametrize("add,steps", [
    ([1], 1), ([0, 5, 7], 3),
    ([2**30 - 1], 9),            # just below what a step's end adds on
    ([2**32 - 1] * 3, 1),        # past the word within a step
    ([2**32 - 1, 1], 5),         # to exactly 2^32
    ([2**31] * 40, 2),           # many times around, by several warps
    ([2**32, 3 * 2**40 + 17], 2),  # one value larger than the word
    ([2**16 - 1, 2**16, 2**16 + 1], 5),  # both sides of what one of its words holds
    ([2**16 - 1] * 80_000, 3),   # as many as fill that one in a step
    (list(range(1, 5000)), 70),
])
def test_nothing_is_lost(op, add, steps):
    assert op.opmos_test_count(np.array(add, np.uint64), steps) == sum(add) * steps
