"""Heuristics of graphs a resident server does not serve. Kernels are loaded at
their first launch, which may wait for an idle device: a server loads those of
every size range before its own kernel starts. Each case is a process of its own,
where nothing has been loaded yet."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# The server is closed after 20 s whatever happens, so a call that waited for its
# end goes on then and the case fails by its time.
PROGRAM = """
import sys, threading, time
import numpy as np
import oracle, synth
from paper_2411_16667_gb300 import opmos as op

g = synth.small_grid(1, 12, 12, 2)
b = synth.small_grid(2, *(int(x) for x in sys.argv[1:3]), 1)
exp = oracle.heuristic(b, 5)
G, B = op.opmos_graph.from_synth(g), op.opmos_graph.from_synth(b)
srv = op.opmos_server([G], op.opmos_default_options(mem_budget_bytes=4 << 30))
guard = threading.Timer(20, srv.close)
guard.start()
t = time.time()
h = op.opmos_heur(B, 5)
took = time.time() - t
guard.cancel()
ticket = srv.submit(0, 2, 0, g.n - 1)
end = time.time() + 20
status, r = srv.poll(ticket)
while status == op.PENDING and time.time() < end:
    status, r = srv.poll(ticket)
srv.close()
assert took < 10, took
assert status == op.OK and np.array_equal(r.costs, oracle.solve(g, 0, g.n - 1).costs)
assert np.array_equal(h.copy(), exp)
print("same")
"""


# distances, then list flags in shared memory, then neither (more than 753,664 nodes)
@pytest.mark.parametrize("rows,cols", [(20, 20), (230, 230), (870, 870)])
def test_heuristic_of_another_size_beside_a_server(rows, cols):
    import paper_2411_16667_gb300 as pkg
    pkg.build()
    run = subprocess.run([sys.executable, "-c", PROGRAM, str(rows), str(cols)], capture_output=True, text=True,
                         timeout=120)
    assert run.returncode == 0 and run.stdout.split() == ["same"], run.stderr
