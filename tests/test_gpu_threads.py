"""Contexts of several host threads at the same time: a small column, whose
multigrid tails take 13 KB of shared memory, and a footing whose tails take
60, each stepped in a thread of its own, must give what they give alone.  The
call that sets a kernel's shared-memory limit is made slow, so that one thread's
limit, were it its own, would still be set when the other launches."""
import pytest

from tests import shim

pytestmark = pytest.mark.gpu

PROGRAM = """
import threading
import numpy as np
from paper_1905_00671_gb300 import inputs as I, mpm

MAKE = [lambda: I.terzaghi_column(ncell_y=20, ncell_x=4), lambda: I.small_footing(seed=7, body=(60, 28), pad=2)]
CONTEXTS = 15

def steps(w):
    sim = mpm.Simulation(w)
    for _ in range(2):
        sim.step()
    out = sim.read(("x", "u", "p"))
    sim.close()
    return out

works = [m() for m in MAKE]
alone = [steps(w) for w in works]
got = [[], []]

def work(i, more):
    try:
        while more():
            got[i].append(steps(works[i]))
    except Exception as e:
        got[i].append(e)

footing = threading.Thread(target=work, args=(1, lambda: len(got[1]) < CONTEXTS))
column = threading.Thread(target=work, args=(0, lambda: footing.is_alive()))
footing.start()
column.start()
footing.join()
column.join()
assert got[0] and got[1]
for a, runs in zip(alone, got):
    for g in runs:
        assert not isinstance(g, Exception), g
        for f in a:
            np.testing.assert_array_equal(a[f], g[f])
"""


def test_two_threads_step_as_one(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shim.run(shim.build(tmp_path), PROGRAM, SHIM_ATTR_SLEEP_US=2000)
