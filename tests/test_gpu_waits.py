"""How the library waits for results on the host, in processes of their own (a
pending error belongs to a thread)."""
import pytest

from tests import shim

pytestmark = pytest.mark.gpu

HEAD = """
import time
from paper_1905_00671_gb300 import inputs as I, mpm

cudart = ctypes.CDLL("libcudart.so.13")
w = I.consolidation_block(body=(48, 48, 24), pad=2)
"""

PENDING = HEAD + """
lib = mpm.load()
sim = mpm.Simulation(w)
sim.step()
p = ctypes.c_void_p()
assert cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(1 << 60)) == 2    # left pending
rc = [lib.mpm_step(sim.ctx, ctypes.c_double(w.dt), None, None) for _ in range(3)]
print(rc)
assert rc[1:] == [0, 0], rc
"""


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return shim.build(tmp_path_factory.mktemp("shim"))


def test_a_pending_error_is_reported_once(so):
    """An error that another call of the thread left behind fails one step at most."""
    shim.run(so, PENDING)
