"""How the library waits for results on the host, in processes of their own (the
way of waiting and a pending error belong to the process and its thread)."""
import pytest

from tests import shim

pytestmark = pytest.mark.gpu

HEAD = """
import time
from paper_1905_00671_gb300 import inputs as I, mpm

cudart = ctypes.CDLL("libcudart.so.13")
w = I.consolidation_block(body=(48, 48, 24), pad=2)
"""

BLOCKING = HEAD + """
assert cudart.cudaSetDeviceFlags(4) == 0        # cudaDeviceScheduleBlockingSync
sim = mpm.Simulation(w)
sim.step()
wall, cpu = time.perf_counter(), time.thread_time()
sim.step()
wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
print("wall", wall, "cpu", cpu)
assert cpu <= 0.5 * wall, (cpu, wall)
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

FAILED_CREATE = HEAD + """
lib = mpm.load()
sim = mpm.Simulation(w)
sim.step()
for spare in (0, 10 ** 6, 10 ** 8, 10 ** 9):
    shim.shim_set_budget(spare)
    try:
        mpm.Simulation(w)
        assert False, spare
    except mpm.MPMError as e:
        assert e.code == -9, e                  # MPM_ERR_NO_MEMORY
    shim.shim_set_budget(-1)
    rc = lib.mpm_step(sim.ctx, ctypes.c_double(w.dt), None, None)
    assert rc == 0, (spare, rc)
"""


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return shim.build(tmp_path_factory.mktemp("shim"))


def test_a_blocking_application_does_not_spin(so):
    """With blocking synchronisation asked of the runtime, the stepping thread sleeps
    for most of a step whose kernels take tens of milliseconds."""
    shim.run(so, BLOCKING)


def test_a_pending_error_is_reported_once(so):
    """An error that another call of the thread left behind fails one step at most."""
    shim.run(so, PENDING)


def test_a_failed_creation_leaves_other_contexts_alone(so):
    """A context that does not fit is refused, and the step of another goes on."""
    shim.run(so, FAILED_CREATE)
