"""Steps where device memory is short: the sums by first-node bins make the
residual and the Jacobian faster, and a step must do without them before it fails
for want of memory.  The thin block's ring of three bin planes (0.3 GB) is larger
than the records of the per-pair kernel."""
import pytest

from tests import shim

pytestmark = pytest.mark.gpu

PROGRAM = """
import numpy as np
from paper_1905_00671_gb300 import inputs as I, mpm

precision, extra = {precision}, {extra}
w = I.small_block(seed=11, body=(40, 40, 2), pad=5)

def step():
    base = shim.shim_used()
    sim = mpm.Simulation(w, precision=precision)
    st = sim.step()
    out = sim.read(("u", "p")), shim.shim_used() - base, sim.stats()
    sim.close()
    return out

ref, used, st = step()
nn = [c + 1 for c in w.ncell]
nodes, plane, word = nn[0] * nn[1] * nn[2], nn[0] * nn[1], 4 if precision else 8
pair = 378 * (24 if precision else 22) * word     # values of a bin's pairs, padded to 16 bytes
ring, bins = nodes * (pair + 4), nodes * (27 * 4 * 8 + 4)
records = ((st["jac_point_nodes"] + len(w.x)) * 1.25 + 1024) * 22 * 8 if not precision else 0
others = used - ring - bins
assert records < 0.8 * 3 * plane * pair, (records, 3 * plane * pair)
assert others > 0
shim.shim_set_budget(int(others + eval(extra)))
got, _, st = step()
print("refused", shim.shim_refused(), "config", st["jac_config"])
assert shim.shim_refused() > 0
for f in ref:
    assert np.abs(got[f] - ref[f]).max() <= 1e-8 * np.abs(ref[f]).max(), f
"""

# what is left beside the buffers that a step cannot do without
CASES = {
    "fp64-no-room-for-three-planes": (0, "bins + 0.9 * 3 * plane * pair"),
    "fp64-bins-give-way": (0, "records + 0.4 * bins"),
    "mixed-bins-give-way": (1, "0.6 * bins"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_a_step_does_without_the_bins(name, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    precision, extra = CASES[name]
    shim.run(shim.build(tmp_path), PROGRAM.format(precision=precision, extra=repr(extra)))


WIDE = """
from dataclasses import replace
import numpy as np
from paper_1905_00671_gb300 import inputs as I, mpm

w = I.small_block(seed=11, body=(11, 9, 7))
w = replace(w, lp=np.ascontiguousarray(w.lp * 2.8))        # supports of four nodes

def step():
    base = shim.shim_used()
    sim = mpm.Simulation(w, precision=mpm.MPM_MIXED, newton_rtol=1e-6, newton_max=60)
    sim.step()
    out = sim.read(("u", "p")), shim.shim_used() - base, sim.stats()
    sim.close()
    return out

ref, used, st = step()
assert st["jac_config"][1] >= 1000, st["jac_config"]       # staged
staging = int(((st["jac_point_nodes"] + len(w.x)) * 1.25 + 1024) * 24 * 4)
shim.shim_set_budget(used - staging + int({extra}))
sim = mpm.Simulation(w, precision=mpm.MPM_MIXED, newton_rtol=1e-6, newton_max=60)
sim.step()
got, st = sim.read(("u", "p")), sim.stats()
assert shim.shim_refused() > 0
assert st["jac_config"][1] < 1000, st["jac_config"]        # per term
for f in ref:
    assert np.abs(got[f] - ref[f]).max() <= 1e-5 * np.abs(ref[f]).max(), f
shim.shim_set_budget(-1)
sim.step()
assert sim.stats()["jac_config"][1] >= 1000                # staged again
sim.close()
"""


# room for half of the records, or for nothing beside what the step cannot do without
@pytest.mark.parametrize("extra", ["staging / 2", "1024"])
def test_a_mixed_step_does_without_the_staging(extra, tmp_path):
    """Supports of four nodes in the mixed mode: the staged records give way to the
    preconditioner's buffers, the wide A P takes the narrow one's place, and the form
    that needs no records serves (both forms to the Newton tolerance of 1e-6)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shim.run(shim.build(tmp_path), WIDE.format(extra=extra))
