"""The exact solve on the coarsest level where its factorisation and its inverse
change their way: matrices just within and beyond a block's shared memory (167
unknowns in FP64), columns of the inverse in registers up to 96, 192 and 1,024
unknowns.  Grids two nodes wide are their own coarsest level.  Against the numpy
restatement of the preconditioner (bar of tests/test_gpu_precond.py)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00671_gb300 import inputs as I
from tests.precond_reference import SchurMG, fixed_stress_diag

pytestmark = pytest.mark.gpu

# cells along the column -> 4 (cells + 1) displacements, 2 (cells + 1) pressures
CELLS = [23, 24, 40, 41, 47, 48, 96, 255]


@pytest.mark.parametrize("cells", CELLS)
def test_coarsest_level_alone(cells):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm

    w = I.terzaghi_column(ncell_y=cells, ncell_x=1)
    sim = mpm.Simulation(w)
    sim.debug_prepare()
    orc = O.Oracle(w)
    prep = orc.prepare(w.dt)
    X = orc.initial_guess(prep)
    _, Jv = orc.eval(prep, X, w.traction(w.dt))
    fixed = orc.fixed_dofs(prep)
    J = orc.jacobian_matrix(prep, Jv, fixed)
    nn = [w.ncell[0] + 1, w.ncell[1] + 1, 1]
    ref = SchurMG(J, prep["row_ptr"], prep["col"], fixed, nn, 2, fs=fixed_stress_diag(w, prep))
    v = np.random.default_rng(1).standard_normal(orc.nn * 3)
    v[fixed] = 0.0
    z, zr = sim.debug_precond(X, v), ref.apply(v)
    assert np.abs(z - zr).max() <= 1e-7 * np.abs(zr).max()
    sim.close()
