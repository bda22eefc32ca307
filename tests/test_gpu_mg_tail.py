"""The multigrid cycle's coarse levels as one dense operator, at the sizes where
its first level changes: the finest level itself, the first coarse level just
within and just beyond the limit of 1,024 unknowns, in 2D and 3D, against the
numpy restatement of the preconditioner (bar of tests/test_gpu_precond.py)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00671_gb300 import inputs as I
from tests.precond_reference import SchurMG, fixed_stress_diag

pytestmark = pytest.mark.gpu

# cells incl. pad rows -> nodes of the first coarse level x components
CASES = {
    "2d-finest": (lambda: I.small_footing(seed=7, body=(18, 10), pad=2), {}),           # 19 x 13 x 2 = 494
    "2d-within": (lambda: I.small_footing(seed=7, body=(60, 28), pad=2), {}),           # 31 x 16 x 2 = 992
    "2d-beyond": (lambda: I.small_footing(seed=7, body=(64, 28), pad=2), {}),           # 33 x 16 x 2 = 1056
    "2d-within-v33": (lambda: I.small_footing(seed=7, body=(60, 28), pad=2), dict(mg_sweeps=3)),
    "3d-within": (lambda: I.small_block(seed=11, body=(14, 12, 9)), {}),                # 8 x 7 x 6 x 3 = 1008
    "3d-beyond": (lambda: I.small_block(seed=11, body=(14, 12, 11)), {}),               # 8 x 7 x 7 x 3 = 1176
}


@pytest.mark.parametrize("name", list(CASES))
def test_tail_operator_matches_the_cycle(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm

    make, opts = CASES[name]
    w = make()
    sim = mpm.Simulation(w, **opts)
    sim.debug_prepare()
    orc = O.Oracle(w)
    prep = orc.prepare(w.dt)
    X = orc.initial_guess(prep)
    _, Jv = orc.eval(prep, X, w.traction(w.dt))
    fixed = orc.fixed_dofs(prep)
    J = orc.jacobian_matrix(prep, Jv, fixed)
    nn = [w.ncell[k] + 1 for k in range(w.dim)] + [1]
    ref = SchurMG(J, prep["row_ptr"], prep["col"], fixed, nn, w.dim,
                  fs=None if w.dynamic else fixed_stress_diag(w, prep), sweeps=opts.get("mg_sweeps", 1))
    v = np.random.default_rng(1).standard_normal(orc.nn * (w.dim + 1))
    v[fixed] = 0.0
    z, zr = sim.debug_precond(X, v), ref.apply(v)
    assert np.abs(z - zr).max() <= 1e-7 * np.abs(zr).max()
    sim.close()
