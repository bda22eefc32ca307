"""The coarse correction and first post-smoothing sweep on finest levels of the
sizes that tests/test_gpu_mg_post.py leaves out: 2D levels in two parts (32,768 rows
and more) and unsplit (65,536 and more, where rows without free DOFs are skipped),
3D levels in four (16,384 and more).  FP64 against the numpy restatement of the
preconditioner (bar of tests/test_gpu_precond.py); FP32, whose preconditioner has no
inspection call, by the number of iterations of one solve on levels of those sizes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00671_gb300 import inputs as I
from tests.precond_reference import SchurMG, fixed_stress_diag

pytestmark = pytest.mark.gpu

CASES = {
    "2d-two-parts": (lambda: I.small_footing(seed=7, body=(201, 150), pad=20), 34542, 0),
    "2d-unsplit-void-rows": (lambda: I.small_footing(seed=7, body=(260, 200), pad=60), 68121, 15000),
    "3d-four-parts": (lambda: I.small_block(seed=12, body=(31, 29, 17), pad=2), 19200, 0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_post_sweep_of_large_levels(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm

    make, rows, void = CASES[name]
    w = make()
    nb = w.dim + 1
    sim = mpm.Simulation(w)
    sim.debug_prepare()
    orc = O.Oracle(w)
    assert orc.nn == rows
    prep = orc.prepare(w.dt)
    X = orc.initial_guess(prep)
    _, Jv = orc.eval(prep, X, w.traction(w.dt))
    fixed = orc.fixed_dofs(prep)
    assert np.asarray(fixed).reshape(-1, nb).all(axis=1).sum() >= void
    J = orc.jacobian_matrix(prep, Jv, fixed)
    nn = [w.ncell[k] + 1 for k in range(w.dim)] + [1]
    ref = SchurMG(J, prep["row_ptr"], prep["col"], fixed, nn, w.dim,
                  fs=None if w.dynamic else fixed_stress_diag(w, prep))
    v = np.random.default_rng(1).standard_normal(rows * nb)
    v[fixed] = 0.0
    z, zr = sim.debug_precond(X, v), ref.apply(v)
    assert np.abs(z - zr).max() <= 1e-7 * np.abs(zr).max()
    sim.close()


SOLVES = {
    "2d-two-parts": (lambda: I.terzaghi_column(ncell_x=180, ncell_y=200), 36381),
    "2d-unsplit": (lambda: I.terzaghi_column(ncell_x=260, ncell_y=260), 68121),
    "3d-four-parts": (lambda: I.small_block(seed=12, body=(31, 29, 17), pad=2), 19200),
}


@pytest.mark.parametrize("name", list(SOLVES))
def test_fp32_solve_takes_as_many_iterations(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm

    make, rows = SOLVES[name]
    w = make()
    assert np.prod([c + 1 for c in w.ncell[:w.dim]]) == rows
    its = []
    for precision in (mpm.MPM_FP64, mpm.MPM_MIXED):
        sim = mpm.Simulation(w, precision=precision, newton_rtol=0.5, krylov_rtol=1e-5)
        its.append(sim.step()["krylov_iters"][0])
        sim.close()
    assert abs(its[0] - its[1]) <= 2, its
