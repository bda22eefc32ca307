"""The coarse correction and first post-smoothing sweep by the set-up's A P, where
its window, split of rows and block layouts change: supports of three and four
nodes per axis, levels split in every number of parts up to sixteen, odd sizes
(last warps and last groups of 32 blocks partly filled), several sweeps and both
block orders, against the numpy restatement of the preconditioner (bar of
tests/test_gpu_precond.py)."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00671_gb300 import inputs as I
from tests.precond_reference import SchurMG, fixed_stress_diag

pytestmark = pytest.mark.gpu


def wide(w):
    return replace(w, lp=np.ascontiguousarray(w.lp * 2.8))


CASES = {
    "2d-four-parts": (lambda: I.small_footing(seed=7, body=(71, 37), pad=2), {}),
    "2d-wide": (lambda: wide(I.small_footing(seed=7, body=(40, 33), pad=2)), {}),
    "2d-orig": (lambda: I.small_footing(seed=8, shape=I.ORIG, body=(63, 31), pad=2), {}),
    "3d-sixteen-parts": (lambda: I.small_block(seed=11, body=(13, 11, 9)), {}),
    "3d-eight-parts": (lambda: I.small_block(seed=12, body=(23, 19, 17)), {}),
    "3d-wide": (lambda: wide(I.small_block(seed=11, body=(11, 9, 7))), {}),
    "3d-wide-v22-upper": (lambda: wide(I.small_block(seed=11, body=(11, 9, 7))), dict(mg_sweeps=2, schur_order=1)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_post_sweep_matches_the_cycle(name):
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
                  fs=None if w.dynamic else fixed_stress_diag(w, prep), sweeps=opts.get("mg_sweeps", 1),
                  lower=opts.get("schur_order", 0) == 0)
    v = np.random.default_rng(1).standard_normal(orc.nn * (w.dim + 1))
    v[fixed] = 0.0
    z, zr = sim.debug_precond(X, v), ref.apply(v)
    assert np.abs(z - zr).max() <= 1e-7 * np.abs(zr).max()
    sim.close()
