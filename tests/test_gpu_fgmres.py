"""FGMRES on its less travelled ways."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1905_00671_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mpm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm as m

    m.load()
    return m


def columns():
    return [I.terzaghi_column(ncell_y=30, ncell_x=6, h=0.25, k=1e-10, load=10e3),
            I.terzaghi_column(ncell_y=24, ncell_x=8, h=0.25, k=1e-11, load=50e3)]


def test_batch_takes_both_gram_schmidt_passes(mpm):
    """A batch's iteration takes as many kernels in FP64 as in FP32, whose
    iterations always orthogonalise twice.  Kernels per iteration: from two solves
    of one Newton iteration each, to different tolerances."""
    per_iteration = []
    for precision in (mpm.MPM_FP64, mpm.MPM_MIXED):
        runs = []
        for rtol in (1e-2, 1e-5):
            batch = mpm.Batch(columns(), precision=precision, newton_rtol=0.5, krylov_rtol=rtol)
            st = batch.step()
            assert st["newton_iters"] == 1
            runs.append((st["krylov_total"], st["kernel_launches"]))
            batch.close()
        (i0, l0), (i1, l1) = runs
        assert i1 >= i0 + 5
        per_iteration.append((l1 - l0) / (i1 - i0))
    assert per_iteration[0] == per_iteration[1], per_iteration


def overflowing(w):
    """A few points in the middle so stiff that their blocks are infinite in FP32,
    while the residual (and the rows of the loaded surface) stay finite."""
    E = w.E.copy()
    mid = np.argsort(np.abs(w.x - w.x.mean(axis=0)).sum(axis=1))[:4]
    E[mid] = 1e42
    return replace(w, E=E)


@pytest.mark.parametrize("kind", ["single", "batch", "large"])
def test_values_that_are_not_finite_are_an_error(mpm, kind):
    """Not a solution: a rotation formed from NaN would leave an estimate of zero."""
    if kind == "batch":
        ws = columns()
        x = mpm.Batch([ws[0], overflowing(ws[1])], precision=mpm.MPM_MIXED)
    else:
        # ("large": above 2^20 unknowns, where the iterations are not graphs)
        n = (30, 6) if kind == "single" else (592, 592)
        x = mpm.Simulation(overflowing(I.terzaghi_column(ncell_y=n[0], ncell_x=n[1])), precision=mpm.MPM_MIXED)
    with pytest.raises(mpm.MPMError) as e:
        x.step()
    assert e.value.code == -4, e.value          # MPM_ERR_NONFINITE
    assert "FGMRES" in str(e.value)
    x.close()


@pytest.mark.parametrize("rtol", [0.0, -1.0, 1e-320])
def test_a_tolerance_that_nothing_reaches(mpm, rtol):
    """A batch stops at its iteration cap, as a single system does."""
    for x in (mpm.Simulation(columns()[0], krylov_rtol=rtol, krylov_max=150),
              mpm.Batch(columns(), krylov_rtol=rtol, krylov_max=150)):
        with pytest.raises(mpm.MPMError) as e:
            x.step()
        assert e.value.code == -6, e.value      # MPM_ERR_KRYLOV_STAGNATED
        x.close()
