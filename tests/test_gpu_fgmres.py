"""FGMRES on its less travelled ways."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00671_gb300 import inputs as I
from tests.precond_reference import SchurMG, fixed_stress_diag

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


def tall():
    return [I.terzaghi_column(ncell_y=60, ncell_x=8, h=0.25, k=1e-10, load=10e3),
            I.terzaghi_column(ncell_y=50, ncell_x=9, h=0.25, k=1e-11, load=50e3)]


TIGHT = dict(newton_rtol=1e-13, newton_stag=1e-6, newton_max=12)
# FP64 to the round-off floor; the mixed solve to a Newton tolerance of 1e-11 (bars
# of tests/test_gpu_batch.py)
PRECISION = {0: (dict(TIGHT, krylov_rtol=1e-13, krylov_max=20000), 1e-9),
             1: (dict(newton_rtol=1e-11, newton_max=60), 1e-7)}
# options and the fewest Krylov iterations that show the branch was taken
VARIANTS = {
    "restart-2": (columns, dict(krylov_restart=2), 3),
    "restart-5": (columns, dict(krylov_restart=5), 6),
    # block Jacobi: more columns in a cycle than the triangle's shared memory holds (72)
    "block-jacobi-128": (tall, dict(precond=0, krylov_restart=128), 97),
    "block-jacobi-20": (tall, dict(precond=0, krylov_restart=20), 21),
    # kernels launched one by one: the multigrid's buffers swapped on the host
    "timed": (columns, dict(profile=1023), 3),
    "timed-restart-5-v22-upper": (columns, dict(profile=1023, krylov_restart=5, mg_sweeps=2, schur_order=1), 6),
}


@pytest.fixture(scope="module")
def oracle_steps():
    """u and p after one step of each workload, by name."""
    known = {}

    def of(w):
        key = (w.name, w.ncell, float(w.k[0]))
        if key not in known:
            orc = O.Oracle(w, **TIGHT)
            orc.step()
            known[key] = {f: np.array(orc.state()[f]) for f in ("u", "p")}
        return known[key]
    return of


def assert_close(got, ref, tol, what):
    for f in ("u", "p"):
        r = ref[f].reshape(got[f].shape)
        assert np.abs(got[f] - r).max() <= tol * np.abs(r).max(), (what, f)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["single", "batch"])
@pytest.mark.parametrize("name", list(VARIANTS))
def test_ways_of_the_solve(mpm, oracle_steps, name, kind, precision):
    make, opts, fewest = VARIANTS[name]
    base, tol = PRECISION[precision]
    ws = make()
    opts = dict(base, precision=precision, **opts)
    if kind == "single":
        sim = mpm.Simulation(ws[0], **opts)
        st = sim.step()
        assert_close(sim.read(("u", "p")), oracle_steps(ws[0]), tol, name)
        sim.close()
    else:
        batch = mpm.Batch(ws, **opts)
        st = batch.step()
        for w, got in zip(ws, batch.read(("u", "p"))):
            assert_close(got, oracle_steps(w), tol, (name, w.k[0]))
        batch.close()
    assert st["krylov_total"] >= fewest, st


def first_pass_leaves(w, rtol, m=30):
    """Per column of the first Newton iteration's FGMRES (on the oracle's Jacobian):
    the part of the new vector's norm that the first Gram-Schmidt pass leaves."""
    orc = O.Oracle(w)
    prep = orc.prepare(w.dt)
    R, Jv = orc.eval(prep, orc.initial_guess(prep), w.traction(w.dt))
    fixed = orc.fixed_dofs(prep)
    J = orc.jacobian_matrix(prep, Jv, fixed)
    nn = [c + 1 for c in w.ncell[:w.dim]] + [1]
    M = SchurMG(J, prep["row_ptr"], prep["col"], fixed, nn, w.dim, fs=fixed_stress_diag(w, prep))
    d = np.abs(J.diagonal())
    D = np.where(d > 0, 1 / np.sqrt(np.where(d > 0, d, 1)), 1.0)
    b = -D * np.where(fixed, 0.0, R)
    beta = np.linalg.norm(b)
    V, H, left = [b / beta], np.zeros((m + 1, m)), []
    for j in range(m):
        w0 = D * (J @ (D * M.apply(V[j])))
        B = np.array(V)
        h = B @ w0
        w1 = w0 - B.T @ h
        left.append(np.linalg.norm(w1) / np.linalg.norm(w0))
        h2 = B @ w1
        w2 = w1 - B.T @ h2
        H[:j + 1, j], H[j + 1, j] = h + h2, np.linalg.norm(w2)
        V.append(w2 / H[j + 1, j])
        e = np.zeros(j + 2)
        e[0] = beta
        y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
        if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) <= rtol * beta:
            break
    return left


@pytest.mark.parametrize("opts", [{}, dict(krylov_restart=2), dict(mg_sweeps=2), dict(profile=1023),
                                  dict(profile=1023, mg_sweeps=2, krylov_restart=2)], ids=str)
@pytest.mark.parametrize("k", [1e-9, 1e-8])
def test_second_gram_schmidt_pass(mpm, oracle_steps, k, opts):
    """A column one cell wide, whose preconditioner is almost exact: each product
    returns nearly a vector of the basis, the first pass leaves under 1% of it and
    the host launches the second, with the next iteration already on its way (an
    estimate is a thousandth of the one before)."""
    w = I.terzaghi_column(ncell_y=12, ncell_x=1, h=0.25, k=k, load=10e3)
    left = first_pass_leaves(w, 1e-10)
    assert sum(x < 0.01 for x in left) >= 3, left
    sim = mpm.Simulation(w, **dict(TIGHT, krylov_rtol=1e-10, krylov_max=100, **opts))
    st = sim.step()
    if not opts:
        assert abs(st["krylov_iters"][0] - len(left)) <= 1, (st["krylov_iters"], len(left))
    assert_close(sim.read(("u", "p")), oracle_steps(w), 1e-9, opts)
    sim.close()
