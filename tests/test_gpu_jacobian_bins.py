"""The staged Jacobian by first-node bins at the sizes where its passes, boxes
and plane ring change: bins of more points than one pass takes, boxes of two
and three nodes per axis, 3D Newmark steps, and a grid whose planes do not all
fit the ring.

Bars as in the entry-wise parity tests: each block entry type within 1e-11
(FP64) or 2e-5 (FP32) of that type's largest entry in the oracle's Jacobian."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00671_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mpm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm as m

    m.load()
    return m


def rel(a, b):
    scale = max(np.abs(b).max(), 1e-300)
    return np.abs(np.asarray(a, dtype=np.float64) - np.asarray(b, dtype=np.float64)).max() / scale


def dynamic(w):
    return replace(w, dynamic=True, dt=1e-3, alpha_vis=0.04, v0=0.01 * np.random.default_rng(2).standard_normal(w.x.shape))


CASES = {
    # 25 (16) points a bin in passes of 4
    "2d-gimp-25ppc": lambda: I.jittered(I.strip_footing(body=(9, 7), pad=2, h=0.25, ppc_axis=5, half_width=0.5), 4),
    "2d-orig-16ppc": lambda: I.jittered(I.strip_footing(body=(9, 7), pad=2, h=0.25, ppc_axis=4, half_width=0.5,
                                                       shape=I.ORIG, dynamic=False, dt=1.0), 5),
    # 27 points a bin in passes of 8
    "3d-gimp-27ppc": lambda: I.jittered(I.consolidation_block(body=(3, 4, 3), h=0.25, ppc_axis=3, patch_half=0.25), 6),
    "3d-orig-27ppc": lambda: I.jittered(I.consolidation_block(body=(3, 4, 3), h=0.25, ppc_axis=3, patch_half=0.25,
                                                             shape=I.ORIG), 7),
    "3d-gimp-newmark": lambda: dynamic(I.small_block(seed=11, body=(5, 4, 3))),
    "3d-gimp-newmark-hencky": lambda: replace(dynamic(I.small_block(seed=12, body=(4, 3, 3))), model=I.MODEL_HENCKY),
}


@pytest.mark.parametrize("name", list(CASES))
def test_jacobian_by_bins_matches_the_oracle(mpm, name):
    w = CASES[name]()
    nb = w.dim + 1
    orc = O.Oracle(w)
    prep = orc.prepare(w.dt)
    rng = np.random.default_rng(3)
    X = orc.initial_guess(prep).reshape(-1, nb)
    X[:, :w.dim] += 1e-5 * rng.standard_normal((orc.nn, w.dim))
    X[:, w.dim] += 1e3 * rng.standard_normal(orc.nn)
    X = X.reshape(-1)
    _, Jo = orc.eval(prep, X, w.traction(w.dt))
    Jo = Jo.reshape(-1, nb, nb)
    sim = mpm.Simulation(w, precision=mpm.MPM_MIXED)
    sim.debug_prepare()
    nnzb = len(prep["col"])
    _, J64 = sim.debug_eval(X, nnzb=nnzb)
    J32 = sim.debug_jacobian32(X, nnzb, 1)
    for J, bar in ((J64, 1e-11), (J32, 2e-5)):
        J = J.reshape(-1, nb, nb)
        for r in range(nb):
            for c in range(nb):
                assert rel(J[:, r, c], Jo[:, r, c]) <= bar, (bar, r, c)
    sim.close()


def test_jacobian_on_a_ring_shorter_than_the_grid(mpm):
    """The FP64 pair sums of 301 planes (8.8 GB) exceed the ring, the FP32 ones
    (4.8 GB) fit: the two assemblies agree to FP32 accuracy."""
    w = I.jittered(I.consolidation_block(body=(20, 20, 299), h=0.25, ppc_axis=1, patch_half=0.5), 9)
    sim = mpm.Simulation(w, precision=mpm.MPM_MIXED)
    sim.debug_prepare()
    _, col = sim.debug_pattern()
    rng = np.random.default_rng(4)
    X = np.zeros((w.nnodes, 4))
    X[:, :3] = 1e-5 * rng.standard_normal((w.nnodes, 3))
    X[:, 3] = 1e3 * rng.standard_normal(w.nnodes)
    X = X.reshape(-1)
    J32 = sim.debug_jacobian32(X, len(col), 1).reshape(-1, 4, 4)
    _, J64 = sim.debug_eval(X, nnzb=len(col))
    J64 = J64.reshape(-1, 4, 4)
    for r in range(4):
        for c in range(4):
            assert rel(J32[:, r, c], J64[:, r, c]) <= 2e-5, (r, c)
    sim.close()
