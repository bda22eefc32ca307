"""mpm_bin_noalloc where its kernels change their way: cells of 1 to 8 points
(ranked by 8 lanes) and of more (sorted in place), grids around whole blocks of
the scan, points on the faces between cells, where a floor taken from a
reciprocal has to give way to the division.  Cells and orders are whole numbers
and must be those of NumPy's correctly rounded division exactly."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_00671_gb300 import mpm

    lib = mpm.load()
    lib.mpm_bin_noalloc.argtypes = [C.POINTER(mpm.mpm_grid), C.c_int64, C.c_void_p, C.c_void_p,
                                    C.c_void_p, C.c_void_p]
    lib.mpm_bin_noalloc.restype = C.c_int
    return torch, mpm, lib


def run(env, ncell, h, origin, x):
    torch, mpm, lib = env
    g = mpm.mpm_grid()
    g.dim = len(ncell)
    for k in range(g.dim):
        g.ncell[k], g.origin[k] = ncell[k], origin[k]
    g.h = h
    n = x.shape[0]
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    cell = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    order = torch.full((n,), -7, dtype=torch.int64, device="cuda")
    rc = lib.mpm_bin_noalloc(C.byref(g), n, xd.data_ptr(), cell.data_ptr(), order.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
    return rc, cell.cpu().numpy(), order.cpu().numpy()


def expected(ncell, h, origin, x):
    c = np.floor((x - np.asarray(origin)) / h).astype(np.int64)
    inside = ((c >= 0) & (c < np.asarray(ncell))).all(axis=1)
    idx = c[:, 0]
    stride = 1
    for k in range(1, len(ncell)):
        stride *= ncell[k - 1]
        idx = idx + stride * c[:, k]
    return inside, idx


GRIDS = [((1, 1), 1), ((1, 1), 9), ((1, 1), 3000), ((64, 64), 4), ((4095, 1), 1), ((4097, 1), 2),
         ((200, 102), 4), ((512, 512), 1), ((16, 16, 16), 8), ((17, 16, 16), 9), ((64, 64, 64), 1)]


@pytest.mark.parametrize("ncell,ppc", GRIDS)
def test_cells_and_order(env, ncell, ppc):
    rng = np.random.default_rng(5)
    h, origin = 0.1, [-0.3] * len(ncell)
    n = ppc * int(np.prod(ncell))
    x = np.asarray(origin) + h * rng.random((n, len(ncell))) * np.asarray(ncell)
    inside, idx = expected(ncell, h, origin, x)
    x, idx = x[inside], idx[inside]
    rc, cell, order = run(env, ncell, h, origin, x)
    assert rc == 0
    np.testing.assert_array_equal(cell, idx)
    np.testing.assert_array_equal(order, np.argsort(idx, kind="stable"))


@pytest.mark.parametrize("h,origin", [(0.1, 0.0), (1.0 / 3.0, -0.7), (0.025, 1e3), (3e-7, 0.0)])
def test_points_on_the_faces(env, h, origin):
    """Coordinates at every face, and up to two representable numbers to either
    side of it; the point left of the first face is outside."""
    nc = 4000
    f = origin + h * np.arange(nc)
    lo1, hi1 = np.nextafter(f, -np.inf), np.nextafter(f, np.inf)
    xs = np.concatenate([f, lo1, hi1, np.nextafter(lo1, -np.inf), np.nextafter(hi1, np.inf)])
    x = np.stack([xs, np.full_like(xs, origin + 0.5 * h)], axis=1)
    ncell, org = (nc, 2), [origin, origin]
    inside, idx = expected(ncell, h, org, x)
    assert not inside.all()
    rc, cell, order = run(env, ncell, h, org, x)
    assert rc == -2
    np.testing.assert_array_equal(cell, np.where(inside, idx, -1))
    assert (order == -7).all()                      # nothing ordered after an error
    x, idx = x[inside], idx[inside]
    rc, cell, order = run(env, ncell, h, org, x)
    assert rc == 0
    np.testing.assert_array_equal(cell, idx)
    np.testing.assert_array_equal(order, np.argsort(idx, kind="stable"))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e300])
def test_values_outside_any_grid(env, bad):
    x = np.full((3, 2), 0.5)
    x[1, 0] = bad
    rc, cell, order = run(env, (4, 4), 1.0, [0.0, 0.0], x)
    assert rc == -2
    np.testing.assert_array_equal(cell, [0, -1, 0])
    assert (order == -7).all()
