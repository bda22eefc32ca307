"""mpm_bin_noalloc on points a few of the smallest numbers to the left of the first
face: the correctly rounded quotient is then zero for some, which are inside, and a
negative number for others, which are not."""
import numpy as np
import pytest

from tests.test_gpu_bin_noalloc import env, expected, run  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [1.0, 3.0, 6.0, 10.0, 14.0])
def test_points_just_left_of_the_first_face(env, h):  # noqa: F811
    tiny = np.nextafter(0.0, 1.0)
    xs = -np.arange(0, 40) * tiny
    x = np.stack([xs, np.full_like(xs, 0.5 * h)], axis=1)
    inside, idx = expected((4, 4), h, [0.0, 0.0], x)
    assert inside.any() and not inside.all()
    rc, cell, _ = run(env, (4, 4), h, [0.0, 0.0], x)
    assert rc == -2
    np.testing.assert_array_equal(cell, np.where(inside, idx, -1))
    rc, cell, order = run(env, (4, 4), h, [0.0, 0.0], x[inside])
    assert rc == 0
    np.testing.assert_array_equal(cell, idx[inside])
    np.testing.assert_array_equal(order, np.arange(inside.sum()))
