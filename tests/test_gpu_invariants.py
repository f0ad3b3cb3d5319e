"""GRAY_RENDER_INVARIANTS divides, where a product with a reciprocal rounds twice
and overflows below the normal range."""
import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def invariants(image, r, theta, k):
    """Invariants of FP64 states written into the position and momentum planes
    (32 bytes per ray each, planes on 256-byte boundaries)."""
    n = image.n
    tr = gray.Tracer(gray.Options(precision=gray.FP64), n)
    tr.setup([image])
    planes = tr.state.view(torch.float64)
    X = planes[:4 * n].view(n, 4)
    first = (32 * n + 255) // 256 * 32
    K = planes[first:first + 4 * n].view(n, 4)
    X[:, 1] = torch.as_tensor(r, dtype=torch.float64, device=X.device)
    X[:, 2] = torch.as_tensor(theta, dtype=torch.float64, device=X.device)
    K[:] = torch.as_tensor(k, dtype=torch.float64, device=X.device)
    inv = tr.invariants()
    tr.close()
    return inv


def test_null_norm_of_a_radial_ray_in_flat_space_is_zero():
    """Sigma and Delta are both r^2 rounded, so g_rr = 1 and the norm of k =
    (5/4, 5/4, 0, 0) is exactly zero at every radius."""
    im = I.Image(a=0.0, M=0.0, incl=1.0, nx=4096, ny=1)
    r = np.random.default_rng(3).uniform(2.0, 1000.0, im.n)
    inv = invariants(im, r, 1.0, [1.25, 1.25, 0.0, 0.0])
    assert np.all(inv[:, 3] == 0.0)
    assert np.all(inv[:, 0] == 1.25) and np.all(inv[:, 1] == 0.0)


@pytest.mark.parametrize("theta", [1e-150, 1e-160, 1e-161, np.pi])
def test_carter_constant_next_to_the_pole(theta):
    """sin^2 below the normal range divides like any other: Q = -a^2 E^2 there,
    with L_z^2 / sin^2 a product of sin^2 and far below its rounding."""
    a = 0.5
    im = I.Image(a=a, incl=1.0, nx=3, ny=1)
    inv = invariants(im, 10.0, theta, [1.0, -1.0, 0.0, 0.1])
    # |L_z| < 12 sin^2, so L_z^2 / sin^2 < 144 sin^2 <= 3e-30; E, a^2 E^2 and cos^2
    # round six times
    want = -a * a * inv[:, 0] ** 2
    assert np.all(np.abs(inv[:, 2] - want) <= 6 * 2.0 ** -53 * np.abs(want) + 144 * np.sin(theta) ** 2)
