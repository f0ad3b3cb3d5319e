"""Initial states in single precision are the double ones rounded to a pair.

The split of a double into its nearest float and the rounded remainder runs on
the integer pipe inside 2^-60 .. 2^61 and on the conversion instructions
outside; both round to nearest, so the stored pair is exactly numpy's."""
import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def states(rays, precision):
    tr = gray.Tracer(gray.Options(precision=precision, r_sw=0.02), rays.shape[0])
    tr.setup_rays(torch.from_numpy(rays).cuda())
    rec = tr.records()
    tr.close()
    return rec


@pytest.mark.parametrize("r_obs", [10.0, 1000.0, 1e15, 1e25])
@pytest.mark.parametrize("precision", ["fp32", "fp32_kahan", "fp32_kahan_sel64"])
def test_initial_pairs_are_the_rounded_doubles(precision, r_obs):
    rays = I.mixed_rays(5000, offset=123)
    rays[:, 4] = r_obs
    # exact zeros, values below and across both ends of the integer path
    rays[:40, 0] = np.repeat([0.0, -0.0, 1e-300, -1e-30, 2.0 ** -59, 2.0 ** -61, 2.0 ** -23, 1.0], 5)
    rays[40:80, 1] = np.repeat([0.0, 1e-300, 1e-30, 2.0 ** -60], 10)
    rays[80:90, 2] = 0.0
    y = states(rays, gray.FP64)[:, 8:16]
    got = states(rays, gray.PRECISIONS[precision])
    hi = y.astype(np.float32)
    lo = (hi.astype(np.float64) - y).astype(np.float32) if precision != "fp32" else np.zeros_like(hi)
    assert np.array_equal(got[:, 8:16], hi.astype(np.float64) - lo.astype(np.float64))
    assert np.array_equal(got[:, 4:8], hi[:, :4].astype(np.float64))
    assert np.all(got[:, :4] == 0) and np.all(got[:, 16] == 0)


def test_single_rays_keep_the_constants_of_images_bit_for_bit():
    """A ray set up by itself stores the same constants as a one-pixel image with
    its hole: spin, mass, distance and the spin's and mass's low words (a zero
    low word is +0)."""
    spins = [0.0, 0.5, -0.5, 0.3, -0.3, 0.9, 0.998, 1e-9]
    n = len(spins)
    images = [I.Image(a=a, incl=1.0, nx=1, ny=1, alpha0=2.0, alpha1=4.0, beta0=1.0, beta1=3.0) for a in spins]
    rays = torch.tensor([[3.0, 2.0, a, 1.0, images[0].r_obs] for a in spins], dtype=torch.float64, device="cuda")
    plane = (32 * n + 255) // 256 * 256  # FP64: position, momentum, final point, constants
    stored = []
    for lone in (False, True):
        tr = gray.Tracer(gray.Options(precision=gray.FP64), n)
        tr.setup_rays(rays) if lone else tr.setup(images)
        stored.append(tr.state[3 * plane:3 * plane + 32 * n].cpu().numpy())
        tr.close()
    assert np.array_equal(stored[0], stored[1])
