"""The zone's Eq. 4 test in single precision is certain only of what the
double-single test decides.

States near the horizon with g(k, k) set from 1e-9 to 1e-1 of its largest term
off the threshold, on both sides: closer than single precision resolves, and
further.  Close to the horizon the two terms of v = (r^2 + a^2) k^ph - a k^t
cancel to sqrt(Delta) of their size.  The bound on the single-precision error
covers every input, so no decision may differ (no tolerance)."""
import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray

pytestmark = pytest.mark.gpu


def states(rng, n, a, cap_frac, eps):
    """Rows (M, a, eps, y[8]) from cap_frac r_+ outwards, |g(k, k)| about eps
    |g_tt (k^t)^2|: w and v free, k^r from the norm."""
    rp = 1.0 + np.sqrt(1.0 - a * a)
    r = rp * (1.0 + (cap_frac - 1.0) * 10.0 ** rng.uniform(0.0, 2.0, n))
    th = np.where(rng.random(n) < 0.3, 10.0 ** rng.uniform(-6, -1, n), rng.uniform(0.01, np.pi - 0.01, n))
    s2 = np.sin(th) ** 2
    Sigma, P = r * r + a * a * np.cos(th) ** 2, r * r + a * a
    Delta = (r - rp) * (r - (2.0 - rp))
    w = 10.0 ** rng.uniform(-2, 2, n)
    # v and k^th share Delta w^2 with k^r
    f, u = rng.uniform(-1, 1, n), rng.random(n)
    f = np.where(rng.random(n) < 0.3, f * 10.0 ** rng.uniform(-6, 0, n), f)
    v = f * np.sqrt(Delta) * w / np.sqrt(s2)
    kp = (v + a * w) / Sigma
    kt = w + a * s2 * kp
    rest = Delta * w * w * (1 - f * f)
    kh = np.sqrt(u * rest) / Sigma * rng.choice([-1.0, 1.0], n)
    thr = eps * np.abs((1.0 - 2.0 * r / Sigma) * kt * kt)
    off = 10.0 ** rng.uniform(-9, -1, n) * rng.choice([-1.0, 1.0], n) * np.maximum(thr, Delta * w * w / Sigma)
    norm = rng.choice([-1.0, 1.0], n) * (thr + off)
    kr2 = Delta / Sigma * (norm + (Delta * w * w - s2 * v * v) / Sigma - Sigma * kh * kh)
    ok = kr2 > 0
    kr = -np.sqrt(np.where(ok, kr2, 1.0))
    z = np.zeros(n)
    rows = np.stack([z + 1.0, z + a, z + eps, z, r, th, z, kt, kr, kh, kp], axis=1)
    return rows[ok]


@pytest.mark.parametrize("a", [0.0, 0.5, 0.9, 0.998, 0.99999, -0.9999999])
@pytest.mark.parametrize("cap_frac, eps", [(1.01, 1e-3), (1.001, 1e-4), (1.00001, 1e-3), (1.00001, 1e-5),
                                           (1.0000001, 1e-6), (1.5, 1e-2)])
def test_certain_decisions_are_the_double_single_ones(a, cap_frac, eps):
    rng = np.random.default_rng(7)
    rows = states(rng, 400000, a, cap_frac, eps)
    out = gray.gray_eval(gray.EVAL_XI_ZONE, gray.FP32, torch.from_numpy(rows).cuda()).cpu().numpy()
    fails, certain, want = out[:, 0] == 1, out[:, 1] == 1, out[:, 2] == 1
    assert len(rows) > 50000 and 0 < want.sum() < len(rows)
    wrong = certain & (fails != want)
    assert not wrong.any(), (wrong.sum(), certain.mean(), rows[wrong][:3])
    assert certain.any()  # the single-precision test does decide


def test_values_without_a_decision_go_to_the_double_single_test():
    """NaN, infinite and underflowing momenta are never decided in single
    precision."""
    row = np.array([1.0, 0.9, 1e-3, 0.0, 1.46, 1.0, 0.0, 3.0, -1.0, 0.1, 0.5])
    rows = np.stack([row] * 8)
    for k, (slot, x) in enumerate([(7, np.nan), (8, np.nan), (9, np.inf), (10, -np.inf), (7, 1e30), (8, 1e25)]):
        rows[k, slot] = x
    rows[6, 7:] *= 1e-25
    rows[7, 4] = 1.0 + np.sqrt(1.0 - 0.81)  # on the horizon: Delta = 0 or a rounding
    out = gray.gray_eval(gray.EVAL_XI_ZONE, gray.FP32, torch.from_numpy(rows).cuda()).cpu().numpy()
    wrong = (out[:, 1] == 1) & (out[:, 0] != out[:, 2])
    assert not wrong.any() and np.all(out[:4, 1] == 0) and out[6, 1] == 0
