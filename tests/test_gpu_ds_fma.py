"""The zone's double-single product-sum is as exact as a product and a sum.

The rms error of x y + z over |x y| + |z| must not pass that of the normalised
product followed by the sum on the same operands, for terms of like size, of
unlike sizes and cancelling ones; and no error passes 9 u^2 of |x y| + |z|, u =
2^-24: the product loses 2 and 3 u^2 |x y| in its low word's two additions and
u^2 |x y| with the product of the low words, the sum u^2 and 2 u^2 of |x y| + |z|
in its two."""
import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray

pytestmark = pytest.mark.gpu


def two_product(a, b):
    """a b as an unevaluated sum of two doubles (Dekker's splitting)."""
    def split(x):
        t = 134217729.0 * x
        h = t - (t - x)
        return h, x - h
    p = a * b
    ah, al = split(a)
    bh, bl = split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def pair(x):
    hi = x.astype(np.float32).astype(np.float64)
    lo = (x - hi).astype(np.float32).astype(np.float64)
    return hi + lo


@pytest.mark.parametrize("kind", ["like", "unlike", "small_z", "large_z", "cancel", "cancel_deep"])
def test_product_sum_is_as_exact_as_product_and_sum(kind):
    rng = np.random.default_rng(11)
    n = 1 << 20
    x, y = (rng.uniform(1, 2, n) * rng.choice([-1.0, 1.0], n) for _ in range(2))
    z = rng.uniform(1, 2, n) * rng.choice([-1.0, 1.0], n)
    if kind == "unlike":
        z *= 2.0 ** rng.integers(-6, 7, n)
    elif kind == "small_z":
        z *= 2.0 ** -rng.integers(8, 20, n)
    elif kind == "large_z":
        z *= 2.0 ** rng.integers(8, 20, n)
    elif kind == "cancel":
        z = -x * y * (1 + 2.0 ** -rng.integers(2, 12, n))
    elif kind == "cancel_deep":
        z = -x * y * (1 + 2.0 ** -rng.integers(12, 32, n))
    x, y, z = pair(x), pair(y), pair(z)
    out = gray.gray_eval(gray.EVAL_FMA_DS, gray.FP32,
                         torch.from_numpy(np.stack([x, y, z], axis=1)).cuda()).cpu().numpy()
    p, pe = two_product(x, y)
    scale = np.abs(p) + np.abs(z)

    def error(hi, lo):
        # every term is a double; p + z and hi cancel before the rest is added
        s = p + z
        bb = s - p
        se = (p - (s - bb)) + (z - bb)
        return ((s - hi) + se + pe - lo) / scale
    fma, two = error(out[:, 0], out[:, 1]), error(out[:, 2], out[:, 3])
    assert np.abs(fma).max() <= 9 * 2.0 ** -48
    assert np.sqrt(np.mean(fma ** 2)) <= np.sqrt(np.mean(two ** 2))
