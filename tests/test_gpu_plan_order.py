"""The planned queue is a permutation of the images' rays in descending
predicted cost, whatever the images' sizes (last strips of one to three rows,
single columns, polar grids, several images at an offset)."""
import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LISTS = {
    "one_pixel": [I.Image(a=0.5, incl=1.0, nx=1, ny=1)],
    "one_column": [I.Image(a=0.5, incl=1.0, nx=1, ny=70)],
    "one_row": [I.Image(a=0.5, incl=1.0, nx=70, ny=1)],
    "ragged": [I.Image(a=0.9, incl=1.2, nx=33, ny=ny) for ny in (4, 5, 6, 7)],
    "mixed": [I.polar_image(0.9, 40.0, 37, 11), I.Image(a=0.7, incl=0.6, nx=50, ny=41), I.polar_image(0.2, 70.0, 9, 1)],
    # more images than travel as a kernel argument
    "many": [I.Image(a=0.1 * k, incl=0.3 + 0.1 * k, nx=9 + k, ny=21 - k) for k in range(9)],
}


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("name", LISTS)
def test_planned_queue_is_a_permutation(name, fused):
    images, first, stride, budget = LISTS[name], 13, 3, 120
    n = sum(im.n for im in images)
    tr = gray.Tracer(gray.Options(precision=gray.FP32_KAHAN_SEL64, max_steps=20000, r_sw=0.02), n + 40)
    gray.gray_clear(tr.ctx, tr.state, tr.n, 0, tr.n)
    if fused:
        q = tr.setup_plan(images, first_ray=first, probe_stride=stride, probe_budget=budget)
    else:
        tr.setup(images, first_ray=first)
        q = tr.plan(images, first_ray=first, probe_stride=stride, probe_budget=budget)
    rec = tr.records()
    q = q.cpu().numpy()
    assert np.array_equal(np.sort(q), np.arange(first, first + n))
    # the documented key: the largest cost among the 4 x 4 probes around the
    # pixel's cell, in 1024 buckets over 0 .. 9 budget
    key = np.zeros(first + n)
    off = first
    for im in images:
        probe = rec[off:off + im.n].reshape(im.ny, im.nx, -1)[::stride, ::stride]
        cost = np.where(probe[..., 0] == gray.ACTIVE, probe[..., 1] + 8 * probe[..., 2], probe[..., 1])
        for row in range(im.ny):
            for col in range(im.nx):
                r, c = row // stride, col // stride
                near = cost[max(0, r - 1):r + 3, max(0, c - 1):c + 3]
                key[off + row * im.nx + col] = near.max()
        off += im.n
    bucket = np.minimum(1023, np.floor(key[q] * (1024.0 / 9.0) / budget))
    assert np.all(np.diff(bucket) <= 1e-9 + (np.abs(key[q][:-1] * (1024.0 / 9.0) / budget % 1.0) < 1e-3))
    _, n_active, _ = tr.trace(order=torch.from_numpy(q).cuda())
    assert n_active == 0
    tr.close()


@pytest.mark.parametrize("side", [80, 84, 88, 150])
def test_double_precision_probes_advance_as_a_trace(side):
    """Around 48 probes per SM the planner's probe pass changes kernel: with every
    pixel a probe, its states are those of a trace of the same budget."""
    im = I.Image(a=0.9, incl=1.2, nx=side, ny=side)
    recs = []
    for plan in (True, False):
        tr = gray.Tracer(gray.Options(precision=gray.FP64, max_steps=20000), im.n)
        if plan:
            q = tr.setup_plan([im], probe_stride=1, probe_budget=40)
            assert np.array_equal(np.sort(q.cpu().numpy()), np.arange(im.n))
        else:
            tr.setup([im])
            tr.trace(step_budget=40)
        recs.append(tr.records())
        tr.close()
    assert np.array_equal(recs[0], recs[1], equal_nan=True)
