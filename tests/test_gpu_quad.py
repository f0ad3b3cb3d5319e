"""Double precision with four lanes per ray against one ray per lane.

Queues of up to 64 to 200 rays per SM (by step rule and order) are traced by
the four-lane kernel, longer ones by the one-lane kernel, whose last rays the
four-lane kernel takes over.  Both
do the same operations on the same operands, so a ray's record is the same
bits in each (no tolerance): an image alone, and as many copies of it in one
buffer as pass the limit."""
import math

import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = {
    # fewer rays than a warp's eight quads, one more, an odd number of warps
    "1": (I.Image(a=0.9, incl=1.0, nx=1, ny=1, alpha0=3.0, alpha1=4.0, beta0=1.0, beta1=2.0), {}),
    "7": (I.Image(a=0.9, incl=1.0, nx=7, ny=1), {}),
    "9": (I.Image(a=0.9, incl=1.0, nx=3, ny=3), {}),
    # pole crossings, Euler redos, far stage angles, both stop surfaces
    "kerr": (I.Image(a=0.99, incl=math.radians(90.0), nx=37, ny=23), {}),
    "face_on_eq2": (I.Image(a=0.998, incl=math.radians(12.0), nx=29, ny=17), {"step_rule": gray.STEP_EQ2}),
    "equator": (I.Image(a=0.95, incl=math.radians(60.0), nx=30, ny=21, alpha0=-15, alpha1=15, beta0=-15, beta1=15),
                {"stop_equator": 1}),
    "flat": (I.Image(a=0.3, M=0.0, incl=1.0, nx=16, ny=9), {}),
    "retrograde": (I.Image(a=-0.7, incl=math.radians(120.0), nx=19, ny=18), {}),
    "step_cap": (I.Image(a=0.9, incl=1.2, nx=17, ny=16), {"max_steps": 211}),
}


def records(images, opt, budgets):
    tr = gray.Tracer(opt, sum(im.n for im in images))
    tr.setup(images)
    for b in budgets:
        tr.trace(step_budget=b)
    rec = tr.records()
    tr.close()
    return rec


@pytest.mark.parametrize("budgets", [(0,), (5, 1, 200, 0)], ids=["whole", "split"])
@pytest.mark.parametrize("name", CASES)
def test_four_lanes_per_ray_give_the_bits_of_one(name, budgets):
    im, options = CASES[name]
    opt = gray.Options(precision=gray.FP64, **{"max_steps": 20000, **options})
    alone = records([im], opt, budgets)
    limit = 200 * torch.cuda.get_device_properties(0).multi_processor_count
    copies = limit // im.n + 1
    many = records([im] * copies, opt, budgets).reshape(copies, im.n, -1)
    assert np.all(alone[:, 0] != gray.ACTIVE)
    same = (many == alone[None]) | (np.isnan(many) & np.isnan(alone[None]))
    assert np.all(same), np.argwhere(~same)[:5]


def test_a_short_state_with_a_long_queue_keeps_its_hand_off_list():
    """A queue longer than the four-lane limit over a state of fewer rays (its
    surplus entries lie outside the buffer and are skipped)."""
    im = I.Image(a=0.9, incl=1.0, nx=9, ny=7)
    opt = gray.Options(precision=gray.FP64, max_steps=20000)
    want = records([im], opt, (0,))
    limit = 200 * torch.cuda.get_device_properties(0).multi_processor_count
    order = torch.full((limit + 100,), -1, dtype=torch.int32, device="cuda")
    order[50:50 + im.n] = torch.arange(im.n, dtype=torch.int32, device="cuda")
    tr = gray.Tracer(opt, im.n)
    tr.setup([im])
    rc, n_active, _ = tr.trace(order=order)
    rec = tr.records()
    tr.close()
    assert rc == 0 and n_active == 0 and np.array_equal(rec, want)


def test_few_rays_of_a_long_buffer_reach_the_four_lane_kernel():
    """Warps that pass over finished or empty slots only count them as well, so
    the few rays left of a long buffer are handed over (the hand-off list is the
    state's last plane) and end with the bits of a trace alone."""
    im = I.Image(a=0.9, incl=1.0, nx=40, ny=30)
    opt = gray.Options(precision=gray.FP64, max_steps=20000)
    want = records([im], opt, (0,))
    n = 300 * torch.cuda.get_device_properties(0).multi_processor_count
    tr = gray.Tracer(opt, n)
    gray.gray_clear(tr.ctx, tr.state, n, 0, n)
    tr.setup([im], first_ray=n // 2)
    plane = lambda size: (size * n + 255) // 256 * 256
    first = 4 * plane(32) + 2 * plane(16)
    listed = tr.state[first:first + 4 * n].view(torch.int32)
    listed.fill_(-1)
    _, n_active, _ = tr.trace()
    rec = tr.records(first_ray=n // 2, n=im.n)
    rays = listed.cpu().numpy()
    rays = rays[rays >= 0]
    tr.close()
    assert n_active == 0 and np.array_equal(rec, want, equal_nan=True)
    assert len(rays) > im.n // 2 and len(set(rays)) == len(rays)
    assert rays.min() >= n // 2 and rays.max() < n // 2 + im.n


@pytest.mark.parametrize("name", CASES)
def test_one_lane_kernel_alone_gives_the_bits_of_four(name):
    """Fewer steps per call than lie between two refills (16): every ray yields
    inside its first block of steps, before any can be handed over, so the whole
    trajectory stays with the one-lane kernel, the longest rays' ends included."""
    im, options = CASES[name]
    opt = gray.Options(precision=gray.FP64, **{"max_steps": 20000, **options})
    alone = records([im], opt, (0,))
    limit = 200 * torch.cuda.get_device_properties(0).multi_processor_count
    copies = limit // im.n + 1
    tr = gray.Tracer(opt, copies * im.n)
    tr.setup([im] * copies)
    n_active = 1
    while n_active:
        _, n_active, _ = tr.trace(step_budget=15)
    rec = tr.records().reshape(copies, im.n, -1)
    tr.close()
    same = (rec == alone[None]) | (np.isnan(rec) & np.isnan(alone[None]))
    assert np.all(same), np.argwhere(~same)[:5]


@pytest.mark.parametrize("side", [84, 88, 150])
def test_budgets_do_not_change_results(side):
    """Calls of few steps, of some and of all take different kernels and
    hand-overs around 48 rays per SM; a ray's record is the same bits."""
    im = I.Image(a=0.95, incl=math.radians(80.0), nx=side, ny=side)
    opt = gray.Options(precision=gray.FP64, max_steps=20000)
    want = records([im], opt, (0,))
    for budgets in ((40, 600, 0), (512, 512, 0), (1024, 1025, 0), (1,) * 5 + (0,)):
        assert np.array_equal(records([im], opt, budgets), want, equal_nan=True), budgets


def test_warps_whose_lanes_are_all_busy_hand_over_too():
    """A warp full of long rays has no idle lane to ask the queue for more; it
    must still learn that the queue is empty.  Equal rays, whole warps of them,
    in a buffer of empty slots: all of them are handed over."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, full = 300 * sms, 32 * (20 * sms // 32)
    opt = gray.Options(precision=gray.FP64, max_steps=20000)
    one = torch.tensor([[3.0, 2.0, 0.9, 1.2, 1000.0]], dtype=torch.float64, device="cuda")
    tr = gray.Tracer(opt, 1)
    tr.setup_rays(one)
    tr.trace()
    want = tr.records()
    tr.close()
    tr = gray.Tracer(opt, n)
    gray.gray_clear(tr.ctx, tr.state, n, 0, n)
    tr.setup_rays(one.repeat(full, 1), first_ray=0)
    plane = lambda size: (size * n + 255) // 256 * 256
    first = 4 * plane(32) + 2 * plane(16)
    listed = tr.state[first:first + 4 * n].view(torch.int32)
    listed.fill_(-1)
    _, n_active, _ = tr.trace()
    rec = tr.records(first_ray=0, n=full)
    rays = listed.cpu().numpy()
    tr.close()
    assert n_active == 0 and np.all(rec == want)
    assert np.array_equal(np.sort(rays[rays >= 0]), np.arange(full))
