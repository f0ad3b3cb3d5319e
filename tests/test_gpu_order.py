"""The lead-first queue of a trace without a caller's order.

Under the benchmark rule a trace of more than 1.6 times the rays that the single-precision pass holds at
once (512 per SM) orders its ACTIVE rays itself; a ray's result does not depend on its place in
the queue, so every record equals, bit for bit (no tolerance), that of the
same trace under an explicit order."""
import math

import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def trace(opt, n, prepare, budgets, order):
    tr = gray.Tracer(opt, n)
    prepare(tr)
    for b in budgets:
        q = torch.arange(n, dtype=torch.int32, device="cuda") if order else None
        _, n_active, st = tr.trace(step_budget=b, order=q)
    rec = tr.records()
    tr.close()
    return rec, n_active, st


@pytest.mark.parametrize("extra", [1, 1023, 5000])
@pytest.mark.parametrize("precision", ["fp32", "fp32_kahan", "fp32_kahan_sel64"])
def test_lead_first_queue_equals_an_explicit_order(precision, extra):
    n = 512 * 8 * torch.cuda.get_device_properties(0).multi_processor_count // 5 + extra
    opt = gray.Options(precision=gray.PRECISIONS[precision], max_steps=20000, r_sw=0.02)
    rays = torch.from_numpy(I.mixed_rays(n, offset=11 * n)).cuda()

    def prepare(tr):
        tr.setup_rays(rays)
        gray.gray_clear(tr.ctx, tr.state, n, 77, 1500)  # empty slots across a block of the ordering

    got = trace(opt, n, prepare, (0,), False)
    want = trace(opt, n, prepare, (0,), True)
    assert got[1:] == want[1:] and got[1] == 0
    assert np.array_equal(got[0], want[0], equal_nan=True)


@pytest.mark.parametrize("image", ["flat", "face_on"])
def test_lead_first_queue_of_a_resumed_trace(image):
    """All rays in one class (M = 0: none leads; face-on: L_z = 0, all lead),
    most of them finished when the second call orders what is left."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    side = int(math.isqrt(512 * 8 * sms // 5)) + 3
    im = I.Image(a=0.3, M=0.0, incl=1.0, nx=side, ny=side) if image == "flat" else \
        I.Image(a=0.9, incl=0.0, nx=side, ny=side)
    opt = gray.Options(precision=gray.FP32_KAHAN_SEL64, max_steps=20000, r_sw=0.02)
    got = trace(opt, im.n, lambda tr: tr.setup([im]), (513, 0), False)
    want = trace(opt, im.n, lambda tr: tr.setup([im]), (513, 0), True)
    assert got[1:] == want[1:] and got[1] == 0
    assert np.array_equal(got[0], want[0], equal_nan=True)


@pytest.mark.parametrize("surplus", [-1, 0, 1])
def test_as_many_active_rays_as_the_limit(surplus):
    """The limit counts ACTIVE rays: below and at it the pass takes the buffer as
    it lies, above it the lead-first queue."""
    limit = 512 * 8 * torch.cuda.get_device_properties(0).multi_processor_count // 5
    n = limit + 4000
    opt = gray.Options(precision=gray.FP32_KAHAN_SEL64, max_steps=20000, r_sw=0.02)
    rays = torch.from_numpy(I.mixed_rays(n, offset=5 * n)).cuda()

    def prepare(tr):
        tr.setup_rays(rays)
        gray.gray_clear(tr.ctx, tr.state, n, 501, 4000 - surplus)

    got = trace(opt, n, prepare, (0,), False)
    want = trace(opt, n, prepare, (0,), True)
    assert got[1:] == want[1:] and got[1] == 0
    assert np.array_equal(got[0], want[0], equal_nan=True)
