"""gray_cancel while the last rays are with another kernel than they began in:
the double-precision hand-over to four lanes per ray, and the teams of four
warps at the end of the zone pass.

Each trace is cancelled after a part of its time, at several parts, then
finished; every ray ends with the bits of a trace that was not interrupted, and
every step is counted once."""
import math
import threading
import time

import numpy as np
import pytest
import torch

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = {
    # 250 rays per SM: the one-lane kernel hands over its last 32 per SM
    "hand_over": (I.Image(a=0.9, incl=math.radians(75.0), nx=230, ny=170), dict(precision=gray.FP64)),
    # a ray of ~1000 zone steps ends the zone pass alone in a team
    "zone_team": (I.Image(a=0.94, incl=math.radians(40.0), nx=61, ny=61),
                  dict(precision=gray.FP32_KAHAN_SEL64, step_rule=gray.STEP_EQ2, h_min=1e-9, r_sw=0.02)),
}


@pytest.mark.parametrize("name", CASES)
def test_cancelled_late_passes_resume_bit_for_bit(name):
    im, options = CASES[name]
    opt = gray.Options(max_steps=20000, **options)
    ref = gray.Tracer(opt, im.n)
    for _ in range(2):
        ref.setup([im])
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        _, _, want_stats = ref.trace()
        full = time.perf_counter() - t0
    want = ref.records()
    ref.close()

    tr = gray.Tracer(opt, im.n)
    stopped = 0
    for part in np.linspace(0.3, 0.95, 14):
        tr.setup([im])
        torch.cuda.synchronize()
        out = []
        th = threading.Thread(target=lambda: out.append(tr.trace()))
        th.start()
        time.sleep(part * full)
        gray.gray_cancel(tr.ctx, True)
        th.join()
        gray.gray_cancel(tr.ctx, False)
        total = np.array(out[0][2][:3])
        stopped += out[0][1] > 0
        rc, n_active, st = tr.trace()
        total += np.array(st[:3])
        assert rc == 0 and n_active == 0
        assert np.array_equal(tr.records(), want, equal_nan=True), part
        assert np.array_equal(total, want_stats[:3]), part
    tr.close()
    assert stopped > 0  # some of the calls were cut short
