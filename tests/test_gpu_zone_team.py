"""The last zone rays of a block in a team of four warps.

A block hands its last rays over 32 steps after the hand-off list is drained.
A trace in calls of at most 20 steps never gets there, so its records are
those of a ray per lane; both run the same operations, so the records are the
same bits (no tolerance)."""
import math

import numpy as np
import pytest

from paper_1303_5057_gb300 import gray
from paper_1303_5057_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# rays near a pole take up to a thousand zone steps under Eq. 2
EQ2 = dict(step_rule=gray.STEP_EQ2, h_min=1e-9)
CASES = {
    # the column alpha = 0 crosses the pole; all rays stop inside the zone
    "pole_column": (I.Image(a=0.94, incl=math.radians(40.0), nx=61, ny=61), dict(EQ2, r_sw=0.02)),
    # a wide zone: rays climb out of it as well, and it holds whole passages
    "wide_zone": (I.Image(a=0.99, incl=math.radians(85.0), nx=33, ny=40), dict(EQ2, r_sw=1.0)),
    "wide_zone_bench": (I.Image(a=0.9, incl=math.radians(60.0), nx=40, ny=33), dict(r_sw=0.9)),
    "equator": (I.Image(a=0.998, incl=math.radians(30.0), nx=41, ny=41, alpha0=-4, alpha1=4, beta0=-4, beta1=4),
                dict(EQ2, r_sw=1.0, stop_equator=1)),
    # the step cap falls inside the zone
    "step_cap": (I.Image(a=0.94, incl=math.radians(40.0), nx=61, ny=61), dict(EQ2, r_sw=0.02, max_steps=520)),
    # one ray
    "one": (I.Image(a=0.94, incl=math.radians(40.0), nx=1, ny=1, alpha0=-0.01, alpha1=0.01, beta0=-3, beta1=-2.9),
            dict(EQ2, r_sw=0.02)),
}


@pytest.mark.parametrize("name", CASES)
def test_team_equals_a_ray_per_lane(name):
    im, options = CASES[name]
    opt = gray.Options(precision=gray.FP32_KAHAN_SEL64, **{"max_steps": 20000, **options})
    recs, stats = [], []
    for budget in (0, 20):
        tr = gray.Tracer(opt, im.n)
        tr.setup([im])
        total = np.zeros(3, dtype=np.int64)
        n_active = 1
        while n_active:
            _, n_active, st = tr.trace(step_budget=budget)
            total += np.array(st[:3])
        recs.append(tr.records())
        stats.append(total)
        tr.close()
    assert np.array_equal(recs[0], recs[1], equal_nan=True)
    assert np.array_equal(stats[0], stats[1])  # steps, Euler redos and zone steps counted once
    if name in ("pole_column", "wide_zone"):
        assert recs[0][:, 16].max() > 200  # long enough to be handed over
