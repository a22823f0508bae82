"""Launch options out of range are refused before anything is sized by them: the search for a tile of
10^9 z values took seconds."""
import math
import time

import pytest

from paper_1311_2481_gb300 import build, tc


@pytest.mark.parametrize("kw", [dict(theta_zt=10 ** 9), dict(theta_zt=65), dict(theta_zt=-1), dict(stage_rows=-1)])
def test_refused_at_once(kw):
    build.build()
    args = (24, 4, 4, 1, 0.5, 50.0, 0.0, 2 * math.pi / 3.16, 1e-3)
    plan = tc.Plan(*args, host_only=True)
    t = time.perf_counter()
    with pytest.raises(tc.TCError) as e:
        tc.Plan(*args, host_only=True, **kw)
    if "theta_zt" in kw:
        with pytest.raises(tc.TCError):
            plan.set(tc.TC_SET_THETA_ZT, kw["theta_zt"])
    assert e.value.status == tc.TC_ERR_ARG
    assert time.perf_counter() - t < 1.0
