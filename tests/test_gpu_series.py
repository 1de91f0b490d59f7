"""The sample series of a context that runs both on its own and in a batch:
either may have to replace the buffer by a larger one, and the other must then
write to that one."""
import numpy as np
import pytest

from gpu_util import gpu_package

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 5), (3, 5, 4)]
# bursts (of the first member alone, of both in the batch); room for 20 samples
# at first, so that each grows the buffer once
PLANS = {"solo grows": [("solo", 90), ("batch", 50), ("solo", 30)],
         "batch grows": [("solo", 10), ("batch", 70), ("solo", 60), ("batch", 15)],
         "both grow": [("batch", 10), ("solo", 50), ("batch", 150), ("solo", 140), ("batch", 20)]}


@pytest.fixture(scope="module")
def P():
    return gpu_package()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("timed", [False, True])        # resident run, launched passes
@pytest.mark.parametrize("plan", sorted(PLANS))
def test_series_of_a_context_in_a_batch(P, plan, prec, timed):
    def ctxs():
        cs = [P.Ctx(sh, T0=300.0, seed=i, precision=prec, burst_steps=20)
              for i, sh in enumerate(SHAPES)]
        for c in cs:
            c.set_timing(timed)
        return cs

    ref, cs = ctxs(), ctxs()                # ref: each member always on its own
    b = P.Batch(cs)
    b.set_timing(timed)
    for who, steps in PLANS[plan]:
        members = [0] if who == "solo" else [0, 1]
        if who == "solo":
            cs[0].fine_burst(steps)
        else:
            b.fine_burst([steps, steps])
        for i in members:
            ref[i].fine_burst(steps)
            got, want = cs[i].series(), ref[i].series()
            assert len(got) == steps and np.array_equal(got, want)
    b.close()
    for c in cs + ref:
        c.close()
