"""Every route rounds alike, for exponents other than 7 and 6 too: bursts inside
one kernel (resident, swept) against launched passes, bit for bit."""
import numpy as np
import pytest

from gpu_util import gpu_package

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,m", [(9, 6), (12, 7), (10, 8)])
@pytest.mark.parametrize("shape,lanes", [((5, 6, 5), 0), ((12, 12, 12), 16), ((19, 20, 21), 4)])
def test_routes_of_other_exponents_agree(P, prec, n, m, shape, lanes):
    out = []
    for timed in (False, True):
        c = P.Ctx(shape, T0=100.0, seed=2, precision=prec, lanes=lanes,
                  potential=P.default_potential(n=n, m=m))
        c.set_timing(timed)
        r = c.fine_burst(40)
        assert r.nsteps == 40
        out.append((c.series().copy(), *c.get_state()))
        c.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
