"""FP64 forces and energies against the same sums in extended precision (113 or
64 bits).  The positions are exact in both, so that what is measured is the
rounding of the pair terms, of their constants and of the sums.

Formed pair by pair in the textbook way (s = a/r, powers of s, FP64 throughout)
forces were off by 1.17e-15 of their norm on such blocks and energies by
1.8e-16; with the constants of the regrouped form each rounded on its own, by
1.22e-15 and 1.6e-16.  The bounds are 1.0e-15 and 1.7e-16."""
import numpy as np
import pytest

import pta_inputs as PI
from gpu_util import gpu_package

pytestmark = pytest.mark.gpu

X = np.longdouble


@pytest.fixture(scope="module")
def P():
    return gpu_package()


def _reference(pos, p):
    x = pos.astype(X)
    eps, c, a, rc = X(p.eps), X(p.c), X(p.a), X(p.rc)
    An, Am = (a / rc) ** p.n, (a / rc) ** p.m
    Bn, Bm = p.n / rc * An, p.m / rc * Am
    d = x[None] - x[:, None]
    r2 = (d * d).sum(2)
    np.fill_diagonal(r2, 2 * rc * rc)
    inside = r2 < rc * rc
    r = np.sqrt(np.where(inside, r2, rc * rc))
    s = a / r
    sn, sm = s ** p.n, s ** p.m
    rho = np.where(inside, sm - Am + Bm * (r - rc), X(0)).sum(1)
    en = np.where(inside, sn - An + Bn * (r - rc), X(0)).sum(1)
    dB = -eps * c / 2 / np.sqrt(rho)
    g = eps * (-p.n * sn / r + Bn) + (dB[:, None] + dB[None]) * (-p.m * sm / r + Bm)
    g = np.where(inside, g / r, X(0))
    return (g[:, :, None] * d).sum(1), eps * en / 2 - eps * c * np.sqrt(rho)


def test_forces_and_energies_against_extended_precision(P):
    errors = []
    for shape in ((4, 4, 4), (5, 4, 6), (6, 5, 7)):
        for seed in (1, 2):
            c = P.Ctx(shape, T0=0.0, precision=0)
            pos = PI.gaussian_jitter_fcc(shape, 0.1, seed=seed)
            pos = np.round(pos * 2.0**24) / 2.0**24
            c.set_state(pos, np.zeros_like(pos))
            f, pe, _ = c.forces()
            for got, want in zip((f, pe), _reference(pos, c.potential)):
                errors.append(np.sqrt(((got - want) ** 2).sum() / (want**2).sum()))
            c.close()
    ef, ee = (float(np.mean(errors[i::2])) for i in (0, 1))
    print("forces %.2e, energies %.2e" % (ef, ee))
    assert ef < 1.0e-15 and ee < 1.7e-16
