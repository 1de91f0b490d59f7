"""K, U and T of a state are summed in FP64 in both precisions: against sums in
extended precision of what each atom contributes, which is known exactly (its
energy and force are returned; velocities are chosen so that its kinetic energy
is rounded once).  A sum of n terms along the reduction tree (lanes of a warp,
warps of a block, blocks, groups: at most 24 additions deep) is off by at most
24 x 2^-53 of the sum of their sizes.  In mixed precision the terms are FP32
numbers, multiples of the smallest one's last place, so that their FP64 sums
are exact while they stay below 2^53 of it (a pair of FP32 numbers holds 2^48)."""
import numpy as np
import pytest

from gpu_util import gpu_package

pytestmark = pytest.mark.gpu

GPA = 1.602176634e-19 / 1e-30 / 1e9
MV2 = 1.66053906660e-27 * 1e-20 / 1e-30 / 1.602176634e-19
DEPTH = 24 * 2.0**-53


@pytest.fixture(scope="module")
def P():
    return gpu_package()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape,lanes", [((2, 2, 3), 1), ((11, 9, 10), 1), ((20, 20, 21), 1),
                                         ((21, 20, 20), 16), ((9, 7, 8), 4)])
def test_sums_are_fp64(P, prec, shape, lanes):
    c = P.Ctx(shape, T0=300.0, seed=4, precision=prec, lanes=lanes)
    pos, _ = c.get_state()
    rng = np.random.default_rng(7)
    pos = np.round((pos + rng.normal(0, 0.1, pos.shape)) * 2.0**20) / 2.0**20
    # slow and fast atoms; squares and their sums are exact
    slow = rng.random((len(pos), 1)) < 0.5
    vel = np.where(slow, rng.integers(3, 9, pos.shape), rng.integers(200, 256, pos.shape))
    vel = vel * rng.choice([-1, 1], pos.shape) * 2.0**-14
    flags = c.flags()
    vel[flags != 0] = 0.0
    c.set_state(pos, vel)
    f, pe, (K, U, T) = c.forces()
    ke_fac = 0.5 * c.params.mass_amu * MV2
    v2 = (vel * vel).sum(1)
    ke = (np.float32(ke_fac) * v2.astype(np.float32) if prec else ke_fac * v2)
    ke, pe, r = (a.astype(np.longdouble) for a in (ke, pe, -f[flags == 2, 2]))
    assert abs(U - pe.sum()) <= DEPTH * np.abs(pe).sum()
    # the factor itself is off by a few roundings in FP64 (in FP32 it is the same)
    assert abs(K - ke.sum()) <= (DEPTH + (0 if prec else 8 * 2.0**-53)) * ke.sum()
    t_fac = GPA / (shape[0] * shape[1] * 4.05**2)
    assert abs(T - r.sum() * t_fac) <= (DEPTH + 8 * 2.0**-53) * np.abs(r).sum() * t_fac
    if prec:
        for total, terms in ((K, ke), (U, pe)):
            size = np.abs(terms[terms != 0])
            assert size.sum() <= 2.0**53 * np.spacing(np.float32(size.min(initial=1.0)))
            assert total == terms.sum()
    c.close()
