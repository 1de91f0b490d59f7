"""Resident runs (one cooperative kernel from list build to list build, used
for tables that fit the GPU at one block per SM) against the passes launched
one by one, which kernel timing uses: bit for bit, alone and in batches whose
members end their bursts at different steps or fail."""
import numpy as np
import pytest

import pta_inputs as PI
from gpu_util import gpu_package

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


def _run(P, shape, prec, steps, timed, seed=3, **kw):
    c = P.Ctx(shape, T0=300.0, seed=seed, precision=prec, **kw)
    c.apply_strain(1e-3)
    c.set_timing(timed)
    a = c.fine_burst(steps)
    out = (c.series().copy(), *c.get_state(), a.rebuilds, a.prunes)
    c.close()
    return out


def _equal(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


# one warp; fewer tiles than SMs; a partial last tile; more than 32 groups of
# pair blocks; the largest lane counts
@pytest.mark.parametrize("prec,shape,lanes", [
    (1, (1, 1, 3), 1), (0, (3, 2, 4), 2), (1, (6, 5, 7), 0), (0, (5, 6, 5), 0), (1, (9, 11, 10), 8),
    (1, (17, 16, 15), 4), (0, (11, 9, 10), 16)])
def test_resident_equals_launched(P, prec, shape, lanes):
    _equal(_run(P, shape, prec, 130, False, lanes=lanes), _run(P, shape, prec, 130, True, lanes=lanes))


# more tiles than resident warps: each block sweeps its tiles (uneven shares, a
# partial last tile, both precisions, the fewest and the most lanes)
@pytest.mark.parametrize("prec,shape,lanes", [
    (1, (12, 12, 12), 16), (0, (11, 13, 12), 16), (1, (19, 20, 21), 4), (1, (28, 27, 29), 1),
    (0, (28, 27, 29), 1), (1, (19, 20, 18), 8)])
def test_sweeps_equal_launched(P, prec, shape, lanes):
    _equal(_run(P, shape, prec, 45, False, lanes=lanes), _run(P, shape, prec, 45, True, lanes=lanes))


# members with different lanes share one sweep
def test_a_swept_batch_equals_its_members(P):
    shapes, steps = [(19, 20, 19), (5, 6, 5), (13, 12, 14)], [40, 60, 25]
    solo = [_run(P, sh, 1, n, False, seed=i) for i, (sh, n) in enumerate(zip(shapes, steps))]
    cs = [P.Ctx(sh, T0=300.0, seed=i, precision=1) for i, sh in enumerate(shapes)]
    assert len({c.layout()["lanes"] for c in cs}) > 1
    b = P.Batch(cs)
    b.apply_strain([1e-3] * len(cs))
    b.fine_burst(steps)
    for c, s in zip(cs, solo):
        _equal((c.series().copy(), *c.get_state()), s[:3])
    b.close()
    for c in cs:
        c.close()


# and one launch of each pass, with the members in any order
@pytest.mark.parametrize("prec,order", [(1, (0, 1, 2)), (1, (2, 0, 1)), (0, (1, 2, 0))])
def test_a_launched_batch_of_uneven_lanes_equals_its_members(P, prec, order):
    shapes, steps = [(9, 20, 19), (5, 6, 5), (13, 12, 14)], [40, 60, 25]
    solo = [_run(P, sh, prec, n, False, seed=i) for i, (sh, n) in enumerate(zip(shapes, steps))]
    cs = [P.Ctx(shapes[i], T0=300.0, seed=i, precision=prec) for i in order]
    assert len({c.layout()["lanes"] for c in cs}) > 1
    b = P.Batch(cs)
    b.set_timing(True)
    b.apply_strain([1e-3] * len(cs))
    b.fine_burst([steps[i] for i in order])
    for c, i in zip(cs, order):
        _equal((c.series().copy(), *c.get_state()), solo[i][:3])
    b.close()
    for c in cs:
        c.close()


# the sums of a launched pass: one group of blocks, several, a partial last one,
# and more than one round of the finishing kernel (beyond 128 groups).  Each
# atom's energy is one FP32 (FP64) number and the tree's error per level is
# below 2^-44 (2^-53) of the sum of their sizes.
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape,lanes", [((2, 2, 3), 1), ((11, 9, 10), 1), ((20, 20, 21), 1),
                                         ((21, 20, 20), 16)])
def test_sums_of_a_launched_pass(P, prec, shape, lanes):
    c = P.Ctx(shape, T0=300.0, seed=4, precision=prec, lanes=lanes)
    f, pe, obs = c.forces()
    assert abs(obs[1] - pe.sum(dtype=np.longdouble)) <= 24 * 2.0**-44 * np.abs(pe).sum()
    c.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_a_burst_longer_than_one_launch(P, prec):
    # a cold crystal asks for no list build, so the run reaches its limit of
    # 4,000 steps per launch inside the burst
    kw = dict(T0=1.0, seed=2, precision=prec)
    out = []
    for timed in (False, True):
        c = P.Ctx((3, 3, 4), **kw)
        c.set_timing(timed)
        a = c.fine_burst(4100)
        out.append((c.series().copy(), *c.get_state(), a.nsteps))
        c.close()
    assert out[0][3] == 4100
    _equal(out[0], out[1])


@pytest.mark.parametrize("prec", [0, 1])
def test_members_of_a_resident_batch_end_on_their_own(P, prec):
    shapes, steps = [(4, 4, 4), (6, 5, 7), (3, 3, 5), (5, 5, 5), (4, 3, 4), (3, 4, 3)], \
        [90, 140, 1, 0, 33, 139]
    solo = [_run(P, sh, prec, n, False, seed=i) if n else None
            for i, (sh, n) in enumerate(zip(shapes, steps))]
    cs = [P.Ctx(sh, T0=300.0, seed=i, precision=prec) for i, sh in enumerate(shapes)]
    assert len({c.layout()["lanes"] for c in cs}) == 1      # one launch group
    b = P.Batch(cs)
    b.apply_strain([1e-3] * len(cs))
    res = b.fine_burst(steps)
    for c, r, s, n in zip(cs, res, solo, steps):
        assert r.nsteps == n and r.status == 0
        if n:
            _equal((c.series().copy(), *c.get_state()), s[:3])
    b.close()
    for c in cs:
        c.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_a_failing_member_stops_alone(P, prec):
    # two atoms on one site: the first sample is not finite
    shape = (4, 4, 5)
    good = _run(P, shape, prec, 60, False, seed=9)
    bad = P.Ctx(shape, T0=300.0, seed=1, precision=prec)
    pos, vel = bad.get_state()
    i = int(np.flatnonzero(bad.flags() == 0)[0])
    pos[i] = pos[i + 1]
    bad.set_state(pos, vel)
    ok = P.Ctx(shape, T0=300.0, seed=9, precision=prec)
    b = P.Batch([bad, ok])
    b.apply_strain([1e-3, 1e-3])
    r = b.fine_burst([60, 60])
    assert r[0].status == -5 and r[0].nsteps == 0
    assert r[1].status == 0 and r[1].nsteps == 60
    _equal((ok.series().copy(), *ok.get_state()), good[:3])
    b.close()
    with pytest.raises(P.PTAError) as e:      # and alone
        bad.fine_burst(20)
    assert e.value.status == -5
    bad.close()
    ok.close()
