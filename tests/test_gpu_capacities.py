"""Contexts of different list capacities alive at once, and capacities beyond
what the list build can hold in shared memory."""
import numpy as np
import pytest

import pta_inputs as PI
from gpu_util import force_error, gpu_package, on_grid, sorted_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


def _ctx(P, shape, seed, **kw):
    c = P.Ctx(shape, T0=300.0, seed=seed, **kw)
    pos = on_grid(PI.jittered_fcc(shape, 0.2, seed=seed))
    c.set_state(pos, c.get_state()[1])
    return c


# the list build of the first context needs more shared memory (neigh_cap 4096:
# the largest that can be asked for) than that of the ones used after it
@pytest.mark.parametrize("cap", [1024, 1600, 4096])
def test_a_context_is_not_limited_by_a_later_smaller_one(P, cap):
    a = _ctx(P, (5, 4, 6), 1, precision=1, neigh_cap=cap)
    f, pe, obs = a.forces()
    counts, lists = a.neighbours(cap=512)
    b = _ctx(P, (4, 4, 4), 2, precision=1, skin=0.5)
    b.forces()
    f2, pe2, obs2 = a.forces()
    counts2, lists2 = a.neighbours(cap=512)
    for x, y in ((f, f2), (pe, pe2), (obs, obs2), (counts, counts2), (lists, lists2)):
        assert np.array_equal(x, y)
    a.close()
    b.close()


# graphs captured after the smaller context's: launched passes and resident run
def test_graphs_captured_after_a_smaller_context(P):
    def start(c):
        c.apply_strain(1e-3)
        return c

    small = _ctx(P, (4, 4, 4), 2, precision=1, skin=0.5)
    out = []
    for later in (False, True):
        a = start(_ctx(P, (5, 4, 6), 1, precision=1, neigh_cap=4096))
        if later:
            small.forces()
        a.fine_burst(40)
        a.set_timing(True)              # captures launched passes
        if later:
            small.fine_burst(5)
        r = a.fine_burst(40)
        assert r.status == 0 and r.rebuilds >= 1
        out.append((a.series().copy(), *a.get_state()))
        a.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    small.close()


# automatic capacity beyond neigh_cap's range: 22,176 entries at a skin of 30 A,
# whose candidates do not fit in shared memory
@pytest.mark.parametrize("prec,shape,lanes", [(1, (4, 4, 4), 0), (0, (8, 8, 8), 2), (1, (9, 3, 7), 16)])
def test_capacities_beyond_shared_memory(P, oracle, prec, shape, lanes):
    skin = 30.0
    c = P.Ctx(shape, T0=0.0, precision=prec, lanes=lanes, skin=skin)
    assert c.layout()["neigh_cap"] > 4096
    pos = on_grid(PI.jittered_fcc(shape, 0.3, seed=3))
    c.set_state(pos, np.zeros_like(pos))
    n = len(pos)
    f, pe, _ = c.forces()
    f_ref, pe_ref, _ = oracle.eam(pos, oracle.Potential(
        eps=c.potential.eps, c=c.potential.c, a=c.potential.a, rc=c.potential.rc, n=7, m=6))
    assert force_error(f, f_ref) < (1e-10 if prec == 0 else 1e-5)
    assert np.max(np.abs(pe - pe_ref) / np.abs(pe_ref)) < (1e-11 if prec == 0 else 1e-5)
    c_gpu, l_gpu = c.neighbours(cap=n)
    c_ref, l_ref = oracle.pairs(pos, c.potential.rc + skin, cap=n, method="brute")
    assert np.array_equal(c_gpu, c_ref)
    assert sorted_rows(c_gpu, l_gpu) == sorted_rows(c_ref, l_ref)
    c.close()


def test_a_batch_of_small_and_large_capacities(P):
    def members():
        return [_ctx(P, (4, 4, 4), 1, precision=1), _ctx(P, (5, 4, 4), 2, precision=1, skin=30.0),
                _ctx(P, (3, 4, 5), 3, precision=1, neigh_cap=4096)]

    solo = []
    for c in members():
        c.apply_strain(1e-3)
        c.fine_burst(30)
        solo.append((c.series().copy(), *c.get_state()))
        c.close()
    cs = members()
    b = P.Batch(cs)
    b.apply_strain([1e-3] * 3)
    b.fine_burst([30] * 3)
    for c, s in zip(cs, solo):
        for x, y in zip((c.series().copy(), *c.get_state()), s):
            assert np.array_equal(x, y)
    b.close()
    for c in cs:
        c.close()
