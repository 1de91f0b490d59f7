"""Verlet lists in their two parts (near entries read as they stand, far
entries pruned into the inner list) over the layouts the parameters can ask
for: a skin narrower than the near part (no far entries), pruning off (far
entries behind each lane's near ones), a pruning margin wider than the near
part (a fresh list is pruned before use), few and many lanes per atom."""
import numpy as np
import pytest

import pta_inputs as PI
from gpu_util import force_error, gpu_package, on_grid, sorted_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


def _pot(oracle, p):
    return oracle.Potential(eps=p.eps, c=p.c, a=p.a, rc=p.rc, n=p.n, m=p.m)


@pytest.mark.parametrize("prec,lanes,skin,margin", [
    (1, 1, 0.25, 0.0), (0, 2, 0.25, 0.0), (1, 2, 2.0, 0.8), (0, 16, 2.0, 0.8), (1, 8, 1.0, 0.05),
    (0, 1, 2.0, -1.0), (1, 16, 2.0, -1.0)])
def test_lists_and_forces_of_every_layout(P, oracle, prec, lanes, skin, margin):
    shape = (5, 7, 4)
    ctx = P.Ctx(shape, T0=0.0, precision=prec, lanes=lanes, skin=skin, prune_margin=margin)
    pos = on_grid(PI.jittered_fcc(shape, 0.3, seed=lanes))
    ctx.set_state(pos, np.zeros_like(pos))
    c_gpu, l_gpu = ctx.neighbours(cap=512)
    c_ref, l_ref = oracle.pairs(pos, ctx.potential.rc + skin, cap=512, method="brute")
    assert np.array_equal(c_gpu, c_ref)
    assert sorted_rows(c_gpu, l_gpu) == sorted_rows(c_ref, l_ref)
    f, pe, _ = ctx.forces()
    f_ref, pe_ref, _ = oracle.eam(pos, _pot(oracle, ctx.potential))
    assert force_error(f, f_ref) < (1e-10 if prec == 0 else 1e-5)
    assert np.max(np.abs(pe - pe_ref) / np.abs(pe_ref)) < (1e-11 if prec == 0 else 1e-5)
    ctx.close()


@pytest.mark.parametrize("prec,lanes", [(0, 4), (1, 1), (1, 8)])
def test_pruning_margin_changes_no_bit(P, prec, lanes):
    out = []
    for margin in (0.3, 0.9, -1.0):
        ctx = P.Ctx((6, 5, 7), T0=300.0, seed=4, precision=prec, lanes=lanes, prune_margin=margin)
        ctx.apply_strain(2e-3)
        ctx.fine_burst(150)
        out.append((ctx.series().copy(), *ctx.get_state()))
        ctx.close()
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,m", [(9, 6), (12, 7), (7, 1)])
def test_other_exponents(P, oracle, prec, n, m):
    pot = P.default_potential(n=n, m=m)
    ctx = P.Ctx((5, 4, 6), T0=0.0, precision=prec, potential=pot)
    pos = on_grid(PI.gaussian_jitter_fcc((5, 4, 6), 0.1, seed=n))
    ctx.set_state(pos, np.zeros_like(pos))
    f, pe, _ = ctx.forces()
    f_ref, pe_ref, _ = oracle.eam(pos, _pot(oracle, pot))
    assert force_error(f, f_ref) < (1e-10 if prec == 0 else 1e-5)
    # c is that of the 7-6 crystal, so these energies cross zero: relative to
    # their rms
    scale = np.sqrt(np.mean(pe_ref ** 2))
    assert np.max(np.abs(pe - pe_ref)) / scale < (1e-11 if prec == 0 else 1e-5)
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_an_atom_one_record_period_away_is_no_neighbour(P, oracle, prec):
    # records repeat every 2^32 quanta (64 A at the default radii): an atom
    # far outside the cell grid, where its record equals that of a place inside
    # the lattice, is still listed by its true distance
    shape = (5, 5, 5)
    ctx = P.Ctx(shape, T0=0.0, precision=prec)
    pos = on_grid(PI.jittered_fcc(shape, 0.1, seed=2))
    pos[17] -= [64.0, 0.0, 0.0]
    ctx.set_state(pos, np.zeros_like(pos))
    c_gpu, l_gpu = ctx.neighbours(cap=512)
    c_ref, l_ref = oracle.pairs(pos, ctx.potential.rc + ctx.params.skin, cap=512, method="brute")
    assert np.array_equal(c_gpu, c_ref)
    assert sorted_rows(c_gpu, l_gpu) == sorted_rows(c_ref, l_ref)
    ctx.close()


@pytest.mark.parametrize("prec,shape,lanes", [(0, (7, 4, 5), 1), (1, (4, 9, 3), 4), (1, (1, 1, 40), 2),
                                              (0, (40, 1, 3), 16)])
def test_lists_of_crowded_and_far_flung_atoms(P, oracle, prec, shape, lanes):
    # more atoms in a place than a warp holds, atoms spread over the grid's
    # margin and beyond every face of it (counted in the cells at its edge), and
    # atoms one grid step on either side of a cell's edge
    rng = np.random.default_rng(lanes)
    ctx = P.Ctx(shape, T0=0.0, precision=prec, lanes=lanes)
    pos = on_grid(PI.jittered_fcc(shape, 0.2, seed=lanes))
    n = len(pos)
    pick = rng.permutation(n)
    size = 3.615 * np.array(shape)
    crowd, far = pick[:min(48, n // 4)], pick[-min(60, n // 4):]
    pos[crowd] = 0.5 * size + rng.uniform(-0.7, 0.7, (len(crowd), 3))
    pos[far] = rng.uniform(-1.5 * size - 40.0, 2.5 * size + 40.0, (len(far), 3))
    edge = pick[len(crowd):len(crowd) + 8]
    pos[edge, 0] = np.round(pos[edge, 0] / 2.8) * 2.8 + 2.0**-12 * np.tile([-1, 1], 4)
    pos = on_grid(pos)
    ctx.set_state(pos, np.zeros_like(pos))
    c_gpu, l_gpu = ctx.neighbours(cap=512)
    c_ref, l_ref = oracle.pairs(pos, ctx.potential.rc + ctx.params.skin, cap=512, method="brute")
    assert np.array_equal(c_gpu, c_ref)
    assert sorted_rows(c_gpu, l_gpu) == sorted_rows(c_ref, l_ref)
    ctx.close()
