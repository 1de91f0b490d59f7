"""Cell grids whose cells are divided along x (specimens that fill them) and grids
that are not (thin specimens, whose grid is mostly empty): neighbour lists
against brute force with crowded atoms, atoms on cell edges and atoms beyond
the grid, and forces against the oracle."""
import numpy as np
import pytest

import pta_inputs as PI
from gpu_util import force_error, gpu_package, on_grid, sorted_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


@pytest.mark.parametrize("prec,shape,lanes", [(0, (11, 12, 10), 4), (1, (14, 9, 13), 1),
                                              (1, (10, 11, 10), 16), (0, (120, 2, 3), 2),
                                              (1, (3, 60, 3), 8)])
def test_lists_of_divided_and_undivided_cells(P, oracle, prec, shape, lanes):
    rng = np.random.default_rng(lanes)
    ctx = P.Ctx(shape, T0=0.0, precision=prec, lanes=lanes)
    pos = on_grid(PI.jittered_fcc(shape, 0.2, seed=lanes))
    n = len(pos)
    f, pe, _ = (ctx.set_state(pos, np.zeros_like(pos)), ctx.forces())[1]
    f_ref, pe_ref, _ = oracle.eam(pos, oracle.Potential(
        eps=ctx.potential.eps, c=ctx.potential.c, a=ctx.potential.a, rc=ctx.potential.rc, n=7, m=6))
    assert force_error(f, f_ref) < (1e-10 if prec == 0 else 1e-5)
    assert np.max(np.abs(pe - pe_ref) / np.abs(pe_ref)) < (1e-11 if prec == 0 else 1e-5)
    pick = rng.permutation(n)
    size = 4.05 * np.array(shape)
    crowd, far, edge = pick[:48], pick[48:120], pick[120:184]
    pos[crowd] = 0.5 * size + rng.uniform(-0.7, 0.7, (48, 3))
    reach = 0.25 * size.max() + 25.0
    pos[far] = rng.uniform(-reach - 15.0, size + reach + 15.0, (72, 3))
    if prec == 1:
        pos[far] = np.clip(pos[far], -500.0, 500.0)
    pos[edge, 0] = np.round(pos[edge, 0] / 2.525) * 2.525 + 2.0**-12 * np.tile([-1, 1], 32)
    pos = on_grid(pos)
    ctx.set_state(pos, np.zeros_like(pos))
    c_gpu, l_gpu = ctx.neighbours(cap=512)
    c_ref, l_ref = oracle.pairs(pos, ctx.potential.rc + ctx.params.skin, cap=512, method="brute")
    assert np.array_equal(c_gpu, c_ref)
    assert sorted_rows(c_gpu, l_gpu) == sorted_rows(c_ref, l_ref)
    ctx.close()
