"""List capacities beyond what the list build can hold in shared memory."""
import numpy as np
import pytest

import pta_inputs as PI
from gpu_util import force_error, gpu_package, on_grid, sorted_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


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
