"""List maintenance inside resident batches: members that ask for list builds
and prunings at steps of their own, some in the same pass, against the same
specimens advanced by launched passes, bit for bit and with equal counts.  A
launch then begins with a pruning due for some members (after a build with a
margin wider than the near part; where another member's build, or the limit of
steps per launch, ended the launch before), which every block has to see."""
import numpy as np
import pytest

from gpu_util import gpu_package

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return gpu_package()


def _results(c, a):
    return (c.series().copy(), *c.get_state(), a.rebuilds, a.prunes)


def _equal(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("margin", [0.9, 0.3, 0.02])
def test_members_build_and_prune_at_different_steps(P, prec, margin):
    shapes = [(6, 5, 7), (4, 4, 5), (7, 7, 6), (3, 4, 3), (8, 5, 5)]
    temps, steps = [1200.0, 300.0, 800.0, 2000.0, 100.0], 260
    kw = dict(precision=prec, prune_margin=margin, skin=1.2)
    solo = []
    for i, (sh, T) in enumerate(zip(shapes, temps)):
        c = P.Ctx(sh, T0=T, seed=i, **kw)
        c.set_timing(True)                      # launched passes
        c.apply_strain(1e-3)
        solo.append(_results(c, c.fine_burst(steps)))
        c.close()
    assert len({s[-2] for s in solo}) > 2       # builds at different steps
    assert margin > 0.3 or len({s[-1] for s in solo}) > 2
    cs = [P.Ctx(sh, T0=T, seed=i, **kw) for i, (sh, T) in enumerate(zip(shapes, temps))]
    b = P.Batch(cs)
    b.apply_strain([1e-3] * len(cs))
    for c, a, s in zip(cs, b.fine_burst([steps] * len(cs)), solo):
        _equal(_results(c, a), s)
    b.close()
    for c in cs:
        c.close()


def test_a_pruning_due_at_the_limit_of_steps_per_launch(P):
    # so narrow a margin that every step prunes, 4,000 steps per launch
    out = []
    for timed in (False, True):
        c = P.Ctx((3, 3, 4), T0=30.0, seed=2, precision=1, prune_margin=1e-4)
        c.set_timing(timed)
        out.append(_results(c, c.fine_burst(4030)))
        c.close()
    assert out[0][-1] > 4000
    _equal(out[0], out[1])
