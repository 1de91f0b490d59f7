"""A resident run whose grid barriers run out of polls (the limit set to 0, so
that every block gives up at its first barrier): the call reports PTA_ECUDA,
and whatever would use the specimens' states afterwards is refused, through
their own runners, the batch and a new batch alike."""
import pytest

from gpu_util import gpu_package

pytestmark = pytest.mark.gpu

ECUDA, EINVAL = -3, -1


@pytest.fixture(scope="module")
def P():
    return gpu_package()


def _refused(P, call, status=ECUDA):
    with pytest.raises(P.PTAError) as e:
        call()
    assert e.value.status == status


def _all_refused(P, c):
    for call in (c.get_state, c.series, c.flags, c.forces, c.neighbours, c.coarse_step, c.save,
                 lambda: c.apply_strain(1e-3), lambda: c.fine_burst(5),
                 lambda: c.ramp_burst(5, 1e-5), lambda: c.relax(5, 10, 1.0)):
        _refused(P, call)
    _refused(P, lambda: P.Batch([c]), EINVAL)


# a resident run, a sweep
@pytest.mark.parametrize("prec,shape", [(1, (4, 4, 5)), (0, (4, 4, 5)), (1, (19, 20, 21)),
                                        (0, (11, 13, 24))])
@pytest.mark.parametrize("call", ["fine_burst", "ramp_burst", "coarse_step", "relax"])
def test_alone(P, monkeypatch, prec, shape, call):
    c = P.Ctx(shape, T0=300.0, seed=1, precision=prec, burst_steps=20)
    monkeypatch.setenv("PTA_BARRIER_POLLS", "0")
    _refused(P, {"fine_burst": lambda: c.fine_burst(20), "ramp_burst": lambda: c.ramp_burst(20, 1e-5),
                 "coarse_step": c.coarse_step, "relax": lambda: c.relax(20, 40, 1.0)}[call])
    _all_refused(P, c)
    c.close()
    monkeypatch.delenv("PTA_BARRIER_POLLS")
    d = P.Ctx(shape, T0=300.0, seed=1, precision=prec)      # the device is well
    assert d.fine_burst(20).nsteps == 20
    d.close()


@pytest.mark.parametrize("call", ["fine_burst", "coarse_step", "tick"])
def test_in_a_batch(P, monkeypatch, call):
    cs = [P.Ctx((4, 4, 5), T0=300.0, seed=i, precision=1, burst_steps=20) for i in range(3)]
    cs[1].fine_burst(10)                                    # has a runner of its own
    monkeypatch.setenv("PTA_BARRIER_POLLS", "0")
    b = P.Batch(cs)
    monkeypatch.delenv("PTA_BARRIER_POLLS")
    calls = {"fine_burst": lambda: b.fine_burst([20] * 3), "coarse_step": b.coarse_step, "tick": b.tick}
    _refused(P, calls[call])
    for f in (*calls.values(), lambda: b.apply_strain([1e-3] * 3)):
        _refused(P, f)
    for c in cs:
        _all_refused(P, c)
    b.close()
    for c in cs:
        c.close()


@pytest.mark.parametrize("text", ["", "many", "12x"])
def test_a_limit_that_is_no_number_is_none(P, monkeypatch, text):
    monkeypatch.setenv("PTA_BARRIER_POLLS", text)
    c = P.Ctx((4, 4, 5), T0=300.0, seed=1, precision=1)
    assert c.fine_burst(20).nsteps == 20
    c.close()
