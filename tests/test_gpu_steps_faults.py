"""A grid barrier of the one-launch steps (slpic_step calls of 4 or more steps) that gives up,
by a wait limit far below an L2 round trip.  The launch ends at a whole step, all CTAs the same
one: the error is reported, the handle stands at that step with that step's particles,
deposits and counters, and steps on from there like a run that was never cut short."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def _sim(prob, every):
    sim = binding.Simulation(prob)
    binding.slpic_set_tuning(sim.h, compact_every=every)
    sim.load_state(inputs.load_state(prob))
    sim.prepare()
    return sim


def _sorted(c, o, v):
    k = np.lexsort((v[:, 2], v[:, 1], v[:, 0], o, c))
    return c[k], o[k], v[k]


def _same(a, b):
    da, db = a.diagnostics(), b.diagnostics()
    for k in ("step", "count", "absorbed", "injected", "field_energy"):
        assert da[k] == db[k], k
    for s in range(a.ns):
        assert np.array_equal(a.charge_raw(s), b.charge_raw(s))
        for x, y in zip(_sorted(*a.particles(s)), _sorted(*b.particles(s))):
            assert np.array_equal(x, y)
    for x, y in zip(a.fields(), b.fields()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("every,before,steps", [(16, 6, 64), (2, 5, 9000)])
def test_a_barrier_that_gives_up_ends_the_launch_at_a_whole_step(every, before, steps):
    prob = inputs.sheath_problem(n_cells=256, ppc=300, v0=0.05)
    sim, twin = _sim(prob, every), _sim(prob, every)
    sim.step(before)
    sim.synchronize()
    binding.slpic_set_wait_limit(sim.h, 100)
    sim.step(steps)
    with pytest.raises(binding.SlpicError) as err:
        sim.synchronize()
    assert err.value.code == binding.SLPIC_ERR_TIMEOUT
    sim.synchronize()  # reported once
    at = sim.diagnostics()["step"]
    assert before <= at < before + steps  # cut short
    binding.slpic_set_wait_limit(sim.h, 0)
    twin.step(at)
    _same(sim, twin)
    for n in (20, 3):
        sim.step(n)
        twin.step(n)
        _same(sim, twin)
    sim.close()
    twin.close()


@pytest.mark.parametrize("limit", [1500, 3000, 6000, 12000, 24000])
def test_limits_about_as_long_as_the_waits(limit):
    """Waits that run out after some steps, or never: the handle stands at a whole step."""
    prob = inputs.sheath_problem(n_cells=256, ppc=300, v0=0.05)
    sim, twin = _sim(prob, 5), _sim(prob, 5)
    binding.slpic_set_wait_limit(sim.h, limit)
    sim.step(400)
    try:
        sim.synchronize()
        assert sim.diagnostics()["step"] == 400
    except binding.SlpicError as e:
        assert e.code == binding.SLPIC_ERR_TIMEOUT
    at = sim.diagnostics()["step"]
    twin.step(at)
    _same(sim, twin)
    sim.close()
    twin.close()


def test_a_limit_that_no_wait_reaches_changes_nothing():
    prob = inputs.sheath_problem(n_cells=128, ppc=100, v0=0.1)
    sim, twin = _sim(prob, 16), _sim(prob, 16)
    binding.slpic_set_wait_limit(sim.h, 200_000_000)
    sim.step(40)
    twin.step(40)
    _same(sim, twin)
    sim.close()
    twin.close()
