"""One-launch steps (slpic_step calls of 4 or more steps) with much to do at one place, against the
same steps in calls of 3, which run as the three kernels, bit for bit: sources on both sides of
the line from which the CTAs make them in shares (2,048 particles a step, all species), with one
to four species, a full store and a barrier that gives up; and more pushes that need the walk
than a CTA's list of 512 holds."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding, inputs
from test_gpu_steps import _by_threes, _pair, _random, _same, _with_species

pytestmark = pytest.mark.gpu


def _rate(prob, per_step):
    """A rate source of per_step particles a step of every species."""
    w = prob["species"][0]["w"]
    for sp in prob["species"]:
        sp["w"] = w
    prob["source"].update(mode=inputs.SRC_RATE, rate=per_step * w / prob["dt"])
    return prob


def _sheath(n_cells, species=2, capacity=120000):
    prob = _with_species(inputs.sheath_problem(n_cells=n_cells, ppc=50, v0=0.1), species)
    prob["source"]["ref_species"] = 0
    for sp in prob["species"]:
        sp["capacity"] = capacity
    return prob


@pytest.mark.parametrize("species,per_step", [(1, 2047.5), (1, 2048.5), (2, 1024.0), (2, 1025.0), (2, 6000.5),
                                              (3, 700.25), (4, 513.0)])
@pytest.mark.parametrize("n_cells,every", [(64, 4), (1500, 16)])
def test_rate_sources_on_both_sides_of_the_line(n_cells, every, species, per_step):
    prob = _rate(_sheath(n_cells, species), per_step)
    a, b = _pair(prob, _random(prob, [4000] * species), every)
    for n in (5, 8):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
    assert a.diagnostics()["injected"][0] >= int(12 * per_step)
    a.close()
    b.close()


@pytest.mark.parametrize("periodic_profile", [False, True])
def test_a_strong_wall_source(periodic_profile):
    prob = inputs.paper_sheath_problem(ppc=30000, v0=0.05, capacity_factor=0.2)
    if periodic_profile:
        prob["v0_profile"] = 0.5 + 0.5 * np.linspace(0.0, 1.0, prob["n_cells"])
    a, b = _pair(prob, inputs.empty_state(prob))
    for n in (6, 19):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
    assert sum(a.diagnostics()["injected"][:2]) > 25 * 2048
    a.close()
    b.close()


def test_a_source_that_no_longer_fits():
    prob = _rate(_sheath(200, capacity=40000), 3000.0)
    a, b = _pair(prob, _random(prob, [2000, 3000]))
    codes = []
    for sim, go in ((a, a.step), (b, lambda n: _by_threes(b, n))):
        go(24)
        with pytest.raises(binding.SlpicError) as err:
            sim.synchronize()
        codes.append(err.value.code)
    assert codes == [binding.SLPIC_ERR_CAPACITY] * 2
    _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("limit", [100, 3000, 6000, 12000, 24000])
def test_a_barrier_that_gives_up_beside_a_source_in_shares(limit):
    prob = _rate(_sheath(256, capacity=300000), 2000.0)
    a, b = _pair(prob, _random(prob, [40000, 40000]), 5)
    binding.slpic_set_wait_limit(a.h, limit)
    a.step(100)
    try:
        a.synchronize()
        assert limit > 100 and a.diagnostics()["step"] == 100
    except binding.SlpicError as e:
        assert e.code == binding.SLPIC_ERR_TIMEOUT
    binding.slpic_set_wait_limit(a.h, 0)
    _by_threes(b, a.diagnostics()["step"])
    for n in (0, 10):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
    a.close()
    b.close()


def test_more_walks_than_the_list_holds():
    prob = inputs.sheath_problem(n_cells=50, ppc=20000, v0=0.3, kind=inputs.BETA_RELATIVISTIC, mass_ratio=4.0)
    prob["phi_hi"] = 60.0
    a, b = _pair(prob, _random(prob, [1_000_000, 1_000_000]))
    a.step(1)
    b.step(1)
    walks = [sum(a.diagnostics()["iterative"])]
    for n in (4, 6):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
        walks.append(sum(a.diagnostics()["iterative"]))
    assert (walks[-1] - walks[0]) / 10 > 1.5 * 512 * 151  # a step, beyond all the lists
    a.close()
    b.close()
