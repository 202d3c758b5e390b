"""Many steps in one launch (slpic_step calls of 4 or more steps) against the same steps in
calls of 3, which run as the three kernels: particles, deposits, fields, counters and
errors bit for bit, at the sizes where the launch's split and its sums can go wrong: no
particles, fewer than a warp, a warp and one, one and four species, two cells, node counts
above one per thread, every beta kind, a profile, every source, intervals of compaction
from 2, a full store, and more steps than one launch takes."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding, inputs

pytestmark = pytest.mark.gpu

ONE, HEAV, REL = inputs.BETA_ONE, inputs.BETA_HEAVISIDE, inputs.BETA_RELATIVISTIC


def _sorted(c, o, v):
    k = np.lexsort((v[:, 2].view(np.uint32), v[:, 1].view(np.uint32), v[:, 0].view(np.uint32),
                    o.view(np.uint32), c))
    return c[k], o[k], v[k]


def _same(a, b):
    da, db = a.diagnostics(), b.diagnostics()
    for k in ("step", "count", "absorbed", "injected", "iterative", "field_energy"):
        assert da[k] == db[k], k
    for x, y in zip(a.fields(), b.fields()):
        assert np.array_equal(x, y)
    for s in range(a.ns):
        assert np.array_equal(a.charge_raw(s), b.charge_raw(s))
        for x, y in zip(_sorted(*a.particles(s)), _sorted(*b.particles(s))):
            assert np.array_equal(x, y)


def _by_threes(sim, n):
    while n:
        k = min(3, n)
        sim.step(k)
        n -= k


def _pair(prob, state, every=16):
    sims = [binding.Simulation(prob) for _ in range(2)]
    for sim in sims:
        binding.slpic_set_tuning(sim.h, compact_every=every)
        sim.load_state(state)
        sim.prepare()
    return sims


def _random(prob, counts, seed=7):
    rng = np.random.default_rng(seed)
    return [inputs.random_state(rng, n, prob["n_cells"], vscale=sp["vth"])
            for n, sp in zip(counts, prob["species"])]


def _with_species(prob, n):
    prob["species"] = [dict(prob["species"][k % 2], w=prob["species"][k % 2]["w"] / (n // 2 or 1))
                       for k in range(n)]
    prob["source"]["ref_species"] = n - 1
    return prob


@pytest.mark.parametrize("counts", [(0, 0), (1, 0), (31, 33), (32, 1), (70, 4801), (40000, 39999)])
@pytest.mark.parametrize("kind,periodic", [(HEAV, False), (REL, False), (HEAV, True), (ONE, True)])
def test_counts_and_shapes(kind, periodic, counts):
    prob = (inputs.periodic_problem(n_cells=64, ppc=800, kind=kind) if periodic else
            inputs.sheath_problem(n_cells=65, ppc=800, v0=0.2, kind=kind))
    if not periodic:
        prob["phi_hi"] = 3.0
    a, b = _pair(prob, _random(prob, counts))
    for n in (4, 17, 23):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("n_cells,species,every", [(2, 2, 2), (3, 1, 5), (1023, 4, 16), (1024, 2, 3), (3000, 3, 16)])
def test_grids_species_and_intervals(n_cells, species, every):
    prob = _with_species(inputs.sheath_problem(n_cells=n_cells, ppc=max(4, 20000 // n_cells), v0=0.1,
                                               capacity_factor=3.0), species)
    if n_cells < 8:  # the source band must lie inside the grid
        prob["source"].update(lo_cells=0.5, len_cells=0.75)
    a, b = _pair(prob, _random(prob, [prob["species"][0]["ppc"] * n_cells] * species), every)
    for n in (every + 4, 20):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("kind", [ONE, HEAV, REL])
def test_wall_source_from_an_empty_box_with_a_profile(kind):
    prob = inputs.paper_sheath_problem(kind=kind, ppc=200, v0=0.05)
    if kind != ONE:
        prob["v0_profile"] = 0.5 + 0.5 * np.linspace(0.0, 1.0, prob["n_cells"])
    a, b = _pair(prob, inputs.empty_state(prob))
    for n in (4, 90, 61):
        a.step(n)
        _by_threes(b, n)
        _same(a, b)
    a.close()
    b.close()


def test_rate_source_and_a_full_store():
    prob = inputs.sheath_problem(n_cells=128, ppc=40, v0=0.2, source_mode=inputs.SRC_RATE, rate=30.0,
                                 capacity_factor=1.3)
    a, b = _pair(prob, inputs.load_state(prob))
    for k in range(20):  # until the source no longer fits
        codes = []
        for sim, go in ((a, a.step), (b, lambda n: _by_threes(b, n))):
            go(8)
            try:
                sim.synchronize()
                codes.append(0)
            except binding.SlpicError as e:
                codes.append(e.code)
        assert codes[0] == codes[1]
        _same(a, b)
        if codes[0]:
            break
    assert codes[0] == binding.SLPIC_ERR_CAPACITY
    a.close()
    b.close()


def test_more_steps_than_a_launch_takes():
    prob = inputs.periodic_problem(n_cells=16, ppc=20)
    a, b = _pair(prob, inputs.load_state(prob))
    a.step(4103)
    _by_threes(b, 4103)
    _same(a, b)
    a.close()
    b.close()
