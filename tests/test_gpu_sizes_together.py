"""Simulations of several sizes alive at once.  A kernel's limit of dynamic shared memory belongs
to the kernel, not to a handle: creating a small simulation must leave a larger live one what
its launches need.  The larger one is made first, the smaller second; both then give what each
gives alone."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding, binding2d, inputs

pytestmark = pytest.mark.gpu


def _direct(nx, ny):
    prob = inputs.plasma2d_problem(nx=nx, ny=ny, ppc=2, seed=3, solver="fft", v0=0.2)
    sim = binding2d.Simulation2D(prob)
    sim.load_state(inputs.load_state2d(prob))
    return sim


def _direct_run(sim, rho):
    sim.prepare()
    sim.step(2)
    return [*sim.fields(), sim.solve_poisson(rho)[0]]


# the mode solves' values in shared memory by the rows, the transforms' row by the width
@pytest.mark.parametrize("large,small", [((64, 1024), (64, 600)), ((8192, 4), (4096, 4)), ((8192, 40), (4096, 40))])
def test_direct_solver_with_a_smaller_grid_beside_it(large, small):
    rng = np.random.default_rng(1)
    rho = [rng.normal(size=(ny + 1, nx)) for nx, ny in (large, small)]
    sims = [_direct(*large), _direct(*small)]
    got = [_direct_run(s, r) for s, r in zip(sims, rho)]
    for s in sims:
        s.close()
    for size, r, mine in zip((large, small), rho, got):
        alone = _direct(*size)
        for a, b in zip(mine, _direct_run(alone, r)):
            assert np.array_equal(a, b)
        alone.close()


def _batch_run(b, probs, states):
    for i, st in enumerate(states):
        b.load_state(i, st)
    b.prepare()
    b.step(18)  # past a compacting step
    out = [f for i in range(len(probs)) for f in b.fields(i)]
    b.close()
    return out


# in place: the staged kernel beside 11,000 nodes, the per-warp kernel at 15,000
@pytest.mark.parametrize("cells", [11000, 15000])
def test_batch_with_a_smaller_batch_beside_it(cells):
    probs = [[inputs.sheath_problem(n_cells=n, ppc=20, v0=0.05) for n in sizes] for sizes in ((cells, 70), (60, 50))]
    states = [[inputs.load_state(p) for p in ps] for ps in probs]
    batches = [binding.Batch(ps) for ps in probs]
    got = [_batch_run(*a) for a in zip(batches, probs, states)]
    for ps, st, mine in zip(probs, states, got):
        for a, b in zip(mine, _batch_run(binding.Batch(ps), ps, st)):
            assert np.array_equal(a, b)


def test_fp64_form_with_a_smaller_grid_beside_it():
    probs = [inputs.sheath_problem(n_cells=n, ppc=4, v0=0.1) for n in (9000, 64)]
    states = [inputs.load_state(p) for p in probs]
    sims = [binding.SimulationFP64(p) for p in probs]
    for sim, prob, state in zip(sims, probs, states):
        for s, st in enumerate(state):
            sim.load_cells(s, *st)
        sim.prepare()
        sim.step(3)
        rho = sim.fields()[0]
        assert np.isfinite(rho).all() and rho.size == prob["n_cells"] + 1
        assert sum(sim.count(s) for s in range(2)) > 0
        sim.close()
