"""Simulations of several sizes alive at once.  A kernel's limit of dynamic shared memory belongs
to the kernel, not to a handle: creating a small simulation must leave a larger live one what
its launches need.  The larger one is made first, the smaller second; both then give what each
gives alone."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding2d, inputs

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
