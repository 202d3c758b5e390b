"""The direct 2D solver at every period it takes (nx = 2 .. 8,192: each first pass of the
transform, each width of a row, one or three levels of butterflies at a time) and at row counts
on both sides of its lines: one interior row, fewer rows than segments, empty segments at the
top, segments of one batch of 8 rows and more, and more rows than shared memory holds (3,500).  Against
the oracle's direct solve (plain DFT, Thomas): FP64's rounding times the condition number of the
5-point operator, at least the 1e-12 the other sizes are held to; and a second solve of the
same charge gives the same bits."""
import math

import numpy as np
import pytest

from oracle import oracle as orc
from paper_1511_08225_gb300 import binding2d, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [
    (2, 2), (2, 3300), (2, 9000), (4, 2), (4, 33), (4, 34), (8, 257), (8, 258), (16, 65), (32, 3), (32, 1025),
    (64, 1026), (128, 64), (256, 512), (256, 514), (512, 250), (512, 260), (1024, 128), (1024, 130),
    (2048, 40), (2048, 70), (4096, 5), (4096, 40), (8192, 3), (8192, 20)])
def test_every_period_and_row_count(nx, ny):
    prob = inputs.plasma2d_problem(nx=nx, ny=ny, ppc=1, seed=1, solver="fft")
    prob["phi_lo"], prob["phi_hi"] = 0.7, -0.2
    for sp in prob["species"]:
        sp["capacity"] = 64
    sim = binding2d.Simulation2D(prob)
    rng = np.random.default_rng(nx + ny)
    rho = 0.2 * rng.normal(size=(ny + 1, nx)) + 0.1 * np.sin(np.pi * np.arange(ny + 1) / ny)[:, None]
    phi, it, res = sim.solve_poisson(rho)
    ref = orc.poisson2d_direct(rho, prob["dx"], 0.7, -0.2)
    cond = 8.0 / (4.0 * math.sin(math.pi / (2 * ny)) ** 2)
    tol = max(1e-12, 2.3e-16 * cond)
    assert it == 0 and np.abs(phi - ref).max() <= tol * np.abs(ref).max()
    assert (phi[0] == 0.7).all() and (phi[-1] == -0.2).all()
    assert np.array_equal(phi, sim.solve_poisson(rho)[0])
    sim.close()
