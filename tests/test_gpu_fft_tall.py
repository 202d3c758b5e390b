"""The direct 2D solver with three levels of butterflies a pass on narrow, tall grids: rows with
fewer points than a thread holds (nx = 2 and 4, whose first heights on that side of the line are
65,537 and 32,769), as many (8), and several rows to a CTA (8 to 128).  Against the oracle's
direct solve, to FP64's rounding times the condition number of the 5-point operator.  That
rounding also bounds the residual, so the residual target is loose here."""
import math

import numpy as np
import pytest

from oracle import oracle as orc
from paper_1511_08225_gb300 import binding2d, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 65537), (2, 65540), (4, 32769), (4, 32772), (8, 16385), (8, 16400),
                                   (16, 8200), (32, 4100), (64, 2060), (128, 1030)])
def test_narrow_rows(nx, ny):
    prob = inputs.plasma2d_problem(nx=nx, ny=ny, ppc=1, seed=1, solver="fft", cg_rtol=1e-4)
    prob["phi_lo"], prob["phi_hi"] = 0.7, -0.2
    for sp in prob["species"]:
        sp["capacity"] = 64
    sim = binding2d.Simulation2D(prob)
    rng = np.random.default_rng(nx + ny)
    rho = 0.2 * rng.normal(size=(ny + 1, nx)) + 0.1 * np.sin(np.pi * np.arange(ny + 1) / ny)[:, None]
    phi, it, _ = sim.solve_poisson(rho)
    ref = orc.poisson2d_direct(rho, prob["dx"], 0.7, -0.2)
    cond = 8.0 / (4.0 * math.sin(math.pi / (2 * ny)) ** 2)
    assert it == 0 and np.abs(phi - ref).max() <= max(1e-12, 2.3e-16 * cond) * np.abs(ref).max()
    sim.close()
