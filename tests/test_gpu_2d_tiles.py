"""The 2D tile kernel at its edges: species sizes around its chunk of 512 slots and its 4-slot
copies; a window that runs over the end of a row; all charge on one node (the largest sums of
the window's 32-bit words) or spread within a cell; particles that leave through a plate, so
that later chunks hold holes, start from one or hold nothing live; one beta for all species
(fixed at compile time) and mixed ones.  As for the other window tests, the potential that each
step leaves is the direct solve of the charge recomputed particle by particle, 1e-11 of its
largest value (roundoff of the two solvers); and the counts add up."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1511_08225_gb300 import binding2d, inputs

pytestmark = pytest.mark.gpu

NX, NY = 64, 20


@pytest.mark.parametrize("n", [1, 3, 4, 5, 511, 512, 513, 2047, 2049])
@pytest.mark.parametrize("where", ["node", "cell", "leaving", "gone"])
@pytest.mark.parametrize("mixed", [False, True])
def test_tile_edges(n, where, mixed):
    prob = inputs.plasma2d_problem(nx=NX, ny=NY, dx=0.5, v0=0.3, ppc=4, dt=1.5, mass_ratio=25.0,
                                   T_i=0.5, source_mode=inputs.SRC_NONE)
    prob["solver"] = "fft"
    if mixed:
        prob["species"][1]["kind"] = inputs.BETA_RELATIVISTIC
    rng = np.random.default_rng(n)
    g = binding2d.Simulation2D(prob)
    for s in range(2):
        m = n if s == 0 else n + 7
        cell = np.full(m, (NY // 2) * NX + NX - 1, np.int32)  # its nodes: the last column and the first
        off = np.zeros((m, 2), np.float32)
        v = np.zeros((m, 3), np.float32)
        if where != "node":
            off[:] = rng.random((m, 2), dtype=np.float32) * np.float32(0.999)
            v[:] = rng.normal(scale=0.2, size=(m, 3))
        if where == "leaving":
            cell[:] = (NY - 1) * NX + rng.integers(0, NX, m)
            v[:, 1] += 0.2
        if where == "gone":
            cell[:] = (NY - 1) * NX + NX - 1
            off[:, 1] = 0.99
            v[:, 1] = 1.0
        g.load(s, cell, off, v)
    g.prepare()
    q = [g.charge_raw(s).sum() for s in range(2)]
    if where == "node":  # at rest: beta = 1, all of it on one node
        assert q == [n << 40, (n + 7) << 40]
    for steps in (1, 1, 3):
        g.step(steps)
        rho, phi, _, _ = g.fields()
        ref = orc.poisson2d_direct(rho, prob["dx"], prob["phi_lo"], prob["phi_hi"])
        assert np.abs(phi - ref).max() <= 1e-11 * max(1.0, np.abs(ref).max())
        d = g.diagnostics()
        for s in range(2):
            live = (g.particles(s)[0] >= 0).sum()
            assert d["count"][s] == live and live + sum(d["absorbed"][s]) == (n if s == 0 else n + 7)
    if where == "gone":
        assert sum(d["absorbed"][0]) > 0
    g.close()
