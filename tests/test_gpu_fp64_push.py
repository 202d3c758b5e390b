"""The FP64 form's push where its branches meet, against the oracle's quadrature: one step
of test particles (of negligible charge) in the uniform field of two biased plates, at
field strengths that put the series parameter |a| dt v0 / |v|^2 on both sides of its
limit 0.02 and the step across the band |v| <= v0, for speeds from inside the band to far
above it, along and against the field.  Counts around the 128-particle tile.  The bar is
that of test_gpu_fp64.py (1e-9 of |v|; the oracle's quadrature is the looser side)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1511_08225_gb300 import binding, inputs

from _match import match
from test_gpu_fp64 import _key64

pytestmark = pytest.mark.gpu

HEAV, REL = inputs.BETA_HEAVISIDE, inputs.BETA_RELATIVISTIC


@pytest.mark.parametrize("kind", [HEAV, REL])
@pytest.mark.parametrize("field,n", [(1e-4, 1), (2e-3, 127), (4e-3, 128), (0.05, 129), (1.0, 257)])
def test_push_branches_match_oracle(kind, field, n):
    v0 = 0.3
    prob = inputs.sheath_problem(n_cells=16, ppc=8, v0=v0, kind=kind, source_mode=inputs.SRC_NONE)
    prob["phi_hi"] = -field * prob["n_cells"] * prob["dx"]
    for sp in prob["species"]:
        sp["w"] = 1e-12
        sp["m"] = 1.0
        sp["capacity"] = 1024
    rng = np.random.default_rng(n)
    speed = v0 * 10.0 ** rng.uniform(-1.5, 1.0, n)
    speed[::4] = v0 * (1.0 + rng.uniform(-0.05, 0.05, speed[::4].size))  # about the band's edge
    u = rng.normal(size=(n, 3))
    u[1::3, 1:] *= 1e-3  # nearly along the field
    v = speed[:, None] * u / np.linalg.norm(u, axis=1, keepdims=True)
    x = rng.uniform(4.0, 12.0, n) * prob["dx"]
    g, o = binding.SimulationFP64(prob), orc.OracleSim(prob)
    for s in range(2):
        g.load(s, x, v)
        o.load(s, x, v)
    g.prepare()
    o.start()
    g.step(1)
    o.step(1)
    for s in range(2):
        xg, vg = g.particles(s)
        ia, ib = match(_key64(o.v[s]), _key64(vg))
        assert ia.size == xg.size == n
        vn = np.linalg.norm(o.v[s][ia], axis=1)
        assert (np.linalg.norm(vg[ib] - o.v[s][ia], axis=1) <= 1e-9 * vn).all()
    g.close()
