"""The batched kernels' division of work at its edges: instances of very different size in one
batch (parts that span several instances, instances that span several parts), a species without
particles (its source fills it), one with a single particle, a grid with no room for the staged
kernel's ring beside it, another beta and a periodic grid, and more instances than the walk
kernel takes at a time.  Every instance gives exactly what it gives alone."""
import numpy as np
import pytest

from paper_1511_08225_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def _sheath(cells, ppc, kind=inputs.BETA_HEAVISIDE, v0=0.05):
    return inputs.sheath_problem(n_cells=cells, ppc=ppc, v0=v0, kind=kind)


def _alone(prob, state, steps):
    s = binding.Simulation(prob)
    s.load_state(state)
    s.prepare()
    s.step(steps)
    out = (s.diagnostics(), [s.charge_raw(k) for k in range(2)], [s.particles(k) for k in range(2)], s.fields())
    s.close()
    return out


def _sorted(c, o, v):
    key = np.lexsort((v[:, 2], v[:, 1], v[:, 0], o, c))
    return c[key], o[key], v[key]


def _check(probs, states, steps, which):
    b = binding.Batch(probs)
    for i, st in enumerate(states):
        b.load_state(i, st)
    b.prepare()
    b.step(steps)
    b.synchronize()
    for i in which:
        d, q, x, f = _alone(probs[i], states[i], steps)
        e = b.diagnostics(i)
        assert e["count"] == d["count"] and e["absorbed"] == d["absorbed"] and e["injected"] == d["injected"]
        for s in range(2):
            assert np.array_equal(b.charge_raw(i, s), q[s])
            for u, w in zip(_sorted(*b.particles(i, s)), _sorted(*x[s])):
                assert np.array_equal(u, w)
        assert np.array_equal(b.fields(i)[2], f[2])
    b.close()


@pytest.mark.parametrize("cells", [64, 12000, 15000])
def test_uneven_instances(cells):
    probs = [_sheath(32, 3), _sheath(cells, 40), _sheath(100, 900), _sheath(48, 1, inputs.BETA_RELATIVISTIC),
             inputs.periodic_problem(n_cells=128, ppc=200, v0=0.1)]
    states = [inputs.load_state(p) for p in probs]
    none = tuple(a[:0] for a in states[0][0])
    states[0] = [none, tuple(a[:1] for a in states[0][1])]  # no electrons, one ion
    _check(probs, states, 18, range(len(probs)))  # past a compacting step


def test_more_instances_than_a_group_of_the_walk_kernel():
    probs = [_sheath(16 + i % 7, 4 + i % 5, v0=0.02 + 0.001 * (i % 11)) for i in range(300)]
    states = [inputs.load_state(p) for p in probs]
    _check(probs, states, 17, (0, 1, 127, 255, 256, 257, 299))
