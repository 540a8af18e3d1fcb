"""A step call transforms every node first, then (sparse passes) only the marked ones.  What the first
transformation gave an unmarked node is part of the state after the call: a negative DOM there moves to the biomass
whatever the number of steps, and no mass is lost."""
import numpy as np
import pytest

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

AT = 100
LOSS = np.float32(-1e-6)


def _state(n):
    X = synth.random_masses(n, 7, density=0.02)
    X[:, AT] = 0.0
    X[1, AT] = LOSS
    return X


def _check(X, Y):
    assert Y[0, AT] == LOSS
    # 20 transformations and diffusions of values rounded to 2^-32 of themselves (FP32 with a 16-bit residual)
    assert abs(Y.sum() - X.sum()) <= 20 * 2.0 ** -32 * np.abs(X).sum()


@pytest.mark.parametrize("n_steps", [2, 3, 4, 7])
@pytest.mark.parametrize("variant", [5, 6])
def test_simulation(n_steps, variant):
    g = vga.Graph(np.zeros((12, 14, 16), dtype=np.uint8))
    X = _state(g.n)
    sim = vga.Sim(g, synth.paper_params())
    sim.set_kernel(variant, 1024)
    sim.enable_timing(True)  # launches per pass
    sim.set_masses(X)
    sim.step(n_steps)
    _check(X, sim.get_masses())
    sim.close()
    g.close()


@pytest.mark.parametrize("n_steps", [2, 3, 4, 7])
@pytest.mark.parametrize("shape", [(1, 0), (3, 1)])
def test_batch(n_steps, shape):
    """Launches per pass, and persistent ones of three passes."""
    graphs = [vga.Graph(np.zeros(s, dtype=np.uint8)) for s in ((12, 14, 16), (9, 10, 11))]
    b = vga.Batch(graphs, [synth.paper_params()] * 2)
    b.set_launch(*shape)
    X = [_state(g.n) for g in graphs]
    for k in range(2):
        b.set_masses(k, X[k])
    b.step(n_steps)
    for k in range(2):
        Y = b.get_masses(k)
        _check(X[k], Y)
        sim = vga.Sim(graphs[k], synth.paper_params())
        sim.set_masses(X[k])
        sim.step(n_steps)
        assert np.array_equal(sim.get_masses(), Y)
        sim.close()
    b.close()
    for g in graphs:
        g.close()
