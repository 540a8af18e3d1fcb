"""The activity mask is built when a state is uploaded.  What can leave an unmarked node with a DOM below zero later
(an implicit solve, a negative FOM or SOM beside it, a step at the stability bound), and values that are
not finite, must give the same bits whether a small graph's step calls run as one launch or as launches per pass
(which run while kernel timing is on)."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

SHAPES = [(9, 11, 13), (40, 44, 52), (64, 64, 76)]  # 1, 2 and 4 nodes per thread


def _state(n, seed=5):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand((5, n), generator=g, device="cuda", dtype=torch.float64) * 2e-4
    marked = torch.rand(n, generator=g, device="cuda") < 0.05
    for c in (0, 2, 3, 4):
        X[c] = torch.where(marked, X[c], 0.0)
    X[1] = torch.where(torch.rand(n, generator=g, device="cuda") < 0.1, X[1], 0.0)
    return X, marked


def _both(shape, run):
    """run(sim, marked nodes, X) in both forms: the states after it."""
    g, out = vga.Graph(np.zeros(shape, dtype=np.uint8)), []
    for timing in (False, True):
        X, marked = _state(g.n)
        sim = vga.Sim(g, synth.paper_params())
        sim.enable_timing(timing)
        run(sim, marked, X)
        out.append(sim.get_masses())
        sim.close()
    g.close()
    assert np.array_equal(out[0], out[1], equal_nan=True)
    return out[0]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("transform", [0, 1])
def test_explicit_after_an_implicit_solve(shape, transform):
    def run(sim, marked, X):
        p = synth.paper_params()
        X[1] = 0.0
        sim.set_masses(X)
        sim.step(3)
        X[3] = torch.where(marked, -1e-3, 0.0)  # negative stocks: the solve spreads their negative DOM
        sim.set_masses(X)
        sim.step(2)
        sim.set_params(dict(p, scheme=vga.VGA_SCHEME_IMPLICIT_PCG, dt=10 * p["dt"]))
        sim.step(1)
        Y = sim.get_masses()
        assert (Y[1][~marked.cpu().numpy()] < 0).any()
        sim.set_params(dict(p, transform=transform))
        for k in (2, 3, 2):
            sim.step(k)

    _both(shape, run)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("comp", [2, 3])
def test_negative_stocks_feed_the_neighbours(shape, comp):
    def run(sim, marked, X):
        X[1] = 0.0
        X[comp] = torch.where(marked, -1e-3, 0.0)
        sim.set_masses(X)
        for k in (4, 2, 3):
            sim.step(k)

    Y = _both(shape, run)
    assert (Y[0] < 0).any()


@pytest.mark.parametrize("shape", SHAPES)
def test_steps_at_the_bound_then_below_it(shape):
    def run(sim, marked, X):
        p = synth.paper_params()
        X[1] = torch.where(X[1] > 1e-4, 1.0, 0.0)
        sim.set_params(dict(p, dt=1.0 / (6.0 * p["D"])))
        sim.set_masses(X)
        sim.step(5)
        sim.set_params(p)
        sim.step(4)
        sim.step(3)

    _both(shape, run)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_values_that_are_not_finite(shape, value):
    def run(sim, marked, X):
        at = int((~marked).nonzero()[7])
        X[1, at] = value
        sim.set_masses(X)
        sim.step(3)
        sim.step(2)

    Y = _both(shape, run)
    assert np.isnan(Y).any()
