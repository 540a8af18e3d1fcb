"""Step calls and adjoint segments of small graphs run as one cooperative launch each.  At the edges of its
shapes (512 threads x 1, 2 or 4 nodes, one block per SM) the states and adjoints must be the bits of
the launch-per-pass kernels, which run while kernel timing is on, and so must the gradients of a sweep with
dL/dX^0; the others, whose sums take the nodes in another order in compensated pairs (about 45 bits),
agree to 1e-10 unless a sum cancels by more than a factor 1000."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

# nodes: 1, 511, 512, 513; around the largest graph of 1, 2 and 4 nodes per thread on 152 SMs; and odd masks
BOXES = [(1, 1, 1), (1, 7, 73), (8, 8, 8), (1, 19, 27), (32, 32, 76), (31, 37, 69), (38, 64, 64), (43, 53, 69), (64, 64, 76),
         (67, 67, 70)]


def _image(shape, porosity):
    if porosity >= 1.0:
        return np.zeros(shape, dtype=np.uint8)
    return synth.pore_mask(shape, porosity, seed=3)


def _state(n, density, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand((5, n), generator=g, device="cuda", dtype=torch.float64) * 2e-4
    marked = torch.rand(n, generator=g, device="cuda") < density
    for c in (0, 2, 3, 4):
        X[c] = torch.where(marked, X[c], 0.0)
    X[1] = torch.where(torch.rand(n, generator=g, device="cuda") < 0.3, X[1], 0.0)
    return X


def _theta(shape, blocks):
    if not blocks:
        return None
    return synth.block_conductances(tuple(-(-s // 4) for s in shape), seed=3, spread=0.09).astype(np.float32)


@pytest.mark.parametrize("shape", BOXES)
@pytest.mark.parametrize("density,transform,blocks", [(0.0, 0, False), (0.05, 0, False), (0.2, 1, False), (0.05, 0, True)])
def test_states(shape, density, transform, blocks):
    g = vga.Graph(_image(shape, 1.0))
    X, theta, out = _state(g.n, density, 5), _theta(shape, blocks), []
    for timing in (False, True):
        sim = vga.Sim(g, synth.paper_params(transform=transform))
        if theta is not None and theta.size:
            sim.set_block_conductances(4, theta)
        sim.enable_timing(timing)
        sim.set_masses(X)
        for k in (2, 5, 1, 6):
            sim.step(k)
        out.append(sim.get_masses())
        assert sim.stats()["steps_done"] == 14
        sim.close()
    assert np.array_equal(out[0], out[1])
    g.close()


@pytest.mark.parametrize("shape,porosity", [((1, 19, 27), 1.0), ((40, 44, 52), 0.4), ((31, 37, 69), 1.0), ((64, 80, 96), 0.35),
                                            ((64, 64, 76), 1.0)])
@pytest.mark.parametrize("blocks", [False, True])
@pytest.mark.parametrize("state_gradient", [False, True])
def test_adjoint(shape, porosity, blocks, state_gradient):
    g = vga.Graph(_image(shape, porosity))
    X, theta, out = _state(g.n, 0.15, 6), _theta(shape, blocks), []
    gen = torch.Generator(device="cuda").manual_seed(9)
    lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
    for timing in (False, True):
        sim = vga.Sim(g, synth.paper_params())
        if theta is not None and theta.size:
            sim.set_block_conductances(4, theta)
        sim.enable_timing(timing)
        sim.set_masses(X)
        sim.adjoint_forward(11, 4)
        XN = sim.get_masses()
        dx = torch.zeros_like(lam) if state_gradient else None
        grad, gth = sim.adjoint_backward(lam, dx, n_theta=0 if theta is None else theta.size)
        out.append((XN, dx.cpu().numpy() if state_gradient else None, grad, gth))
        sim.close()
    (a, da, ga, ta), (b, db, gb, tb) = out
    assert np.array_equal(a, b)
    if state_gradient:
        assert np.array_equal(da, db)
        assert ga == gb
    for k in gb:
        assert abs(ga[k] - gb[k]) <= 1e-10 * abs(gb[k]), (k, ga[k], gb[k])
    if ta is not None:
        assert np.linalg.norm(ta - tb) <= 1e-10 * np.linalg.norm(tb)
    g.close()


def test_negative_dom_takes_the_other_passes():
    """A negative DOM at a node without biomass: the first transformation moves it, so such a state does not
    run as a small-graph launch."""
    g = vga.Graph(_image((12, 14, 16), 1.0))
    X, out = _state(g.n, 0.05, 7), []
    X[:, 100] = 0.0
    X[1, 100] = -1e-6
    for timing in (False, True):
        sim = vga.Sim(g, synth.paper_params())
        sim.enable_timing(timing)
        sim.set_masses(X)
        sim.step(4)
        sim.step(3)
        out.append(sim.get_masses())
        sim.close()
    assert np.array_equal(out[0], out[1])
    g.close()
