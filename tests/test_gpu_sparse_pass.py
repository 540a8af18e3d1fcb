"""The sparse fused pass at the sizes where it can go wrong: block edges (1024 nodes), more marked nodes
in a block than are prefetched (64) and than threads (256), a ragged tail, and graphs above the
size from which it prefetches and alternates its order.  Every state must be the bits of the pass that
transforms every node, which runs other kernels."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu


def _state(n, density, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand((5, n), generator=g, device="cuda") * 2e-4
    marked = torch.rand(n, generator=g, device="cuda") < density
    for c in (0, 2, 3, 4):
        X[c] = torch.where(marked, X[c], 0.0)
    X[1] = torch.where(torch.rand(n, generator=g, device="cuda") < 0.2, X[1], 0.0)
    return X


def _both(g, p, X, steps, theta=None):
    out = []
    for skip in (True, False):
        sim = vga.Sim(g, p)
        if theta is not None:
            sim.set_block_conductances(4, theta)
        sim.set_activity_skip(skip)
        sim.set_state_f32(X)
        for k in steps:
            sim.step(k)
        out.append(sim.get_masses())
        sim.close()
    return out


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 31), (1, 1, 1023), (4, 16, 16), (1, 41, 25), (3, 27, 51)])
@pytest.mark.parametrize("density", [0.0, 0.03, 0.6, 1.0])
@pytest.mark.parametrize("transform,precision", [(0, 0), (1, 0), (0, 1)])
def test_block_edges(shape, density, transform, precision):
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    p = dict(synth.paper_params(transform=transform), state_precision=precision)
    a, b = _both(g, p, _state(g.n, density, 5), (2, 7))
    assert np.array_equal(a, b)
    g.close()


@pytest.mark.parametrize("density", [0.02, 0.9])
def test_block_conductances(density):
    shape = (13, 18, 29)
    g = vga.Graph(synth.pore_mask(shape, 0.6, seed=8))
    nb = tuple(-(-s // 4) for s in shape)
    theta = synth.block_conductances(nb, seed=3, spread=0.09).astype(np.float32)
    a, b = _both(g, synth.paper_params(), _state(g.n, density, 6), (9,), theta)
    assert np.array_equal(a, b)
    g.close()


@pytest.mark.parametrize("density,transform", [(0.01, 0), (0.3, 1)])
def test_large_graph(density, transform):
    """5.4 million nodes: above the size from which the pass prefetches and alternates its order."""
    g = vga.Graph(np.zeros((173, 176, 179), dtype=np.uint8))
    assert g.n > 5 << 20
    a, b = _both(g, synth.paper_params(transform=transform), _state(g.n, density, 7), (6, 3))
    assert np.array_equal(a, b)
    g.close()
