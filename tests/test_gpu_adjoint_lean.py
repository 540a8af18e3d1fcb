"""Backward sweeps that are not asked for dL/dX^0 run other reverse kernels on large graphs (the DOM
adjoint of every node, the other adjoints of the marked nodes only).  Their gradients must be those of
a sweep with dL/dX^0; the premise (no negative DOM at an unmarked node) failing, the sweep repeats in
the full form.  The two forms add the same FP32 terms in another order, in compensated pairs (about 45
bits per sum) and FP64, so they agree to 1e-10 unless a sum cancels by more than a factor 1000."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

SHAPE = (79, 84, 85)  # 564,060 nodes, no multiple of the block sizes


def _setup(density, negative, blocks):
    g = vga.Graph(np.zeros(SHAPE, dtype=np.uint8))
    gen = torch.Generator(device="cuda").manual_seed(3)
    X = torch.rand((5, g.n), generator=gen, device="cuda", dtype=torch.float64) * 1e-4
    marked = torch.rand(g.n, generator=gen, device="cuda") < density
    for c in (0, 2, 3, 4):
        X[c] = torch.where(marked, X[c], 0.0)
    if negative:
        X[1, ::1001] = -1e-5
        X[:, 0] = 0.0
        X[1, 0] = -1e-5  # an unmarked node
    lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
    sim = vga.Sim(g, synth.paper_params())
    n_theta = 0
    if blocks:
        theta = synth.block_conductances(tuple(-(-s // 8) for s in SHAPE), seed=4, spread=0.1).astype(np.float32)
        sim.set_block_conductances(8, theta)
        n_theta = theta.size
    sim.set_masses(X)
    return g, sim, lam, n_theta


@pytest.mark.parametrize("density,negative,blocks", [(0.05, False, True), (0.05, False, False), (0.0, False, True),
                                                     (0.2, False, True), (0.05, True, True)])
def test_gradients_without_state_gradient(density, negative, blocks):
    g, sim, lam, n_theta = _setup(density, negative, blocks)
    sim.adjoint_forward(7, 3)
    got, gth = sim.adjoint_backward(lam, n_theta=n_theta)
    ref, rth = sim.adjoint_backward(lam, torch.empty_like(lam), n_theta=n_theta)
    for k in ref:
        assert abs(got[k] - ref[k]) <= 1e-10 * abs(ref[k]), (k, got[k], ref[k])
    if blocks:
        assert np.linalg.norm(gth - rth) <= 1e-10 * np.linalg.norm(rth)
    again, _ = sim.adjoint_backward(lam, n_theta=n_theta)
    assert again == got  # the same bits on every run
    sim.close()
    g.close()
