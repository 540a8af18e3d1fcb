"""Sweeps without dL/dX^0 on graphs where a thread of the full reverse form takes more than eight groups of nodes:
the per-thread sums of dL/dD go to FP64 every few steps, within segments, between them and at the end.  The
gradients are those of the full form (same FP32 terms, sums in another order: 1e-10 unless a sum cancels by more
than a factor 1000)."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

SHAPE = (149, 150, 151)  # 3.4 M nodes: 11 groups a thread with four blocks per SM


@pytest.mark.parametrize("steps,ckpt", [(30, 30), (26, 4), (22, 11), (23, 12), (40, 13)])
def test_dD(steps, ckpt):
    g = vga.Graph(np.zeros(SHAPE, dtype=np.uint8))
    gen = torch.Generator(device="cuda").manual_seed(3)
    X = torch.zeros((5, g.n), device="cuda", dtype=torch.float64)
    X[1] = torch.rand(g.n, generator=gen, device="cuda", dtype=torch.float64) * 1e-4
    X[0] = torch.where(torch.rand(g.n, generator=gen, device="cuda") < 0.02, 1e-5, 0.0)
    lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
    sim = vga.Sim(g, synth.paper_params())
    sim.set_masses(X)
    sim.adjoint_forward(steps, ckpt)
    got, _ = sim.adjoint_backward(lam)
    again, _ = sim.adjoint_backward(lam)
    ref, _ = sim.adjoint_backward(lam, torch.empty_like(lam))
    assert again == got  # the same bits on every run
    for k in ref:
        assert abs(got[k] - ref[k]) <= 1e-10 * abs(ref[k]), (k, got[k], ref[k])
    sim.close()
    g.close()
