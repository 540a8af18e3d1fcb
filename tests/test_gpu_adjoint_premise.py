"""The reverse forms that take the marked nodes only (sweeps without dL/dX^0 on large graphs, one launch per segment
on small ones) stand on the transformation of an unmarked node being the identity.  Every segment starts with the
transformation of every node: where a DOM is negative there, the node's biomass changes and later segments' rate
gradients with it, and the sweep must give what the full form by launches gives (same FP32 terms, sums in another
order: 1e-10 unless a sum cancels by more than a factor 1000)."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu


def _state(n, gen):
    X = torch.rand((5, n), generator=gen, device="cuda", dtype=torch.float64) * 1e-4
    marked = torch.rand(n, generator=gen, device="cuda") < 0.05
    marked[:50] = False
    for c in (0, 2, 3, 4):
        X[c] = torch.where(marked, X[c], 0.0)
    return X, marked


def _close(got, ref):
    for k in ref:
        assert abs(got[k] - ref[k]) <= 1e-10 * abs(ref[k]), (k, got[k], ref[k])


def test_large_graph_one_negative_dom_at_the_start():
    g = vga.Graph(np.zeros((79, 84, 85), dtype=np.uint8))
    gen = torch.Generator(device="cuda").manual_seed(3)
    X, _ = _state(g.n, gen)
    X[1, 0] = -1e-3  # unmarked: becomes biomass in the first transformation, no DOM is negative after it
    lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
    # with beta = 0 the negative biomass reaches the SOM in the second segment, and no DOM is negative in it
    sim = vga.Sim(g, dict(synth.paper_params(), beta=0.0))
    sim.set_masses(X)
    sim.adjoint_forward(6, 3)
    got, _ = sim.adjoint_backward(lam)
    ref, _ = sim.adjoint_backward(lam, torch.empty_like(lam))
    _close(got, ref)
    sim.close()
    g.close()


@pytest.mark.parametrize("shape", [(9, 11, 13), (40, 44, 52), (64, 64, 76)])
@pytest.mark.parametrize("state_gradient", [False, True])
def test_small_graph_with_negative_stocks(shape, state_gradient):
    g, out = vga.Graph(np.zeros(shape, dtype=np.uint8)), []
    for timing in (False, True):  # launches per step while timing is on
        gen = torch.Generator(device="cuda").manual_seed(3)
        X, marked = _state(g.n, gen)
        X[1] = 0.0
        X[3] = torch.where(marked, -1e-3, 0.0)
        lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
        sim = vga.Sim(g, synth.paper_params())
        sim.enable_timing(timing)
        sim.set_masses(X)
        sim.adjoint_forward(11, 4)
        dx = torch.zeros_like(lam) if state_gradient else None
        grad, _ = sim.adjoint_backward(lam, dx)
        out.append((grad, sim.get_masses(), dx))
        sim.close()
    assert np.array_equal(out[0][1], out[1][1])
    _close(out[0][0], out[1][0])
    if state_gradient:
        assert torch.equal(out[0][2], out[1][2])
    g.close()


@pytest.mark.parametrize("where", ["host", "in place"])
def test_a_repeated_sweep_reads_its_input_again(where):
    """The host form stages both gradients in one buffer, and a caller may pass one for both: the sweep that is
    repeated must not have overwritten dL/dX^N."""
    g = vga.Graph(np.zeros((9, 11, 13), dtype=np.uint8))
    gen = torch.Generator(device="cuda").manual_seed(3)
    X, marked = _state(g.n, gen)
    X[1] = 0.0
    X[3] = torch.where(marked, -1e-3, 0.0)  # repeats, as above
    lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
    sim = vga.Sim(g, synth.paper_params())
    sim.set_masses(X)
    sim.adjoint_forward(11, 4)
    dx = torch.zeros_like(lam)
    ref, _ = sim.adjoint_backward(lam, dx)
    if where == "host":
        out = np.zeros((5, g.n))
        got, _ = sim.adjoint_backward(lam.cpu().numpy(), out)
    else:
        buf = lam.clone()
        got, _ = sim.adjoint_backward(buf, buf)
        out = buf.cpu().numpy()
    assert got == ref and np.array_equal(out, dx.cpu().numpy())
    sim.close()
    g.close()


@pytest.mark.parametrize("shape", [(9, 11, 13), (40, 44, 52), (79, 84, 85)])
@pytest.mark.parametrize("state_gradient", [False, True])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_an_adjoint_that_is_not_finite_spreads(shape, state_gradient, value):
    """dL/dMB^N at an unmarked node: J_T multiplies it by zero on its way to the DOM, which makes a NaN of it,
    not nothing."""
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    gen = torch.Generator(device="cuda").manual_seed(3)
    X, _ = _state(g.n, gen)
    lam = torch.randn((5, g.n), generator=gen, device="cuda", dtype=torch.float64)
    lam[0, 7] = value
    sim = vga.Sim(g, synth.paper_params())
    sim.set_masses(X)
    sim.adjoint_forward(7, 3)
    dx = torch.zeros_like(lam) if state_gradient else None
    grad, _ = sim.adjoint_backward(lam, dx)
    assert np.isnan(grad["D"])
    if state_gradient:
        assert torch.isnan(dx[1]).any()
    sim.close()
    g.close()
