"""Bounded waits of the cooperative launches that exchange tagged words (small-graph step calls and adjoint
sweeps, Scheme 4 solves).  One block leaves before it publishes anything, the waits of the others run out
after a short limit, and the next call that synchronises returns VGA_ERR_TIMEOUT: no fault, no hang.  With the
hook off and a new upload, the same handle gives the bits of a fresh one."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

SPIN = 4096
SHAPE = (16, 16, 20)  # 10 blocks of 512 nodes


def _masses(n, seed=3):
    return synth.random_masses(n, seed, density=0.03)  # at most 512 marked nodes in a block


def _timeout(call):
    with pytest.raises(vga.VgaError) as e:
        call()
    assert e.value.name == "VGA_ERR_TIMEOUT"


@pytest.mark.parametrize("skip", [0, 4, 9])
def test_step_wait_runs_out_and_the_simulation_recovers(skip):
    g = vga.Graph(np.zeros(SHAPE, dtype=np.uint8))
    X = _masses(g.n)
    sim, fresh = (vga.Sim(g, synth.paper_params()) for _ in range(2))
    sim.set_masses(X)
    sim.step(7)
    sim.set_wait_test(skip, SPIN)
    sim.step(20)
    _timeout(sim.sync)
    sim.sync()  # reported once
    sim.set_wait_test(-1, 0)
    for s in (sim, fresh):
        s.set_masses(X)
        s.step(20)
        s.step(5)
    assert np.array_equal(sim.get_masses(), fresh.get_masses())
    for s in (sim, fresh):
        s.close()
    g.close()


@pytest.mark.parametrize("state_gradient", [False, True])
@pytest.mark.parametrize("when", ["forward", "backward"])
def test_adjoint_wait_runs_out_and_the_simulation_recovers(when, state_gradient):
    g = vga.Graph(np.zeros(SHAPE, dtype=np.uint8))
    X = _masses(g.n)
    lam = torch.randn((5, g.n), generator=torch.Generator(device="cuda").manual_seed(4), device="cuda",
                      dtype=torch.float64)
    sim, fresh = (vga.Sim(g, synth.paper_params()) for _ in range(2))

    def sweep(s, dx):
        return s.adjoint_backward(lam, dx)

    sim.set_masses(X)
    sim.set_wait_test(3 if when == "forward" else -1, SPIN)
    sim.adjoint_forward(11, 4)
    sim.set_wait_test(3, SPIN)
    _timeout(lambda: sweep(sim, torch.zeros_like(lam) if state_gradient else None))
    sim.set_wait_test(-1, 0)
    out = []
    for s in (sim, fresh):
        s.set_masses(X)
        s.adjoint_forward(11, 4)
        dx = torch.zeros_like(lam) if state_gradient else None
        grad, _ = sweep(s, dx)
        out.append((grad, s.get_masses(), None if dx is None else dx.cpu().numpy()))
        s.close()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
    assert not state_gradient or np.array_equal(out[0][2], out[1][2])
    g.close()


@pytest.mark.parametrize("skip", [0, 3])
def test_scheme4_wait_runs_out_and_the_handle_recovers(skip):
    shape = (24, 24, 24)
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    labels, q = synth.block_primitives(shape, g.export(labels=False, nbr=False)["voxel_of_node"], 3)
    assert q > 3 * 64  # several blocks
    m0 = torch.rand(q, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda", dtype=torch.float64)
    pg, fresh = (vga.Pngm(g, labels, q) for _ in range(2))
    p = synth.diffusion_params()
    args = (2, vga.VGA_SCHEME_IMPLICIT_PCG, p["D"], p["dt"])
    pg.set_wait_test(skip, SPIN)
    _timeout(lambda: pg.step(m0.clone(), *args))
    pg.set_wait_test(-1, 0)
    out = []
    for h in (pg, fresh):
        m = m0.clone()
        h.step(m, *args)
        out.append(m.cpu().numpy())
        h.close()
    assert np.array_equal(out[0], out[1])
    g.close()


READERS = {
    "get_masses": lambda s: s.get_masses(),
    "get_state_f32": lambda s: s.get_state_f32(),
    "save_state": lambda s: s.save_state(),
    "totals": lambda s: s.totals(),
    "loss_block_mass": lambda s: s.loss_block_mass(8, 2, np.zeros(12)),
    "implicit step": lambda s: (s.set_params(synth.paper_params(scheme=vga.VGA_SCHEME_IMPLICIT_PCG)), s.step(1)),
}


@pytest.mark.parametrize("reader", READERS)
def test_host_read_outs_report_an_unfinished_step_call(reader):
    """None of the calls that hand a result to the host may return a state that a launch left half-way."""
    g = vga.Graph(np.zeros(SHAPE, dtype=np.uint8))
    sim = vga.Sim(g, synth.paper_params())
    sim.set_masses(_masses(g.n))
    sim.set_wait_test(4, SPIN)
    sim.step(20)
    _timeout(lambda: READERS[reader](sim))
    sim.sync()
    sim.close()
    g.close()


@pytest.mark.parametrize("shape", [SHAPE, (64, 64, 76)])
def test_a_sweep_by_launches_reports_an_unfinished_forward_sweep(shape):
    """(64, 64, 76), four nodes per thread with dL/dX^0: the reverse sweep takes launches; with timing on
    it does at every size."""
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    lam = torch.ones((5, g.n), device="cuda", dtype=torch.float64)
    sim = vga.Sim(g, synth.paper_params())
    sim.set_masses(_masses(g.n))
    sim.set_wait_test(4, SPIN)
    sim.adjoint_forward(11, 4)
    sim.set_wait_test(-1, 0)
    sim.enable_timing(shape == SHAPE)
    _timeout(lambda: sim.adjoint_backward(lam, torch.zeros_like(lam)))
    with pytest.raises(vga.VgaError):  # no sweep to reverse is left
        sim.adjoint_backward(lam)
    sim.close()
    g.close()
