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
    X = synth.random_masses(n, seed, density=0.1)
    return np.ascontiguousarray(X)


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
