"""A cooperative launch holds its SMs until it ends, so long calls are several launches: the states, the solver's
counts and the gradients are those of shorter calls, and a sweep of longer segments takes launches per step."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu

STEPS = 1 << 14  # of one launch


@pytest.mark.parametrize("n_steps", [STEPS - 1, STEPS, STEPS + 1, 2 * STEPS + 7])
def test_step_calls(n_steps):
    g = vga.Graph(np.zeros((9, 8, 10), dtype=np.uint8))
    X, out = synth.random_masses(g.n, 3, density=0.05), []
    for timing in (False, True):
        sim = vga.Sim(g, synth.paper_params())
        sim.enable_timing(timing)
        sim.set_masses(X)
        sim.step(2)
        before = sim.stats()["kernel_launches"]
        sim.step(n_steps)
        if not timing:
            assert sim.stats()["kernel_launches"] - before == -(-n_steps // STEPS)
        assert sim.stats()["steps_done"] == n_steps + 2
        out.append(sim.get_masses())
        sim.close()
    assert np.array_equal(out[0], out[1])
    g.close()


@pytest.mark.parametrize("n_steps", [STEPS, STEPS + 1])
def test_sweeps(n_steps):
    g = vga.Graph(np.zeros((6, 7, 9), dtype=np.uint8))
    X, out = synth.random_masses(g.n, 3, density=0.05), []
    lam = torch.ones((5, g.n), device="cuda", dtype=torch.float64)
    for ckpt in (1000, n_steps):
        sim = vga.Sim(g, synth.paper_params())
        sim.set_masses(X)
        before = sim.stats()["kernel_launches"]
        sim.adjoint_forward(n_steps, ckpt)
        if ckpt > STEPS:
            assert sim.stats()["kernel_launches"] - before > STEPS
        dx = torch.zeros_like(lam)
        sim.adjoint_backward(lam, dx)
        out.append((sim.get_masses(), dx.cpu().numpy()))
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    g.close()


@pytest.mark.parametrize("n_steps", [1, 64, 65, 150])
def test_scheme4(n_steps):
    shape = (24, 24, 24)
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    labels, q = synth.block_primitives(shape, g.export(labels=False, nbr=False)["voxel_of_node"], 3)
    m0 = torch.rand(q, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda", dtype=torch.float64)
    pg = vga.Pngm(g, labels, q)
    p = synth.diffusion_params()
    args = (vga.VGA_SCHEME_IMPLICIT_PCG, p["D"], p["dt"])
    m, ref, iters = m0.clone(), m0.clone(), 0
    pg.step(m, n_steps, *args)
    done = pg.info()["last_cg_iterations"]
    relres = pg.info()["last_cg_relres"]
    for _ in range(n_steps):
        pg.step(ref, 1, *args)
        iters += pg.info()["last_cg_iterations"]
    assert np.array_equal(m.cpu().numpy(), ref.cpu().numpy())
    assert done == iters and relres == pg.info()["last_cg_relres"]
    with pytest.raises(vga.VgaError) as e:  # every solve of the call stops at one iteration
        pg.step(m0.clone(), n_steps, *args, 1e-14, 1)
    assert e.value.name == "VGA_ERR_NOT_CONVERGED"
    pg.close()
    g.close()
