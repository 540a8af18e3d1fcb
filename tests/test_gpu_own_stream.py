"""Small simulations on streams of their own overlap: where one launch per call would take more than half of the SMs,
their step calls are launches per pass, with the same bits."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,small", [((8, 10, 12), True), ((31, 35, 35), True), ((40, 40, 40), False),
                                         ((60, 60, 64), False)])
def test_step_calls_on_an_own_stream(shape, small):
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    X, out = synth.random_masses(g.n, 3, density=0.03), []
    for stream in (None, torch.cuda.Stream()):
        sim = vga.Sim(g, synth.paper_params(), stream=stream)
        sim.set_masses(X)
        sim.step(20)
        before = sim.stats()["kernel_launches"]
        sim.step(20)
        launches = sim.stats()["kernel_launches"] - before
        assert launches == 1 if stream is None or small else launches >= 20
        out.append(sim.get_masses())
        sim.close()
    assert np.array_equal(out[0], out[1])
    g.close()


def test_several_streams_at_once():
    g = vga.Graph(np.zeros((40, 40, 40), dtype=np.uint8))
    sims = [vga.Sim(g, synth.paper_params(), stream=torch.cuda.Stream()) for _ in range(4)]
    ref = vga.Sim(g, synth.paper_params())
    X = [synth.random_masses(g.n, k, density=0.03) for k in range(4)]
    for k, s in enumerate(sims):
        s.set_masses(X[k])
    for _ in range(5):
        for s in sims:
            s.step(11)
    for k, s in enumerate(sims):
        ref.set_masses(X[k])
        ref.step(55)
        assert np.array_equal(s.get_masses(), ref.get_masses())
    for s in sims + [ref]:
        s.close()
    g.close()


def test_coarse_solves_leave_room_on_an_own_stream():
    """4096 rows: 64 blocks on the default stream, 16 on another (block 20 is there or not).  Solves stop at a residual of
    1e-12; with equal volumes the masses are then within 1e-12 of the solution per step, whatever the order of the sums."""
    shape = (48, 48, 48)
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    labels, q = synth.block_primitives(shape, g.export(labels=False, nbr=False)["voxel_of_node"], 3)
    m0 = torch.rand(q, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    p = synth.diffusion_params()
    args = (3, vga.VGA_SCHEME_IMPLICIT_PCG, p["D"], p["dt"])
    out = []
    for stream in (None, torch.cuda.Stream()):
        pg = vga.Pngm(g, labels, q, stream=stream)
        m = m0.clone()
        torch.cuda.synchronize()
        pg.step(m, *args)
        out.append(m.cpu().numpy())
        pg.set_wait_test(20, 4096)
        if stream is None:
            with pytest.raises(vga.VgaError) as e:
                pg.step(m, *args)
            assert e.value.name == "VGA_ERR_TIMEOUT"
        else:
            pg.step(m, *args)
        pg.close()
    assert np.linalg.norm(out[0] - out[1]) <= 2 * 3 * 1e-12 * np.linalg.norm(out[0])
    g.close()
