"""Kernel variant 6 asks for temporally blocked passes: it gets them whatever share of the nodes is marked, as long as
a tile's marked nodes fit."""
import numpy as np
import pytest

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("density", [0.1, 0.3, 0.8])
def test_blocked_passes_with_many_marked_nodes(density):
    img = np.ones((16, 16, 64), dtype=np.uint8)
    img[::8, ::8, :] = 0  # 4 lines of 64 nodes
    g = vga.Graph(img, keep_largest=False)
    X, out = synth.random_masses(g.n, 4, density=density), []
    for variant in (6, 2):
        sim = vga.Sim(g, synth.paper_params())
        sim.set_kernel(variant, 1024)
        sim.set_masses(X)
        sim.step(9)
        if variant == 6:
            assert sim.stats()["blocked_passes"] == 8
        out.append(sim.get_masses())
        sim.close()
    assert np.array_equal(out[0], out[1])
    g.close()
