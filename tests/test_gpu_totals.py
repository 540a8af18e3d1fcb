"""The totals pass at the edges of its two forms (one node at a time; four at a time where every thread of the grid
has four), and the graph build where the component sizes just fit, and do not fit, into the build's scratch.

A thread adds at most ceil(n / 262,144) values in float-float, here 5 at most, each to about 2^-47 of the sum so far,
and the threads' sums are added in FP64 over 18 levels and blocks: 5 * 2^-47 + 1100 * 2^-53 < 2e-13 of a sum of
positive values."""
import numpy as np
import pytest
import torch

import paper_2406_04177_gb300 as vga
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 7, 9), (31, 92, 92), (1, 1023, 1025), (1, 1024, 1024),
                                   (101, 101, 103), (107, 103, 101)])
def test_totals_at_the_edges(shape, precision):
    g = vga.Graph(np.zeros(shape, dtype=np.uint8))
    gen = torch.Generator(device="cuda").manual_seed(5)
    X = torch.rand((5, g.n), generator=gen, device="cuda", dtype=torch.float64) * 1e-4
    X[3, : g.n // 2] = 0.0
    p = synth.paper_params()
    p["state_precision"] = precision
    sim = vga.Sim(g, p)
    sim.set_masses(X)
    ref = sim.get_masses().sum(axis=1, dtype=np.longdouble)
    first = sim.totals()
    assert np.all(np.abs(first - ref) <= 2e-13 * ref)
    for _ in range(2):  # the last block leaves the ticket and the flags as it found them
        assert np.array_equal(sim.totals(), first)
    assert sim.stats()["negative_reports"] == 0
    sim.close()
    g.close()


@pytest.mark.parametrize("step", [(2, 2, 2), (1, 2, 2), (1, 1, 2), (2, 2, 3)])
@pytest.mark.parametrize("on_device", [False, True])
def test_component_sizes_in_and_out_of_the_scratch(oracle_lib, step, on_device):
    img = np.ones((8, 10, 12), dtype=np.uint8)
    z, y, x = np.meshgrid(*[np.arange(k) for k in img.shape], indexing="ij")
    pore = (z % step[0] == 0) & (y % step[1] == 0) & (x % step[2] == 0)
    img[pore] = 0  # single voxels, or lines in z and sheets where a step is 1
    og = oracle_lib.graph_build(img, keep_largest=False)
    g = vga.Graph(torch.from_numpy(img).cuda() if on_device else img, keep_largest=False)
    assert (g.n, g.n_components, g.largest) == (og.n, og.n_components, og.largest)
    ex = g.export()
    assert np.array_equal(ex["labels"], og.labels)
    assert np.array_equal(ex["voxel_of_node"], og.voxel_of_node)
    g.close()
