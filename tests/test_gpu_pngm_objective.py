"""The objective's kernels at the edges of their launches: one pair, the pairs of one launch, one more,
several launches; fewer and more rows than a block has threads.  Against the FP64 oracle.

A residual r_i is a sum of about deg + 3 terms, of which the independent random records leave a tenth or more,
so r_i and each term of the gradient hold to about 10 (deg + 3) eps = 5e-14 at the 20 neighbours that a random
partition gives a row, and the sums of their squares and products to a few times that: 1e-12."""
import numpy as np
import pytest

import synth
from oracle import pngm as opn
from tests.helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [1, 2])
@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("bs,l", [(40, 64), (8, 1), (8, 3), (4, 64), (4, 65), (4, 150)])
def test_objective_over_launches(vga, oracle_lib, kind, tied, bs, l):
    import torch

    img = synth.pore_mask((40, 36, 44), 0.25, 3)
    og = oracle_lib.graph_build(img, keep_largest=True)
    g = vga.Graph(img)
    lab, q = synth.block_primitives(img.shape, og.voxel_of_node, bs)
    cg = opn.coarse_graph(og.nbr, og.voxel_of_node, img.shape, lab, q)
    pg = vga.Pngm(g, lab, q)
    rng = np.random.default_rng(100 * bs + l)
    th = opn.initial_theta(cg) * rng.uniform(0.6, 1.4, len(cg["row"]))
    if tied:
        th = (th + th[cg["rev"]]) / 2
    pg.set_theta(th)
    c = 0.2 / max(np.bincount(cg["row"], weights=th, minlength=q) / cg["vol"])
    R = rng.random((9, q)) * cg["vol"]
    pairs = rng.integers(0, len(R), (l, 2)).astype(np.int32)
    pairs[:, 1] = (pairs[:, 0] + 1 + pairs[:, 1] % (len(R) - 1)) % len(R)  # two different records
    data = torch.from_numpy(R).cuda()
    grad = torch.empty(pg.n_slots, dtype=torch.float64, device="cuda")
    X, Y = R[pairs[:, 0]], R[pairs[:, 1]]
    ref_loss, ref_grad = opn.objective(kind, cg, th, X, Y, c, tied=tied)
    for _ in range(2):  # the work area of an earlier call leaves nothing behind
        loss = pg.objective(kind, data, pairs, c, 1.0, tied=tied, grad=grad)
        assert np.isclose(loss, ref_loss, rtol=1e-12)
        assert rel_l2(grad.cpu().numpy(), ref_grad) <= 1e-12
    m = torch.from_numpy(R[0].copy()).cuda()
    pg.step(m, 2, 0, c, 1.0)  # Scheme 3 uses the same work area
    assert rel_l2(m.cpu().numpy(), opn.scheme3(cg, th, R[0], c, 2)) <= 1e-14
    before = pg.sgd_step(kind, data, pairs, c, 1.0, 0.01, tied=tied, theta_min=0.0)
    assert before == loss
    new_ref, _ = opn.sgd_step(kind, cg, th, X, Y, c, 0.01, tied=tied, theta_min=0.0)
    got = pg.get_theta()
    big = np.abs(ref_grad) > 1e-9 * np.abs(ref_grad).max()
    assert np.array_equal(got[big], new_ref[big])
    if tied:
        assert np.array_equal(got, got[cg["rev"]])
