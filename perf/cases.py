"""Workloads the speed of this framework is judged by, each through its public entry points.

Kinds of case (key "kind"):
  monitor   a small image stepped a few steps at a time, the totals and the state read after each call
  forward   upload a state, advance it with the explicit scheme, read state and totals
  implicit  the same with Scheme 2 at ten times the explicit time step
  gradient  one epoch of conductance fitting: checkpointed forward, block-mass loss, reverse sweep
  autograd  the same model as a torch.autograd.Function: state out, gradients of every input back
  batch     many uneven subvolumes with their own rates advanced together
  image     a new image from the scanner: graph, simulation, a short run, the result
  train     normalised SGD of the coarse primitive model's conductances
  coarse    implicit steps of the coarse primitive model

Images are Gaussian-smoothed white noise (sigma 2 voxels) at a given porosity, one for each size;
masses are those of the paper's Sec. IV.C, conductances and records of the coarse model random, all
from the seed.  Everything is drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2406_04177_gb300 as vga
from paper_2406_04177_gb300 import autograd, fit

D_DOM = 100950.0  # DOM diffusion coefficient, voxel^2 per day
RATES = dict(rho=0.2, mu=0.5, beta=0.55, v_som=0.01, v_fom=0.3, v_dom=9.6, K_dom=1.3824e-5)
EXPLICIT_DT = 0.9 / (6.0 * D_DOM)
DOM_MEAN = 289.5 / (0.05 * 22817014)   # mean mass of a node that holds DOM (5% of the nodes)
MB_MEAN = 2.8132 / (0.01 * 22817014)   # mean mass of a node that holds biomass (1%)
COARSE_DT = 10.0 / 86400.0             # 10 s between two records of the coarse model
BLOCK = 8                              # side of the conductance blocks
COMP_DOM_CO2 = (1 << 1) | (1 << 4)


def listed():
    return [
        # the 64^3 subvolume stepped interactively: a few microseconds of work per step
        dict(name="monitor_64", kind="monitor", nz=64, ny=64, nx=64, porosity=0.17, steps=20),
        # the 256^3 image at 20%
        dict(name="forward_256", kind="forward", nz=256, ny=256, nx=256, porosity=0.20, steps=100,
             organic=0.0, transform="sync"),
        # the paper-scale image, 21 million nodes
        dict(name="forward_512", kind="forward", nz=512, ny=512, nx=512, porosity=0.17, steps=100,
             organic=0.0, transform="sync"),
        # a ragged image with organic matter, biomass and CO2 spread over the pore space (late stages
        # of a decomposition): most nodes transform
        dict(name="organic_211x260x301", kind="forward", nz=211, ny=260, nx=301, porosity=0.25, steps=50,
             organic=0.3, transform="sync"),
        # Scheme 2 at ten times the explicit step, small and paper-scale
        dict(name="implicit_128", kind="implicit", nz=128, ny=128, nx=128, porosity=0.17, steps=3),
        dict(name="implicit_512", kind="implicit", nz=512, ny=512, nx=512, porosity=0.17, steps=1),
        # one epoch of the 128^3 conductance fit
        dict(name="gradient_128", kind="gradient", nz=128, ny=128, nx=128, porosity=0.17, steps=2000, ckpt=100),
        # a larger model inside a torch program
        dict(name="autograd_320", kind="autograd", nz=320, ny=320, nx=320, porosity=0.17, steps=60, ckpt=20),
        # a parameter study over uneven subvolumes
        dict(name="batch_12", kind="batch", count=12, side_lo=64, side_hi=192, steps=2000),
        # one of a series of scans
        dict(name="image_190x224x257", kind="image", nz=190, ny=224, nx=257, porosity=0.22, steps=50),
        # calibration of the coarse model and its implicit steps (16^3 cubes of a 512^3 image)
        dict(name="train_512", kind="train", nz=512, ny=512, nx=512, porosity=0.17, epochs=100),
        dict(name="coarse_512", kind="coarse", nz=512, ny=512, nx=512, porosity=0.17, steps=3),
    ]


def draw(rng):
    kind = rng.choice(["monitor", "forward", "forward", "forward", "implicit", "gradient", "autograd", "batch",
                       "image", "train", "coarse"])

    def box(lo, hi):
        side = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        nz, ny, nx = (max(16, int(round(side * rng.uniform(0.8, 1.2)))) for _ in range(3))
        return dict(nz=nz, ny=ny, nx=nx, porosity=round(rng.uniform(0.15, 0.35), 3))

    if kind == "monitor":
        return dict(kind=kind, **box(32, 128), steps=rng.randint(2, 40))
    if kind == "forward":
        organic = rng.choice([0.0, 0.0, round(rng.uniform(0.02, 0.5), 3)])
        return dict(kind=kind, **box(48, 384), steps=rng.randint(20, 100), organic=organic,
                    transform=rng.choice(["sync", "sync", "async"]))
    if kind == "implicit":
        return dict(kind=kind, **box(48, 320), steps=rng.randint(1, 3))
    if kind == "gradient":
        return dict(kind=kind, **box(40, 128), steps=rng.randint(100, 800), ckpt=rng.choice([25, 50, 100]))
    if kind == "autograd":
        return dict(kind=kind, **box(64, 256), steps=rng.randint(20, 60), ckpt=rng.choice([10, 20, 50]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 12), side_lo=rng.randint(40, 64), side_hi=rng.randint(80, 160),
                    steps=rng.randint(100, 1000))
    if kind == "image":
        return dict(kind=kind, **box(64, 256), steps=rng.randint(10, 60))
    if kind == "train":
        return dict(kind=kind, **box(160, 448), epochs=rng.randint(20, 100))
    return dict(kind=kind, **box(160, 448), steps=rng.randint(1, 4))


# ---- inputs -------------------------------------------------------------------------------------
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _image(shape, porosity, salt=0):
    """uint8 CUDA image [z][y][x], 0 = pore: the lowest `porosity` of a smoothed Gaussian field.  The
    same for every seed, so that the states of one case have one number of nodes."""
    f = torch.randn(shape, generator=_gen(3, 11 + salt), device="cuda")
    w = [math.exp(-0.5 * (k / 2.0) ** 2) for k in range(-8, 9)]
    for dim in range(3):
        n = shape[dim]
        i = torch.arange(-8, n + 8, device="cuda") % (2 * n)
        i = torch.where(i < n, i, 2 * n - 1 - i)  # mirrored at the border
        g = f.index_select(dim, i)
        f = torch.zeros_like(f)
        for k in range(17):
            f.add_(g.narrow(dim, k, n), alpha=w[k] / sum(w))
        del g
    flat = f.reshape(-1)
    part = flat[:: max(1, flat.numel() // 1000000)].sort().values
    return (f > part[int(porosity * (part.numel() - 1))]).to(torch.uint8)


def _kept(graph):
    """Raster index of every node (int64 CUDA tensor) and the boolean node image."""
    vox = torch.from_numpy(graph.export(labels=False, nbr=False)["voxel_of_node"]).cuda()
    return vox, _mask_of(vox, graph.shape)


def _mask_of(vox, shape):
    m = torch.zeros(shape, dtype=torch.bool, device="cuda")
    m.view(-1)[vox] = True
    return m


def _masses(vox, kept, seed, organic=0.0, hydrolysable=False, salt=0):
    """(5, n) float32: DOM in 5% of the nodes, biomass in 1% next to solid; organic > 0: every other
    compartment in that share of the nodes; hydrolysable: FOM and SOM where there is DOM."""
    n = vox.numel()
    g = _gen(seed, 23 + salt)
    r = torch.rand((2, n), generator=g, device="cuda")
    X = torch.zeros((5, n), device="cuda")
    X[1] = torch.where(r[0] < 0.05, r[1] * (2 * DOM_MEAN), 0.0)
    k = kept.to(torch.int8)
    c = torch.zeros_like(k)
    for dim in range(3):
        m = k.shape[dim] - 1
        c.narrow(dim, 1, m).add_(k.narrow(dim, 0, m))
        c.narrow(dim, 0, m).add_(k.narrow(dim, 1, m))
    border = c.view(-1)[vox] < 6
    share = 0.01 / max(float(border.float().mean()), 0.01)
    r = torch.rand((2, n), generator=g, device="cuda")
    X[0] = torch.where(border & (r[0] < share), r[1] * (2 * MB_MEAN), 0.0)
    if hydrolysable:
        X[3] = X[1]
        X[2] = 0.1 * X[1]
    if organic > 0.0:
        for q, mean in ((0, MB_MEAN), (2, DOM_MEAN), (3, DOM_MEAN), (4, MB_MEAN)):
            r = torch.rand((2, n), generator=g, device="cuda")
            X[q] = torch.where(r[0] < organic, r[1] * (2 * mean), X[q])
    return X


def _params(case, scale=None):
    p = dict(RATES, D=D_DOM, dt=EXPLICIT_DT, scheme=0, transform=1 if case.get("transform") == "async" else 0)
    if case["kind"] == "implicit":
        p.update(dt=10 * EXPLICIT_DT, scheme=1, cg_rtol=1e-8, cg_maxit=500)
    for k, s in (scale or {}).items():
        p[k] *= s
    return p


def _n_blocks(shape):
    return tuple(-(-s // BLOCK) for s in shape)


def _n_theta(shape):
    bz, by, bx = _n_blocks(shape)
    return bz * by * (bx - 1) + bz * (by - 1) * bx + (bz - 1) * by * bx


def _theta(shape, seed):
    """Block conductances, log-uniform in [0.5, 1.1] (stable at the explicit time step)."""
    r = torch.rand(_n_theta(shape), generator=_gen(seed, 37), device="cuda")
    return torch.exp(math.log(0.5) + r * (math.log(1.1) - math.log(0.5)))


def _block_of(vox, shape, side):
    nz, ny, nx = shape
    by, bx = -(-ny // side), -(-nx // side)
    return ((vox // (nx * ny)) // side * by + (vox // nx) % ny // side) * bx + vox % nx // side


def _block_targets(vox, shape, X0, seed):
    """DOM and CO2 mass of every block in the data to be fitted: the mean densities after mixing,
    each block off by up to 20%."""
    nb = math.prod(_n_blocks(shape))
    cnt = torch.bincount(_block_of(vox, shape, BLOCK), minlength=nb).double()
    r = torch.rand((2, nb), generator=_gen(seed, 41), device="cuda", dtype=torch.float64)
    level = torch.tensor([float(X0[1].double().mean()), 1e-3 * float(X0[0].double().mean())], dtype=torch.float64,
                         device="cuda")
    return cnt[None, :] * level[:, None] * (0.8 + 0.4 * r)


def _batch_specs(case):
    rng = np.random.Generator(np.random.PCG64(7))
    out = []
    for _ in range(case["count"]):
        side = int(rng.integers(case["side_lo"], case["side_hi"] + 1))
        por = float(rng.uniform(0.10, 0.35))
        scale = {k: float(np.exp(rng.uniform(math.log(0.5), math.log(1.5))))
                 for k in ("rho", "mu", "v_som", "v_fom", "v_dom")}
        out.append(((side,) * 3, por, scale))
    return out


def _labels(vox, shape):
    """Primitive of every node: the 16^3 cube that holds it, non-empty cubes numbered in raster order."""
    used, lab = torch.unique(_block_of(vox, shape, 16), return_inverse=True)
    return lab.to(torch.int32), int(used.numel())


TRAIN_RECORDS, TRAIN_BATCH = 24, 4


def _coarse_inputs(vol, seed):
    """Records of primitive masses: concentrations drifting towards their mean, 10 s apart."""
    q = vol.numel()
    g = _gen(seed, 53)
    c = torch.rand(q, generator=g, device="cuda", dtype=torch.float64) * (2 * 0.05 * DOM_MEAN)
    out = []
    for _ in range(TRAIN_RECORDS):
        out.append(vol * c)
        r = torch.rand(q, generator=g, device="cuda", dtype=torch.float64)
        c = c + (0.02 + 0.02 * r) * (c.mean() - c)
    return torch.stack(out).contiguous()


def _train_pairs():
    return np.stack([np.arange(TRAIN_RECORDS - 1), np.arange(1, TRAIN_RECORDS)], axis=1).astype(np.int32)


# ---- one state and one pass -----------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        graphs, params, masses = [], [], []
        for k, (shape, por, scale) in enumerate(_batch_specs(case)):
            g = vga.Graph(_image(shape, por, salt=100 * (k + 1)))
            vox, kept = _kept(g)
            graphs.append(g)
            params.append(_params(case, scale))
            masses.append(_masses(vox, kept, seed, salt=100 * (k + 1)).double().cpu().numpy())
        s["graphs"] = graphs
        s["batch"] = vga.Batch(graphs, params)
        for k, X in enumerate(masses):
            s["batch"].set_masses(k, X)
        return s
    shape = _shape(case)
    img = _image(shape, case["porosity"])
    g = vga.Graph(img)
    vox, kept = _kept(g)
    if kind == "image":
        s["image"] = img.cpu().numpy()
        s["x0"] = _masses(vox, kept, seed)
        s["out"] = torch.empty_like(s["x0"])
        g.close()
        return s
    s["graph"] = g
    if kind in ("train", "coarse"):
        lab, q = _labels(vox, shape)
        s["pngm"] = vga.Pngm(g, lab, q)
        ex = s["pngm"].export()
        s["theta0"] = s["pngm"].get_theta()
        s["data"] = _coarse_inputs(torch.from_numpy(ex["vol"]).cuda(), seed)
        s["m"] = torch.empty_like(s["data"][0])
        s["seed"] = int(seed)
        return s
    s["x0"] = _masses(vox, kept, seed, organic=case.get("organic", 0.0), hydrolysable=kind in ("gradient", "autograd"))
    s["sim"] = vga.Sim(g, _params(case))
    if kind in ("monitor", "forward", "implicit"):
        s["out"] = torch.empty_like(s["x0"])
        if kind == "monitor":
            s["sim"].set_state_f32(s["x0"])
        return s
    s["theta"] = _theta(shape, seed)
    if kind == "gradient":
        s["target"] = _block_targets(vox, shape, s["x0"], seed).cpu().numpy()
        s["out"] = torch.empty_like(s["x0"])
        s["x0"] = s["x0"].double()
        s["dldx"] = torch.empty_like(s["x0"])
        return s
    r = torch.randn((5, g.n), generator=_gen(seed, 61), device="cuda", dtype=torch.float64)
    s["grad_out"] = r
    s["theta"].requires_grad_(True)
    s["x0"] = s["x0"].double().requires_grad_(True)
    s["rates"] = torch.tensor([_params(case)[k] for k in autograd.RATE_NAMES], dtype=torch.float64, requires_grad=True)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "monitor":
        s["sim"].step(case["steps"])
        return dict(totals=s["sim"].totals(), state=s["sim"].get_state_f32(s["out"]))
    if kind in ("forward", "implicit"):
        sim = s["sim"]
        sim.set_state_f32(s["x0"])
        sim.step(case["steps"])
        return dict(totals=sim.totals(), state=sim.get_state_f32(s["out"]))
    if kind == "gradient":
        sim = s["sim"]
        sim.set_block_conductances(BLOCK, s["theta"])
        sim.set_masses(s["x0"])
        sim.adjoint_forward(case["steps"], case["ckpt"])
        loss, mass = sim.loss_block_mass(BLOCK, COMP_DOM_CO2, s["target"], dL_dX=s["dldx"], want_mass=True)
        grad, gtheta = sim.adjoint_backward(s["dldx"], n_theta=s["theta"].numel())
        return dict(loss=loss, mass=mass, state=sim.get_state_f32(s["out"]),
                    grad=np.array([grad[k] for k in vga.GRAD_NAMES]), gtheta=gtheta)
    if kind == "autograd":
        XN = autograd.run(s["sim"], s["theta"], s["rates"], s["x0"], case["steps"], case["ckpt"], BLOCK)
        gtheta, grates, gx0 = torch.autograd.grad(XN, (s["theta"], s["rates"], s["x0"]), s["grad_out"])
        return dict(state=XN.detach(), gtheta=gtheta, grates=grates, gx0=gx0)
    if kind == "batch":
        b = s["batch"]
        b.step(case["steps"])
        return [b.get_masses(k) for k in range(case["count"])]
    if kind == "image":
        g = vga.Graph(s["image"])
        sim = vga.Sim(g, _params(case))
        sim.set_state_f32(s["x0"])
        sim.step(case["steps"])
        out = dict(components=g.n_components, nodes=g.n, totals=sim.totals(), state=sim.get_state_f32(s["out"]))
        sim.close()
        g.close()
        return out
    pg = s["pngm"]
    if kind == "train":
        pg.set_theta(s["theta0"])
        r = fit.fit_pngm(pg, s["data"], _train_pairs(), D_DOM, COARSE_DT, objective=2, epochs=case["epochs"],
                         batch=TRAIN_BATCH, lr0=0.05 * float(np.mean(s["theta0"])), seed=s["seed"])
        return dict(loss=r["loss"], theta=r["theta"])
    s["m"].copy_(s["data"][0])
    return dict(mass=pg.step(s["m"], case["steps"], vga.VGA_SCHEME_IMPLICIT_PCG, D_DOM, COARSE_DT))


def work(case):
    """Per node and time step: the DOM read and written (8 B), and the 32 B of the other compartments
    for the nodes that transform; each reverse step reads and writes the adjoint's five compartments
    once and reads the recorded DOM.  An implicit step reads and writes the state once."""
    kind = case["kind"]
    if kind == "batch":
        mean = (case["side_lo"] + case["side_hi"]) / 2.0
        n = case["count"] * mean ** 3 * 1.1 * 0.2
        return dict(bytes=n * (case["steps"] * 8.3 + 40), flops=n * case["steps"] * 20.0)
    n = math.prod(_shape(case)) * case["porosity"] * 0.95
    if kind in ("train", "coarse"):
        q = math.prod(-(-s // 16) for s in _shape(case))
        reps = case.get("epochs", 0) or case["steps"]
        per = TRAIN_BATCH * 2 * 8 * q + 2 * 8 * 6 * q if kind == "train" else 8 * (2 * q + 6 * q)
        return dict(bytes=float(reps * per), flops=float(reps * 6 * q * (10 * TRAIN_BATCH if kind == "train" else 10)))
    steps = case["steps"]
    marked = 0.01 if not case.get("organic") else 1.0 - (1.0 - case["organic"]) ** 4
    if kind in ("gradient", "autograd"):
        return dict(bytes=n * (steps * (8.0 + 32 * 0.06 + 44.0) + 160), flops=n * steps * 90.0)
    if kind == "implicit":
        return dict(bytes=n * (steps * 40.0 + 40), flops=n * steps * 30 * 30.0)
    per = 8.0 + 32 * marked
    more = case["nz"] * case["ny"] * case["nx"] if kind == "image" else 0
    return dict(bytes=n * (steps * per + 40) + more, flops=n * steps * (20.0 + 40 * marked))


# ---- the same in 64 bits, in plain torch ------------------------------------------------------------
def _neighbours(kept):
    """For every node (raster order) the index of its neighbour at -x, +x, -y, +y, -z, +z, or -1."""
    idx = torch.full(kept.shape, -1, dtype=torch.int64, device="cuda")
    vox = kept.view(-1).nonzero().view(-1)
    idx.view(-1)[vox] = torch.arange(vox.numel(), device="cuda")
    out = []
    for dim in (2, 1, 0):
        m = kept.shape[dim] - 1
        for lo in (True, False):
            nb = torch.full_like(idx, -1)
            if m > 0:
                a, b = (1, 0) if lo else (0, 1)
                nb.narrow(dim, a, m).copy_(idx.narrow(dim, b, m))
            out.append(nb.view(-1)[vox])
    return vox, out


def _components(n, nbs):
    """Label of every node: the smallest node index of its 6-connected component."""
    lab = torch.arange(n, device="cuda")
    me = lab.clone()
    while True:
        new = lab
        for nb in nbs:
            new = torch.minimum(new, lab[torch.where(nb >= 0, nb, me)])
        root = lab.clone().scatter_reduce_(0, lab, new, "amin")  # hook whole trees
        new = torch.minimum(new, root[new])
        new = new[new]
        new = new[new]
        if torch.equal(new, lab):
            return lab
        lab = new


def _largest(img):
    """The largest component's node image (ties: the first in raster order)."""
    kept = img == 0
    vox, nbs = _neighbours(kept)
    lab = _components(vox.numel(), nbs)
    del nbs
    sizes = torch.bincount(lab, minlength=vox.numel())
    return _mask_of(vox[lab == sizes.argmax()], tuple(img.shape))


def _transform(X, p, dt):
    """One transformation of every node; p's rates are numbers or one value per node."""
    x1, x2, x3, x4, x5 = X
    a, r, m, f, s = (p[k] * dt for k in ("v_dom", "rho", "mu", "v_fom", "v_som"))
    beta = p["beta"]
    if p.get("transform", 0) == 0:
        up = a * (x2 / (p["K_dom"] + x2)) * x1
        up = torch.where(up > x2, x2, up)
        resp, mort = r * x1, m * x1
        over, more = resp + mort > x1, mort > x1
        resp = torch.where(over, torch.where(more, torch.zeros_like(x1), x1 - mort), resp)
        mort = torch.where(over & more, x1, mort)
        tf, ts = f * x4, s * x3
        tf, ts = torch.where(tf > x4, x4, tf), torch.where(ts > x3, x3, ts)
        return (x1 + ((up - mort) - resp), x2 + (beta * mort - up + tf + ts), x3 + ((1 - beta) * mort - ts), x4 - tf,
                x5 + resp)
    zero = torch.zeros_like(x1)
    live = x1 > 0
    up = torch.where(live & (x2 > 0), torch.minimum(a * (x2 / (p["K_dom"] + x2)) * x1, x2), zero)
    x1, x2 = x1 + up, x2 - up
    mort = torch.where(live, torch.minimum(m * x1, x1), zero)
    x1, x2, x3 = x1 - mort, x2 + beta * mort, x3 + (1 - beta) * mort
    resp = torch.where(live, torch.minimum(r * x1, x1), zero)
    x1, x5 = x1 - resp, x5 + resp
    ts = torch.minimum(s * x3, x3)
    x3, x2 = x3 - ts, x2 + ts
    tf = torch.minimum(f * x4, x4)
    return x1, x2 + tf, x3, x4 - tf, x5


def _explicit(X, nbs, p, steps):
    n = X.shape[1]
    me = torch.arange(n, device="cuda")
    nbs = [torch.where(nb >= 0, nb, me) for nb in nbs]
    X = tuple(X)
    c = p["D"] * p["dt"]
    for _ in range(steps):
        x1, y, x3, x4, x5 = _transform(X, p, p["dt"])
        acc = 6.0 * y
        for nb in nbs:
            acc -= y[nb]
        X = (x1, y - c * acc, x3, x4, x5)
    return torch.stack(X)


def _cg(apply, b, diag, rtol, maxit=4000):
    x, r = b / diag, None
    r = b - apply(x)
    z = r / diag
    p, rz = z.clone(), torch.dot(r, z)
    stop = rtol * rtol * float(torch.dot(b, b))
    for k in range(maxit):
        if k % 8 == 0 and float(torch.dot(r, r)) <= stop:
            break
        q = apply(p)
        al = rz / torch.dot(p, q)
        x += al * p
        r -= al * q
        z = r / diag
        rz, old = torch.dot(r, z), rz
        p = z + (rz / old) * p
    return x


def _implicit(X, nbs, p, steps):
    n = X.shape[1]
    me = torch.arange(n, device="cuda")
    deg = sum((nb >= 0).double() for nb in nbs)
    nbs = [torch.where(nb >= 0, nb, me) for nb in nbs]
    c = p["D"] * p["dt"]

    def apply(v):
        acc = 6.0 * v
        for nb in nbs:
            acc -= v[nb]
        return v + c * acc

    X = tuple(X)
    for _ in range(steps):
        x1, y, x3, x4, x5 = _transform(X, p, p["dt"])
        X = (x1, _cg(apply, y, 1.0 + c * deg, 1e-14), x3, x4, x5)
    return torch.stack(X)


def _edges(vox, nbs, shape):
    """(i, j, index of the block face the edge crosses or -1) of every edge, once."""
    nz, ny, nx = shape
    bz, by, bx = _n_blocks(shape)
    ii, jj, ff = [], [], []
    n_x, n_y = bz * by * (bx - 1), bz * (by - 1) * bx
    for axis, nb in enumerate((nbs[1], nbs[3], nbs[5])):
        i = (nb >= 0).nonzero().view(-1)
        v = vox[i]
        x, y, z = v % nx, v // nx % ny, v // (nx * ny)
        kx, ky, kz = x // BLOCK, y // BLOCK, z // BLOCK
        face = (((kz * by + ky) * (bx - 1) + kx), n_x + (kz * (by - 1) + ky) * bx + kx,
                n_x + n_y + (kz * by + ky) * bx + kx)[axis]
        cross = ((x, y, z)[axis] + 1) % BLOCK == 0
        ii.append(i)
        jj.append(nb[i])
        ff.append(torch.where(cross, face, torch.full_like(face, -1)))
    return torch.cat(ii), torch.cat(jj), torch.cat(ff)


def _model(X0, theta, rates, edges, steps, dt):
    """The explicit run with block conductances, differentiable in (X0, theta, rates)."""
    from torch.utils.checkpoint import checkpoint

    ei, ej, ef = edges
    inside = ef < 0
    slot = ef.clamp(min=0)

    def some(X, theta, rates, k):
        p = dict(zip(("D", "rho", "mu", "beta", "v_som", "v_fom", "v_dom", "K_dom"), rates))
        g = torch.where(inside, torch.ones_like(ef, dtype=theta.dtype), theta.index_select(0, slot)) * (p["D"] * dt)
        X = tuple(X)
        for _ in range(k):
            x1, y, x3, x4, x5 = _transform(X, p, dt)
            flux = g * (y.index_select(0, ei) - y.index_select(0, ej))
            X = (x1, y.index_add(0, ei, -flux).index_add(0, ej, flux), x3, x4, x5)
        return torch.stack(X)

    seg = max(5, min(40, int(4e7 // max(1, X0.shape[1]))))
    X, done = X0, 0
    while done < steps:
        k = min(seg, steps - done)
        X = checkpoint(some, X, theta, rates, k, use_reentrant=False)
        done += k
    return X


def _coarse_geometry(vox, nbs, lab, q, shape):
    """(i, j, S_ij / d_ij) of every ordered adjacent pair in row order, and the volumes."""
    nz, ny, nx = shape
    vol = torch.bincount(lab, minlength=q).double()
    cen = torch.stack([torch.zeros(q, dtype=torch.float64, device="cuda").index_add_(0, lab, c.double()) / vol
                       for c in (vox % nx, vox // nx % ny, vox // (nx * ny))])
    keys = []
    for nb in nbs:
        i = (nb >= 0).nonzero().view(-1)
        a, b = lab[i], lab[nb[i]]
        keys.append((a * q + b)[a != b])
    key, S = torch.unique(torch.cat(keys), return_counts=True)
    i, j = key // q, key % q
    d = (cen[:, i] - cen[:, j]).square().sum(0).sqrt()
    return i, j, S.double() / d, vol


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        kepts, masses, per = [], [], []
        for k, (shape, por, scale) in enumerate(_batch_specs(case)):
            kept = _largest(_image(shape, por, salt=100 * (k + 1)))
            vox, nbs = _neighbours(kept)
            p = _params(case, scale)
            kepts.append(nbs)
            per.append(p)
            masses.append(_masses(vox, kept, seed, salt=100 * (k + 1)).double())
        sizes = [m.shape[1] for m in masses]
        offs = np.concatenate([[0], np.cumsum(sizes)])
        nbs = [torch.cat([torch.where(kepts[k][d] >= 0, kepts[k][d] + int(offs[k]), -1) for k in range(len(sizes))])
               for d in range(6)]
        p = dict(per[0])
        reps = torch.tensor(sizes, device="cuda")
        for key in ("rho", "mu", "v_som", "v_fom", "v_dom"):
            p[key] = torch.repeat_interleave(torch.tensor([x[key] for x in per], dtype=torch.float64, device="cuda"),
                                             reps)
        X = _explicit(torch.cat(masses, dim=1), nbs, p, case["steps"])
        return list(torch.split(X, sizes, dim=1))
    shape = _shape(case)
    kept = _largest(_image(shape, case["porosity"]))
    vox, nbs = _neighbours(kept)
    if kind in ("train", "coarse"):
        lab, q = _labels(vox, shape)
        i, j, th, vol = _coarse_geometry(vox, nbs, lab.long(), q, shape)
        data = _coarse_inputs(vol, seed)
        c = D_DOM * COARSE_DT
        if kind == "coarse":
            diag = vol + c * torch.zeros_like(vol).index_add_(0, i, th)
            m = data[0]
            for _ in range(case["steps"]):
                u = _cg(lambda v: vol * v + c * torch.zeros_like(v).index_add_(0, i, th * (v[i] - v[j])), m, diag, 1e-15)
                m = vol * u
            return dict(mass=m)
        order = torch.argsort(j * q + i)  # slot of (j, i) for every slot in row order
        rng = np.random.Generator(np.random.PCG64(int(seed)))
        lr, pairs, losses = 0.05 * float(th.mean()), _train_pairs(), []
        for epoch in range(case["epochs"]):
            if epoch > 0 and epoch % 10 == 0:
                lr *= 0.5
            sel = pairs[rng.choice(len(pairs), size=TRAIN_BATCH, replace=False)]
            x, y = data[torch.from_numpy(sel[:, 0]).long().cuda()], data[torch.from_numpy(sel[:, 1]).long().cuda()]
            dc = (y / vol)[:, i] - (y / vol)[:, j]
            res = x - y - c * torch.zeros_like(x).index_add_(1, i, th * dc)
            losses.append(float(res.square().sum()) / (TRAIN_BATCH * q))
            g = -(2 * c / (TRAIN_BATCH * q)) * (res[:, i] * dc).sum(0)
            th = (th - lr * torch.sign(g + g[order])).clamp(min=0.0)
        return dict(loss=np.array(losses), theta=th)
    X0 = _masses(vox, kept, seed, organic=case.get("organic", 0.0),
                 hydrolysable=kind in ("gradient", "autograd")).double()
    p = _params(case)
    if kind in ("gradient", "autograd"):
        theta = _theta(shape, seed).double().requires_grad_(True)
        rates = torch.tensor([p[k] for k in autograd.RATE_NAMES], dtype=torch.float64, device="cuda",
                             requires_grad=True)
        X0.requires_grad_(True)
        XN = _model(X0, theta, rates, _edges(vox, nbs, shape), case["steps"], p["dt"])
        if kind == "autograd":
            r = torch.randn((5, vox.numel()), generator=_gen(seed, 61), device="cuda", dtype=torch.float64)
            gt, gr, gx = torch.autograd.grad(XN, (theta, rates, X0), r)
            return dict(state=XN.detach(), gtheta=gt, grates=gr.cpu(), gx0=gx)
        nb = math.prod(_n_blocks(shape))
        blk = _block_of(vox, shape, BLOCK)
        zero = torch.zeros((2, nb), dtype=torch.float64, device="cuda")
        mass = zero.index_add(1, blk, torch.stack([XN[1], XN[4]]))
        loss = (mass - _block_targets(vox, shape, X0.detach(), seed)).square().sum()
        gt, gr = torch.autograd.grad(loss, (theta, rates))
        return dict(loss=float(loss), mass=mass.detach(), state=XN.detach(), grad=gr.cpu(), gtheta=gt)
    X = (_implicit if kind == "implicit" else _explicit)(X0, nbs, p, case["steps"])
    out = dict(totals=X.sum(dim=1), state=X)
    return dict(out, components=None, nodes=None) if kind == "image" else out
