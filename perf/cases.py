"""What a user of this framework has it do, as measurable cases.

Each case is one pass through the public entry points of the binding
(`paper_1912_10192_gb300.hamr`): a state is loaded from device memory, advanced
a few steps (or one period of the block tree) and read out whole; or a batch
of states is inverted; or the inversion's network is trained.  States come
from the repository's own generators (torus, tilted disk, flat box,
random inversion states) with the seeded perturbation applied on the device.
"""
import functools
import math

import numpy as np
import torch

from paper_1912_10192_gb300 import hamr
from paper_1912_10192_gb300 import workloads as W

SPIN, GAM, COUR, NG = 0.9375, 13.0 / 9.0, 0.8, 3
F64 = torch.float64
BC_TORUS = (hamr.BC_OUTFLOW_NOINFLOW, hamr.BC_OUTFLOW_NOINFLOW, hamr.BC_POLAR, hamr.BC_POLAR, hamr.BC_PERIODIC,
            hamr.BC_PERIODIC)
# FP64 operations of the plain scheme per cell and step (tests/golden/flops_per_unit.json)
OPS_PER_ZONE_CYCLE = 4605.0
NPARAM, TRAIN_SET = 9154, 1 << 18


def listed():
    return [
        # the smallest call: a host framework's own block, one step without any allocation
        _block("noalloc_24x12x8", "noalloc", 24, 12, 8, steps=1),
        # the plain method's validation block: a few hundred kernels on 32k cells, launches count
        _block("torus_64x32x16", "torus", 64, 32, 16, steps=4),
        # the headline block in FP64 and in the mixed form that production runs choose
        _block("torus_256x128x64", "torus", 256, 128, 64, steps=2),
        _block("torus_256x128x64_mixed", "torus", 256, 128, 64, steps=4, precision=1),
        # a block whose sizes fit no tile, mixed form
        _block("torus_53x37x22_mixed", "torus", 53, 37, 22, steps=4, precision=1),
        # odd sizes with the paper's usual upwinded EMFs and the shock flattener
        _block("options_97x61x34", "torus", 97, 61, 34, steps=2, emf=1, flatten=1),
        # the tilted thin disk at half the resolution of its production grid
        _block("disk_224x96x192_mixed", "disk", 224, 96, 192, steps=2, precision=1),
        # a small refined periodic box: many tiny blocks, two time levels, four periods
        {"name": "tree_box_8", "kind": "tree", "tree": "box", "n": 8, "precision": 0, "periods": 4, "smr": 0},
        # the 512-block torus tree with two refinement levels and four time levels, one whole period
        {"name": "tree_c3_32", "kind": "tree", "tree": "c3", "n": 32, "precision": 0, "periods": 1, "smr": 0},
        {"name": "tree_c3_32_mixed", "kind": "tree", "tree": "c3", "n": 32, "precision": 1, "periods": 1, "smr": 0},
        # stand-alone inversion of a batch of states, start 5% off (re-inversion after another code's step)
        {"name": "con2prim_1000003", "kind": "c2p", "n": 1000003, "cold": False, "network": False, "flags": 0},
        # training of the inversion's network: 32 optimiser steps of the batch that the framework trains with
        {"name": "train_8192", "kind": "train", "batch": 8192, "steps": 32},
    ]


def _block(name, state, n1, n2, n3, steps, precision=0, emf=0, flatten=0, inversion=0, floor_frame=0, smr=0):
    return {"name": name, "kind": "block", "state": state, "n1": n1, "n2": n2, "n3": n3, "steps": steps,
            "precision": precision, "emf": emf, "flatten": flatten, "inversion": inversion,
            "floor_frame": floor_frame, "smr": smr}


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "torus", "torus", "torus", "disk", "box", "c3", "c2p", "c2p", "train"])
    if kind == "noalloc":  # up to the entry point's limit of padded cells
        while True:
            n1, n2, n3 = rng.randint(5, 40), rng.randint(5, 24), 2 * rng.randint(2, 9)
            if (n1 + 6) * (n2 + 6) * (n3 + 6) <= 12288 and (n1 + 6) * (n2 + 6) <= 1536:
                break
        c = _block("", "noalloc", n1, n2, n3, steps=1, emf=rng.randint(0, 1), flatten=rng.randint(0, 1))
    elif kind in ("torus", "disk"):
        f = 1 if kind == "torus" else 2  # the disk wants its vertical resolution
        n1, n2, n3 = _spread(rng, 24 * f, 256), _spread(rng, 16 * f, 128), 2 * _spread(rng, 5 * f, 40)
        prec = rng.choice([0, 1, 1, 2]) if kind == "torus" else 1
        smr = rng.choice([0, 0, 0, 1]) if kind == "torus" else 0
        if smr:
            n3 = max(8, n3 // 4 * 4)
        c = _block("", kind, n1, n2, n3, steps=rng.randint(1, 3), precision=prec, emf=rng.randint(0, 1),
                   flatten=rng.randint(0, 1), inversion=rng.choice([0, 0, 0, 1]),
                   floor_frame=rng.choice([0, 0, 0, 1]), smr=smr)
    elif kind == "box":
        c = {"kind": "tree", "tree": "box", "n": rng.randint(6, 24), "precision": rng.randint(0, 1),
             "periods": rng.randint(1, 4), "smr": 0}
    elif kind == "c3":
        c = {"kind": "tree", "tree": "c3", "n": 4 * rng.randint(2, 7), "precision": rng.randint(0, 1), "periods": 1,
             "smr": 0}
    elif kind == "c2p":
        net = rng.random() < 0.4
        c = {"kind": "c2p", "n": _spread(rng, 500, 2000000), "cold": net and rng.random() < 0.5, "network": net,
             "flags": 0 if net else rng.choice([0, 0, hamr.C2P_AITKEN, hamr.C2P_MIXED])}
    else:
        c = {"kind": "train", "batch": 128 * _spread(rng, 4, 256), "steps": rng.randint(8, 48)}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs

def _device(arrays):
    return tuple(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in arrays)


@functools.lru_cache(maxsize=4)
def _block_base(state, n1, n2, n3):
    """Geometry and unperturbed device state of a block; the same for every seed."""
    if state == "disk":
        geo = W.disk_geometry(n1, n2, n3)
        return (geo,) + _device(W.tilted_disk_block(geo, pert=0.0))
    geo = W.torus_geometry(n1, n2, n3)
    return (geo,) + _device(W.torus_block(geo, pert=0.0))


def _box_blocks(n):
    return W.flat_box_tree(base=(2, 2, 2), n=n, refine=((0, 0, 0),), lat_coarse=1, lat_fine=0)


@functools.lru_cache(maxsize=2)
def _tree_base(tree, n, smr):
    """Blocks of a tree, the views of one block's fields in two flat arrays, and the unperturbed arrays."""
    blocks = _box_blocks(n) if tree == "box" else W.c3_tree(n=n, smr=smr)
    states = W.flat_box_state(blocks) if tree == "box" else W.torus_blocks(blocks, pert=0.0)
    prim = torch.from_numpy(np.concatenate([p.reshape(-1) for p, _ in states])).cuda()
    bface = torch.from_numpy(np.concatenate([b.reshape(-1) for _, b in states])).cuda()
    return blocks, prim, bface


def _block_views(blocks, flat, nf):
    out, at = [], 0
    for b in blocks:
        shp = (nf, b["n3"] + 2 * NG, b["n2"] + 2 * NG, b["n1"] + 2 * NG)
        n = math.prod(shp)
        out.append(flat[at:at + n].view(shp))
        at += n
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _perturbed(u, seed):
    """u_g with the seeded 2% perturbation that starts the instabilities."""
    xi = torch.rand(u.shape, generator=_generator(seed), device="cuda", dtype=F64)
    return u * (1.0 + 0.02 * (2.0 * xi - 1.0))


@functools.lru_cache(maxsize=2)
def _training_set(n):
    """Inputs and targets of n random states, and the fitted standardisation, for the network."""
    pr, x1, x2 = W.random_states(n, seed=500)
    P, x1, x2 = _device((pr.T, x1, x2))
    U = torch.empty((6, n), dtype=F64, device="cuda")
    hamr.prim2cons(P, x1, x2, U, a=SPIN, gam=GAM)
    feat = torch.empty((10, n), dtype=torch.float32, device="cuda")
    targ = torch.empty((2, n), dtype=torch.float32, device="cuda")
    hamr.Mlp.features(U, P[5:8].contiguous(), x1, x2, feat, prim=P, targ=targ, a=SPIN, gam=GAM)
    m = hamr.Mlp(seed=7)
    m.fit_norm(feat, targ)
    norm = m.params()[1]
    m.close()
    return feat, targ, norm


@functools.lru_cache(maxsize=1)
def _trained():
    """Parameters of a network trained as the framework trains it (a short run)."""
    feat, targ, norm = _training_set(TRAIN_SET)
    m = hamr.Mlp(seed=7)
    m.set_params(norm=norm)
    m.train(feat, targ, steps=1500, batch=8192)
    p = m.params()
    m.close()
    return p


def _train_inputs(case, seed):
    """A training set of its own and the initial parameters: the shared set's columns in a seeded order."""
    feat, targ, norm = _training_set(TRAIN_SET)
    at = torch.randperm(TRAIN_SET, generator=_generator(seed), device="cuda")
    return feat[:, at].contiguous(), targ[:, at].contiguous(), norm


def _c2p_inputs(case, seed):
    n = case["n"]
    pr, x1, x2 = W.random_states(n, seed=int(seed) + 1)
    P, x1, x2 = _device((pr.T, x1, x2))
    g = _metric(x1, x2)
    # the conserved state of the true primitives, and the guess that the caller has
    U = _cons(P, _state(P, g), g, _kappa(P))
    guess = P.clone()
    if case["cold"]:
        guess[1] = 1e-3 * guess[0]
        guess[2:5] = 0.0
    else:
        guess[0] *= 1.05
        guess[1] *= 0.95
        guess[2:5] *= 1.02
    return P, U.contiguous(), x1, x2, guess


def prepare(case, seed):
    k = case["kind"]
    if k == "block":
        geo, prim, bface = _block_base(case["state"], case["n1"], case["n2"], case["n3"])
        prim = prim.clone()
        prim[1] = _perturbed(prim[1], seed)
        blk = hamr.block(geo.n1, geo.n2, geo.n3, geo.x1min, geo.x2min, geo.x3min, geo.dx1, geo.dx2, geo.dx3, BC_TORUS)
        grid = hamr.Grid([blk], a=SPIN, gam=GAM, cour=COUR, precision=case["precision"], emf=case["emf"],
                         flatten=case["flatten"], inversion=case["inversion"], floor_frame=case["floor_frame"],
                         smr=case["smr"])
        return {"case": case, "grid": grid, "in": (prim, bface), "out": (prim.clone(), bface.clone())}
    if k == "tree":
        blocks, prim, bface = _tree_base(case["tree"], case["n"], case["smr"])
        views = _block_views(blocks, prim.clone(), 8)
        for i, v in enumerate(views):
            v[1] = _perturbed(v[1], seed * 100003 + i)
        phys = dict(a=SPIN, gam=GAM, cour=COUR) if case["tree"] == "c3" else dict(
            metric=hamr.METRIC_MINKOWSKI, gam=5.0 / 3.0, cour=0.5, floors=0)
        grid = hamr.Grid([hamr.block_from_dict(b) for b in blocks], precision=case["precision"], smr=case["smr"],
                         **phys)
        out = (torch.empty_like(prim), torch.empty_like(bface))
        return {"case": case, "grid": grid, "in": (views, _block_views(blocks, bface, 3)), "out": out,
                "views": (_block_views(blocks, out[0], 8), _block_views(blocks, out[1], 3)),
                "substeps": case["periods"] << max(b["lat"] for b in blocks)}
    if k == "c2p":
        P, U, x1, x2, guess = _c2p_inputs(case, seed)
        net = None
        if case["network"]:
            net = hamr.Mlp(seed=7)
            net.set_params(*_trained())
        return {"case": case, "U": U, "B": P[5:8].contiguous(), "x": (x1, x2), "guess": guess, "net": net,
                "prim": guess.clone(), "status": torch.zeros(case["n"], dtype=torch.int32, device="cuda")}
    feat, targ, norm = _train_inputs(case, seed)
    net = hamr.Mlp(seed=7)
    net.set_params(norm=norm)
    return {"case": case, "net": net, "in": (feat, targ)}


# ---------------------------------------------------------------- one pass

def run(s):
    c = s["case"]
    if c["kind"] == "block" and c["state"] == "noalloc":
        prim, bface = s["out"]
        prim.copy_(s["in"][0])
        bface.copy_(s["in"][1])
        hamr.block_step_noalloc(s["grid"], prim, bface)
        return {"prim": prim, "bface": bface}
    if c["kind"] == "block":
        g = s["grid"]
        g.set_state(*s["in"])
        for _ in range(c["steps"]):
            g.step()
        g.get_state(prim=s["out"][0], bface=s["out"][1])
        return {"prim": s["out"][0], "bface": s["out"][1]}
    if c["kind"] == "tree":
        g = s["grid"]
        for i, (p, b) in enumerate(zip(*s["in"])):
            g.set_state(p, b, block=i)
        g.batch_step(s["substeps"])
        for i, (p, b) in enumerate(zip(*s["views"])):
            g.get_state(block=i, prim=p, bface=b)
        return {"prim": s["out"][0], "bface": s["out"][1]}
    if c["kind"] == "c2p":
        s["prim"].copy_(s["guess"])
        hamr.con2prim(s["U"], s["B"], s["x"][0], s["x"][1], s["prim"], s["status"], a=SPIN, gam=GAM, flags=c["flags"],
                      mlp=s["net"])
        return {"prim": s["prim"], "status": s["status"]}
    loss = s["net"].train(*s["in"], steps=c["steps"], batch=c["batch"])
    return {"loss": loss, "params": s["net"].params()[0]}


def work(case):
    k = case["kind"]
    if k == "block":
        n = case["n1"] * case["n2"] * case["n3"]
        return {"bytes": 2.0 * 88 * n, "flops": OPS_PER_ZONE_CYCLE * n * case["steps"]}
    if k == "tree":
        if case["tree"] == "box":
            shapes = [(case["n"] ** 3, b["lat"]) for b in _box_blocks(8)]
        else:  # counts of the 512-block tree: (cells of a block, LAT level, blocks) as workloads.c3_tree assigns them
            full = W.c3_tree(n=case["n"], smr=case["smr"])
            shapes = [(b["n1"] * b["n2"] * b["n3"], b["lat"]) for b in full]
        top = max(lat for _, lat in shapes)
        cells = sum(n for n, _ in shapes)
        cycles = sum(n << (top - lat) for n, lat in shapes) * case["periods"]
        return {"bytes": 2.0 * 88 * cells, "flops": OPS_PER_ZONE_CYCLE * cycles}
    if k == "c2p":  # conserved state, field, position and guess in, primitives and status out; about 5 iterations
        return {"bytes": 220.0 * case["n"], "flops": 500.0 * case["n"]}
    rows = case["batch"] * case["steps"]
    return {"bytes": 48.0 * rows + 16.0 * NPARAM * case["steps"], "flops": 6.0 * 9000 * rows}


# ---------------------------------------------------------------- the same in plain torch, 64 bits

def exact(case, seed):
    k = case["kind"]
    if k == "block":
        if case["inversion"] or case["floor_frame"] or case["smr"]:
            return None
        geo, prim, bface = _block_base(case["state"], case["n1"], case["n2"], case["n3"])
        prim = prim.clone()
        prim[1] = _perturbed(prim[1], seed)
        P, B = _Scheme(geo, case["emf"], case["flatten"]).advance(prim, bface.clone(), case["steps"])
        return {"prim": P, "bface": B}
    if k == "c2p":  # the primitives that the conserved states were formed from; every start here reaches them
        if case["cold"]:
            return None
        return {"prim": _c2p_inputs(case, seed)[0], "status": None}
    if k == "train":
        return _exact_train(case, seed)
    return None


def _exact_train(case, seed):
    feat, targ, norm = _train_inputs(case, seed)
    m = hamr.Mlp(seed=7)
    theta = torch.from_numpy(m.params()[0]).cuda().double()  # the initial parameters are an input
    m.close()
    nrm = torch.from_numpy(norm).cuda().double()
    X = (feat.double().T - nrm[:10]) / nrm[10:20]
    Y = (targ.double().T - nrm[20:22]) / nrm[22:24]
    m1, m2, losses, n, bt = torch.zeros_like(theta), torch.zeros_like(theta), [], X.shape[0], case["batch"]
    for k in range(case["steps"]):
        at = torch.from_numpy((W.splitmix64(np.uint64(5) ^ np.arange(k * bt, (k + 1) * bt, dtype=np.uint64))
                               % np.uint64(n)).astype(np.int64)).cuda()
        p = theta.clone().requires_grad_(True)
        h, o = X[at], 0
        for rows, cols in ((64, 10), (64, 64), (64, 64), (2, 64)):
            h = h @ p[o:o + rows * cols].view(rows, cols).T + p[o + rows * cols:o + rows * cols + rows]
            o += rows * cols + rows
            if rows == 64:
                h = torch.tanh(h)
        loss = ((h - Y[at]) ** 2).sum() / (2 * bt)
        g, = torch.autograd.grad(loss, p)
        losses.append(float(loss))
        t = k + 1
        lr = 2e-5 + 0.5 * (2e-3 - 2e-5) * (1.0 + math.cos(math.pi * k / max(case["steps"] - 1, 1)))
        m1 = 0.9 * m1 + 0.1 * g
        m2 = 0.999 * m2 + 0.001 * g * g
        theta = theta - lr * (m1 / (1 - 0.9 ** t)) / ((m2 / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"loss": np.array(losses), "params": theta.cpu().numpy()}


def _metric(x1, x2):
    """Kerr-Schild metric in (t, log r, theta, phi): g[mn], inverse c[mn], sqrt(-g), lapse."""
    th = torch.where(x2 < 0, -x2, torch.where(x2 > math.pi, 2 * math.pi - x2, x2))
    r, s, co = torch.exp(x1), torch.sin(th), torch.cos(th)
    a, s2 = SPIN, s * s
    sig = r * r + a * a * co * co
    z = 2 * r / sig
    o = torch.zeros_like(sig)
    g = {"g00": z - 1, "g01": z * r, "g03": -z * a * s2, "g11": (1 + z) * r * r, "g13": -(1 + z) * a * s2 * r,
         "g22": sig, "g33": s2 * (sig + (1 + z) * a * a * s2), "c00": -(1 + z), "c01": z / r,
         "c11": (r * r - 2 * r + a * a) / (sig * r * r), "c13": a / (sig * r), "c22": 1 / sig,
         "c33": 1 / (sig * torch.where(s2 > 0, s2, o + 1)), "det": r * sig * s, "alpha": 1 / torch.sqrt(1 + z)}
    g["idet"] = torch.where(g["det"] != 0, 1 / torch.where(g["det"] != 0, g["det"], o + 1), o)
    return g


def _lower(g, v):
    return [g["g00"] * v[0] + g["g01"] * v[1] + g["g03"] * v[3], g["g01"] * v[0] + g["g11"] * v[1] + g["g13"] * v[3],
            g["g22"] * v[2], g["g03"] * v[0] + g["g13"] * v[1] + g["g33"] * v[3]]


def _state(P, g):
    """u^mu, u_mu, b^mu, b_mu, b^2 of primitives P."""
    q1, q2, q3 = P[2], P[3], P[4]
    gamma = torch.sqrt(1 + g["g11"] * q1 * q1 + g["g22"] * q2 * q2 + g["g33"] * q3 * q3 + 2 * g["g13"] * q1 * q3)
    u = [gamma / g["alpha"], q1 - gamma * g["alpha"] * g["c01"], q2, q3]
    ul = _lower(g, u)
    bt = P[5] * ul[1] + P[6] * ul[2] + P[7] * ul[3]
    b = [bt] + [(P[4 + i] + bt * u[i]) / u[0] for i in (1, 2, 3)]
    bl = _lower(g, b)
    return u, ul, b, bl, sum(x * y for x, y in zip(b, bl))


def _kappa(P):
    return (GAM - 1) * P[1] * P[0] ** (-GAM)


def _row(P, st, kap, d):
    """rho u^d, T^d_t + rho u^d, T^d_i, kappa rho u^d (d = 0: conserved, else flux), without sqrt(-g)."""
    u, ul, b, bl, b2 = st
    eta, pt = P[0] + GAM * P[1] + b2, (GAM - 1) * P[1] + b2 / 2
    t = [eta * u[d] * ul[n] - b[d] * bl[n] + (pt if n == d else 0) for n in range(4)]
    return [P[0] * u[d], t[0] + P[0] * u[d], t[1], t[2], t[3], kap * P[0] * u[d]]


def _cons(P, st, g, kap):
    return torch.stack([x * g["det"] for x in _row(P, st, kap, 0)])


def _quad(P, st, g, d):
    """The fast-speed quadratic along d: A, B and the root of its discriminant."""
    u, _, _, _, b2 = st
    p = (GAM - 1) * P[1]
    num, dn = b2 + GAM * p, P[0] + P[1] + p - GAM * p
    gtd, gdd = (g["c01"] if d == 1 else 0.0), g["c%d%d" % (d, d)]
    A = u[0] * u[0] * dn - num * g["c00"]
    B = u[0] * u[d] * dn - num * gtd
    return A, B, torch.sqrt(torch.clamp(B * B - A * (u[d] * u[d] * dn - num * gdd), min=0))


class _Scheme:
    """The midpoint step of one spherical block in plain torch, fields padded as the framework's."""

    def __init__(self, geo, upwind, flatten):
        self.n = (geo.n1, geo.n2, geo.n3)
        self.dx = (geo.dx1, geo.dx2, geo.dx3)
        self.upwind, self.flatten = upwind, flatten
        ax = lambda lo, h, n, f: lo + (torch.arange(-NG, n + NG, device="cuda", dtype=F64) + f) * h  # noqa: E731
        c1, f1 = ax(geo.x1min, geo.dx1, geo.n1, 0.5), ax(geo.x1min, geo.dx1, geo.n1, 0.0)
        c2, f2 = ax(geo.x2min, geo.dx2, geo.n2, 0.5), ax(geo.x2min, geo.dx2, geo.n2, 0.0)
        grid = lambda x, y: (x[None, None, :].expand(1, len(y), len(x)), y[None, :, None].expand(1, len(y), len(x)))  # noqa: E731
        self.gc, self.gf = _metric(*grid(c1, c2)), [_metric(*grid(f1, c2)), _metric(*grid(c1, f2))]
        for j in (NG, NG + geo.n2):  # no area on the axis
            self.gf[1]["det"][:, j] = 0.0
            self.gf[1]["idet"][:, j] = 0.0
        self.gf.append(self.gc)
        h, self.dg = 1e-3, []
        for s in (0, 1):
            at = lambda m: _metric(*grid(c1 + (m * h if s == 0 else 0), c2 + (m * h if s else 0)))  # noqa: E731
            m = {k: at(k) for k in (-2, -1, 1, 2)}
            self.dg.append({q: (8 * (m[1][q] - m[-1][q]) - (m[2][q] - m[-2][q])) / (12 * h)
                            for q in ("g00", "g01", "g03", "g11", "g13", "g22", "g33")})
        r = torch.exp(c1)[None, None, :]
        self.rhoflr, self.uflr = 1e-7 / r ** 2, 1e-9 * r ** (-10.0 / 3.0)

    def cut(self, x, lo=(0, 0, 0), hi=(0, 0, 0)):
        """x over cells lo[d] .. n_d - 1 + hi[d]; metric planes are one cell thick in x3."""
        i, j, k = (slice(NG + lo[d], NG + self.n[d] + hi[d]) for d in range(3))
        if isinstance(x, dict):
            return {q: v[:, j, i] for q, v in x.items()}
        return x[..., j, i] if x.shape[-3] == 1 else x[..., k, j, i]

    def bc(self, P, B):
        n1, n2, n3 = self.n
        for X in (P, B):  # x3 periodic; x3-face n3 is face 0
            X[:, :NG] = X[:, n3:n3 + NG].clone()
            X[:, NG + n3:] = X[:, NG:2 * NG].clone()
        k = torch.arange(-NG, n3 + NG, device="cuda")
        src = NG + (k + n3 // 2) % n3
        for m in range(NG):  # polar axes: the cells across them, theta components reversed
            for dst, cell, face, fdst in ((NG - 1 - m, NG + m, NG + 1 + m, NG - 1 - m),
                                          (NG + n2 + m, NG + n2 - 1 - m, NG + n2 - 1 - m, NG + n2 + 1 + m)):
                P[:, :, dst] = P[:, src, cell]
                P[3, :, dst] *= -1
                P[6, :, dst] *= -1
                B[0, :, dst] = B[0, src, cell]
                B[2, :, dst] = B[2, src, cell]
                if fdst < n2 + 2 * NG:
                    B[1, :, fdst] = -B[1, src, face]
        B[1, :, NG] = 0.0
        B[1, :, NG + n2] = 0.0
        for m in range(NG):  # x1 outflow without inflow
            for dst, cell, sign in ((NG - 1 - m, NG, 1.0), (NG + n1 + m, NG + n1 - 1, -1.0)):
                P[:, :, :, dst] = P[:, :, :, cell]
                P[2, :, :, dst] = sign * torch.clamp(sign * P[2, :, :, dst], max=0.0)
                B[1, :, :, dst] = B[1, :, :, cell]
                B[2, :, :, dst] = B[2, :, :, cell]
            B[0, :, :, NG - 1 - m] = B[0, :, :, NG]
            if NG + n1 + 1 + m < n1 + 2 * NG:
                B[0, :, :, NG + n1 + 1 + m] = B[0, :, :, NG + n1]

    def centre(self, B):
        c, g = self.cut, self.cut(self.gc)
        up = lambda d: tuple(1 if q == d else 0 for q in range(3))  # noqa: E731
        return [0.5 * (c(B[d]) + c(B[d], up(d), up(d))) * g["idet"] for d in range(3)]

    def edges(self, q, d, flat):
        """Left and right PPM edge values of cells -1 .. n_d along d (whole padded extent across)."""
        dim, n = q.dim() - 1 - d, self.n[d]
        w = lambda o: q.narrow(dim, NG - 1 + o, n + 2)  # noqa: E731
        qs = [w(o) for o in (-2, -1, 0, 1, 2)]
        def slope(a, b, c):
            dl, dr, dc = b - a, c - b, 0.5 * (c - a)
            mag = torch.minimum(dc.abs(), 2 * torch.minimum(dl.abs(), dr.abs()))
            return torch.where(dl * dr > 0, mag * torch.sign(dc), torch.zeros_like(mag))
        sm, sc, sp = (slope(*qs[k:k + 3]) for k in range(3))
        lo = 0.5 * (qs[1] + qs[2]) - (sc - sm) / 6
        hi = 0.5 * (qs[2] + qs[3]) - (sp - sc) / 6
        c = qs[2]
        if flat is not None:
            lo, hi = flat * c + (1 - flat) * lo, flat * c + (1 - flat) * hi
        da, a6, mono = hi - lo, 6 * (c - 0.5 * (lo + hi)), (hi - c) * (c - lo) > 0
        l2 = torch.where(da * a6 > da * da, 3 * c - 2 * hi, lo)
        h2 = torch.where(-da * da > da * a6, 3 * c - 2 * lo, hi)
        return torch.where(mono, l2, c), torch.where(mono, h2, c)

    def flattening(self, P, d):
        dim, n = 2 - d, self.n[d]
        w = lambda q, o: P[q].narrow(dim, NG - 1 + o, n + 2)  # noqa: E731
        pm, pp = (GAM - 1) * w(1, -1), (GAM - 1) * w(1, 1)
        a1, a2 = (pp - pm).abs(), ((GAM - 1) * (w(1, 2) - w(1, -2))).abs()
        f = torch.where(a2 > 0, (10 * (a1 / a2 - 0.75)).clamp(0, 1), torch.ones_like(a1))
        return torch.where((a1 > 0.33 * torch.minimum(pm, pp)) & (w(2 + d, -1) > w(2 + d, 1)), f, torch.zeros_like(a1))

    def fluxes(self, P, B, d):
        """HLL fluxes (6 rows and the three B slots, sqrt(-g) in) at faces 0 .. n_d, padded across."""
        dim, n = 2 - d, self.n[d]
        flat = self.flattening(P, d) if self.flatten else None
        lo, hi = self.edges(torch.cat([P, _kappa(P)[None]]), d, flat)
        left, right = hi.narrow(dim + 1, 0, n + 1), lo.narrow(dim + 1, 1, n + 1)
        g = self.gf[d] if d == 2 else {q: v.narrow(dim, NG, n + 1) for q, v in self.gf[d].items()}
        bn = B[d].narrow(dim, NG, n + 1) * g["idet"]
        side = []
        for e in (left, right):
            p = [bn if q == 5 + d else e[q] for q in range(8)]
            st = _state(p, g)
            A, Bq, sd = _quad(p, st, g, d + 1)
            u, _, b, _, _ = st
            F = _row(p, st, e[8], d + 1) + [b[i] * u[d + 1] - b[d + 1] * u[i] for i in (1, 2, 3)]
            side.append(((Bq + sd) / A, (Bq - sd) / A, F, _row(p, st, e[8], 0) + [p[5], p[6], p[7]]))
        (pl, ml, Fl, Ul), (pr, mr, Fr, Ur) = side
        cp = torch.maximum(pl, pr).clamp(min=0)
        cm = torch.maximum(-ml, -mr).clamp(min=0)
        F = torch.stack([(cm * fr + cp * fl - cp * cm * (ur - ul)) / (cp + cm) * g["det"]
                         for fl, fr, ul, ur in zip(Fl, Fr, Ul, Ur)])
        F = torch.where((g["det"] == 0).expand_as(F[0]), torch.zeros_like(F), F)
        full = torch.zeros((9,) + P.shape[1:], device="cuda", dtype=F64)
        full.narrow(dim + 1, NG, n + 1).copy_(F)
        return full

    def emfs(self, P, F):
        n1, n2, n3 = self.n
        full = lambda x, o: x[NG + o[2]:NG + n3 + 1 + o[2], NG + o[1]:NG + n2 + 1 + o[1], NG + o[0]:NG + n1 + 1 + o[0]]  # noqa: E731
        st = _state(P, self.gc) if self.upwind else None
        out = []
        for e in range(3):
            p, q = (e + 1) % 3, (e + 2) % 3
            if p > q:
                p, q = q, p
            sg = 1.0 if e == 1 else -1.0  # the EMF that a p-face carries is sg F_p(B^q), a q-face -sg F_q(B^p)
            off = lambda *ds: tuple(-sum(1 for x in ds if x == k) for k in range(3))  # noqa: E731
            fp, fq, mp, mq = sg * F[p][6 + q], -sg * F[q][6 + p], F[p][0], F[q][0]
            E = 0.25 * (full(fp, off()) + full(fp, off(q)) + full(fq, off()) + full(fq, off(p)))
            if self.upwind:
                u, _, b, _, _ = st
                i, j = (e + 1) % 3 + 1, (e + 2) % 3 + 1
                ec = (b[i] * u[j] - b[j] * u[i]) * self.gc["det"]
                pick = lambda m, lo, hi: torch.where(m > 0, lo, torch.where(m < 0, hi, 0.5 * (lo + hi)))  # noqa: E731
                v = lambda x, *ds: full(x, off(*ds))  # noqa: E731
                E = E + 0.25 * (pick(v(mp, q), v(fq, p) - v(ec, p, q), v(fq) - v(ec, q))
                                - pick(v(mp), v(ec, p) - v(fq, p), v(ec) - v(fq))
                                + pick(v(mq, p), v(fp, q) - v(ec, p, q), v(fp) - v(ec, p))
                                - pick(v(mq), v(ec, q) - v(fp, q), v(ec) - v(fp)))
            if e != 1:
                E[:, 0] = 0.0
                E[:, n2] = 0.0
            out.append(E)
        return out

    def curl(self, B, E, dt):
        n1, n2, n3 = self.n
        E1, E2, E3 = E
        d1, d2, d3 = self.dx
        k, j, i = slice(NG, NG + n3), slice(NG, NG + n2), slice(NG, NG + n1)
        k1, j1, i1 = slice(NG, NG + n3 + 1), slice(NG, NG + n2 + 1), slice(NG, NG + n1 + 1)
        B = B.clone()
        B[0, k, j, i1] += dt * ((E2[1:, :n2] - E2[:-1, :n2]) / d3 - (E3[:n3, 1:] - E3[:n3, :-1]) / d2)
        B[1, k, j1, i] += dt * ((E3[:n3, :, 1:] - E3[:n3, :, :-1]) / d1 - (E1[1:, :, :n1] - E1[:-1, :, :n1]) / d3)
        B[1, :, NG] = 0.0
        B[1, :, NG + n2] = 0.0
        B[2, k1, j, i] += dt * ((E1[:, 1:, :n1] - E1[:, :-1, :n1]) / d2 - (E2[:, :n2, 1:] - E2[:, :n2, :-1]) / d1)
        return B

    def stage(self, P, B, Un, Bn, dt):
        """One stage: fluxes and sources of (P, B) advance the conserved state Un and faces Bn by dt."""
        c = self.cut
        F = [self.fluxes(P, B, d) for d in range(3)]
        Bo = self.curl(Bn, self.emfs(P, F), dt)
        U = Un.clone()
        for d in range(3):
            up = tuple(1 if q == d else 0 for q in range(3))
            U -= dt / self.dx[d] * (c(F[d][:6], up, up) - c(F[d][:6]))
        Pi, g = c(P), c(self.gc)
        u, _, b, _, b2 = _state(Pi, g)
        eta, pt = Pi[0] + GAM * Pi[1] + b2, (GAM - 1) * Pi[1] + b2 / 2
        for s in (0, 1):
            for q, dq in self.dg[s].items():
                m, n = int(q[1]), int(q[2])
                inv = g.get("c" + q[1:], 0.0)
                T = eta * u[m] * u[n] - b[m] * b[n] + pt * inv
                U[2 + s] += dt * g["det"] * T * c(dq) * (0.5 if m == n else 1.0)
        Po = P.clone()
        i, j, k = (slice(NG, NG + n) for n in self.n)
        Po[:, k, j, i] = self.invert(U, self.centre(Bo), Pi, g)
        self.bc(Po, Bo)
        return Po, Bo

    def invert(self, U, Bc, guess, g):
        shape = guess.shape
        ext = lambda x: x.expand(shape[1:]).reshape(-1)  # noqa: E731
        g = {q: ext(v) for q, v in g.items()}
        U, pr = U.reshape(6, -1), guess.reshape(8, -1).clone()
        Bc = [x.reshape(-1) for x in Bc]
        al, gfac = g["alpha"], (GAM - 1) / GAM
        D = U[0] * al * g["idet"]
        Q = [(U[1] - U[0]) * al * g["idet"]] + [U[q] * al * g["idet"] for q in (2, 3, 4)]
        Qc = [g["c00"] * Q[0] + g["c01"] * Q[1], g["c01"] * Q[0] + g["c11"] * Q[1] + g["c13"] * Q[3], g["c22"] * Q[2],
              g["c13"] * Q[1] + g["c33"] * Q[3]]
        Bn = [al * x for x in Bc]
        Qn = -al * Qc[0]
        Qt2 = sum(x * y for x, y in zip(Q, Qc)) + Qn * Qn
        B2 = g["g11"] * Bn[0] ** 2 + g["g22"] * Bn[1] ** 2 + g["g33"] * Bn[2] ** 2 + 2 * g["g13"] * Bn[0] * Bn[2]
        QB = Q[1] * Bn[0] + Q[2] * Bn[1] + Q[3] * Bn[2]
        QB2, vmax = QB * QB, 1 - 1 / 2500.0
        q = pr[2:5]
        q2 = g["g11"] * q[0] ** 2 + g["g22"] * q[1] ** 2 + g["g33"] * q[2] ** 2 + 2 * g["g13"] * q[0] * q[2]
        W0 = (pr[0] + GAM * pr[1]) * (1 + q2)
        w, v = W0.clone(), (q2 / (1 + q2)).clamp(max=vmax)
        live, ok = torch.ones_like(w, dtype=torch.bool), torch.zeros_like(w, dtype=torch.bool)
        for _ in range(30):
            x = 1 - v
            p = gfac * (w * x - D * x.sqrt())
            f1 = -0.5 * B2 * (1 + v) + 0.5 * QB2 / w ** 2 - w + p - Qn
            f2 = v * (B2 + w) ** 2 - QB2 * (B2 + 2 * w) / w ** 2 - Qt2
            a = -QB2 / w ** 3 - 1 + gfac * x
            b = -0.5 * B2 + gfac * (0.5 * D / x.sqrt() - w)
            cc = 2 * (B2 + w) * (v + QB2 / w ** 3)
            e = (B2 + w) ** 2
            det = a * e - b * cc
            wn = w + (b * f2 - e * f1) / det
            vn = (v + (cc * f1 - a * f2) / det).clamp(0, vmax)
            live = live & (wn > 0)
            done = live & ((wn - w).abs() + (vn - v).abs() * wn < 1e-10 * wn)
            w, v = torch.where(live, wn, w), torch.where(live, vn, v)
            ok, live = ok | done, live & ~done
            if not bool(live.any()):
                break
        sq = (1 - v).sqrt()
        rho, u = D * sq, (w * (1 - v) - D * sq) / GAM
        ok = ok & (rho > 0) & (u > 0)
        at = torch.nonzero(~ok).reshape(-1)
        keep = torch.zeros_like(ok)
        if len(at):  # the entropy equation where the energy one has no root
            d, b2, qb2, qt2, kap = D[at], B2[at], QB2[at], Qt2[at], U[5][at] / U[0][at]
            gr, w1 = GAM / (GAM - 1), W0[at].clone()
            live, good = torch.ones_like(at, dtype=torch.bool), torch.zeros_like(at, dtype=torch.bool)
            for _ in range(30):
                bw = b2 + w1
                num, den = qt2 * w1 ** 2 + qb2 * (b2 + 2 * w1), (w1 * bw) ** 2
                vs = num / den
                dvs = (2 * (qt2 * w1 + qb2) - num * 2 * w1 * bw * (b2 + 2 * w1) / den) / den
                dvs, vs = torch.where(vs > vmax, torch.zeros_like(dvs), dvs), vs.clamp(max=vmax)
                s = (1 - vs).sqrt()
                rh = d * s
                pp = kap * rh ** GAM
                f = w1 * (1 - vs) - rh - gr * pp
                df = 1 - vs - w1 * dvs + 0.5 * d / s * dvs * (1 + gr * GAM * pp / rh)
                wn = w1 - f / df
                live = live & (wn > 0)
                done = live & ((wn - w1).abs() < 1e-10 * wn)
                w1 = torch.where(live, wn, w1)
                good, live = good | done, live & ~done
            bw = b2 + w1
            vs = ((qt2 * w1 ** 2 + qb2 * (b2 + 2 * w1)) / (w1 * bw) ** 2).clamp(max=vmax)
            rh = d * (1 - vs).sqrt()
            ue = kap * rh ** GAM / (GAM - 1)
            good = good & (rh > 0) & (ue > 0) & (vs >= 0)
            w[at], v[at], rho[at], u[at] = w1, vs, rh, ue
            keep[at] = ~good
        pre = 1 / (1 - v).sqrt() / (w + B2)
        Qt = [Qc[1] - al * g["c01"] * Qn, Qc[2], Qc[3]]
        new = [rho, u] + [pre * (Qt[k] + QB * Bn[k] / w) for k in range(3)]
        for k in range(5):
            pr[k] = torch.where(keep, pr[k], new[k])
        for k in range(3):
            pr[5 + k] = Bc[k]
        pr = pr.reshape(shape)
        b2 = _state(pr, self.cut(self.gc))[4]
        pr[0] = torch.maximum(pr[0], torch.maximum(self.cut(self.rhoflr.expand(1, self.n[1] + 2 * NG, -1)), b2 / 50))
        pr[1] = torch.maximum(pr[1], torch.maximum(self.cut(self.uflr.expand(1, self.n[1] + 2 * NG, -1)), b2 / 750))
        return pr

    def rate(self, P):
        Pi, g = self.cut(P), self.cut(self.gc)
        st = _state(Pi, g)
        tot = 0
        for d in (1, 2, 3):
            A, B, sd = _quad(Pi, st, g, d)
            tot = tot + (B.abs() + sd) / A.abs() / self.dx[d - 1]
        return float(tot.max())

    def advance(self, P, B, steps):
        i, j, k = (slice(NG, NG + n) for n in self.n)
        P = P.clone()
        for q, x in enumerate(self.centre(B)):
            P[5 + q, k, j, i] = x
        self.bc(P, B)
        for _ in range(steps):
            dt = COUR / self.rate(P)
            Pi, g = self.cut(P), self.cut(self.gc)
            Un = _cons(Pi, _state(Pi, g), g, _kappa(Pi))
            Ph, Bh = self.stage(P, B, Un, B, 0.5 * dt)
            P, B = self.stage(Ph, Bh, Un, B, dt)
        return P, B
