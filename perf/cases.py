"""Performance cases: what programs built on this library have it do.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes what a program holds before the call (device
arrays, a tree or a network), ``run(state)`` is one pass through the public
entry points, ``work(case)`` the bytes and operations such a pass cannot do
without, and ``exact(case, seed)`` its result in plain float64 torch (direct
sums instead of the treecode, no code of this library).

The kinds of case:
  conv      one convolution call on a tree that the program keeps;
  step      tree build and one Green step, the unit the benchmark times: what
            a program pays on a new mesh;
  iterate   a few Green iterations of one molecule with eigenpair mixing;
  scf       one SCF iteration on a tree that the program keeps;
  direct    the allocation-free direct sum;
  train     one full-batch training step of the warm-start network;
  gradient  its loss and gradient alone;
  warm      features and warm-started orbital of one mesh.
"""
import functools
import math

import numpy as np
import torch

from paper_2003_01833_gb300 import tagi as T
from paper_2003_01833_gb300 import workloads as W

DEV = "cuda"
EXACT_PAIRS = 6e10  # direct-sum pairs times fields that exact() spends at most (under 20 s)
KT = 6.3336e-4      # 200 K in Ha


def listed():
    return [
        # the smallest tree calls: ragged random points, one Hartree field.
        # Launches, allocations and host work are most of it
        {"name": "cube-coulomb", "kind": "conv", "mesh": "cube", "points": 5003, "yukawa": 0, "hartree": True,
         "leaf": 300, "degree": 6, "theta": 0.7, "prec": "fp32c", "ss": True},
        # one orbital on the small uniform hydrogen mesh (32,768 points), the smoke test's call
        {"name": "hydrogen-yukawa", "kind": "conv", "mesh": "hydrogen", "cells": 8, "yukawa": 1, "hartree": False,
         "leaf": 2000, "degree": 6, "theta": 0.7, "prec": "fp32c", "ss": True},
        # the same in the plain float64 form, for programs that need it exact next to a nucleus
        {"name": "hydrogen-yukawa-fp64", "kind": "conv", "mesh": "hydrogen", "cells": 8, "yukawa": 1,
         "hartree": False, "leaf": 2000, "degree": 6, "theta": 0.7, "prec": "fp64", "ss": True},
        # allocation-free float64 direct sum inside another framework's loop
        {"name": "direct-noalloc", "kind": "direct", "points": 12007, "yukawa": 2},
        # Li atom on the coarse mesh (99,000 points): tree build and Green step of two orbitals with Hartree
        {"name": "li-small-step", "kind": "step", "mesh": "li", "tol": 1e-3, "leaf": 2000, "degree": 8,
         "theta": 0.7, "prec": "fp32c"},
        # the benchmark step: Li, 309,000 points
        {"name": "li-step", "kind": "step", "mesh": "li", "tol": 3e-7, "leaf": 2000, "degree": 8, "theta": 0.7,
         "prec": "fp32c"},
        # Green Iteration of the H2 orbital (192,000 points), three mixed steps
        {"name": "h2-iterate", "kind": "iterate", "mesh": "h2", "tol": 3e-6, "steps": 3, "leaf": 2000, "degree": 8,
         "theta": 0.7},
        # one SCF iteration of Li on the coarse mesh with two Green iterations inside
        {"name": "li-small-scf", "kind": "scf", "mesh": "li", "tol": 1e-3, "steps": 2, "leaf": 2000, "degree": 8,
         "theta": 0.7},
        # CO (638,500 points): seven orbitals and the Hartree field in one pass, the largest call
        {"name": "co-fields", "kind": "conv", "mesh": "co", "tol": 3e-7, "yukawa": 7, "hartree": True, "leaf": 2000,
         "degree": 8, "theta": 0.7, "prec": "fp32c", "ss": True},
        # full-batch training step of the 64-unit network on the H2 training set (10.9M points)
        {"name": "mlp64-train", "kind": "train", "points": 10900000, "hidden": 64},
        # loss and gradient of the 32-unit network on one mesh
        {"name": "mlp32-gradient", "kind": "gradient", "points": 192000, "hidden": 32},
        # features and warm-started orbital of one H2 mesh, before its SCF run
        {"name": "mlp64-warm", "kind": "warm", "points": 192000, "hidden": 64},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "conv", "step", "step", "iterate", "scf", "direct", "train",
                       "gradient", "warm"])
    tree = {"leaf": int(_log(rng, 400, 4000)), "degree": rng.choice([5, 6, 6, 7, 8, 8, 8]),
            "theta": round(rng.uniform(0.55, 0.8), 3)}
    if kind == "conv":
        c = {"kind": kind, "prec": rng.choice(["fp32c", "fp32c", "fp32c", "fp64"]), "ss": rng.random() < 0.85, **tree}
        c["mesh"] = rng.choice(["cube", "hydrogen", "li", "h2"] if c["prec"] == "fp32c" else ["cube", "hydrogen"])
        c["yukawa"] = rng.choice([0, 1, 1, 2, 3, 5, 8, 10]) if c["prec"] == "fp32c" else 1
        c["hartree"] = c["yukawa"] == 0 or rng.random() < 0.5
        if c["prec"] == "fp64":
            c["hartree"] = False
        if c["mesh"] == "cube":
            c["points"] = int(_log(rng, 1000, 120000 if c["prec"] == "fp32c" else 25000))
            c["leaf"] = max(50, min(c["leaf"], c["points"] // 8))
        elif c["mesh"] == "hydrogen":
            c["cells"] = rng.randint(4, 12 if c["prec"] == "fp32c" else 8)
        else:
            c["tol"] = _log(rng, 3e-6, 1e-2)
        return c
    if kind == "step":
        return {"kind": kind, "mesh": "li", "tol": _log(rng, 3e-7, 1e-2), "prec": "fp32c", **tree}
    if kind == "iterate":
        return {"kind": kind, "mesh": "h2", "tol": _log(rng, 3e-6, 1e-3), "steps": rng.randint(1, 4), **tree}
    if kind == "scf":
        return {"kind": kind, "mesh": "li", "tol": _log(rng, 1e-5, 1e-2), "steps": rng.randint(1, 3), **tree,
                "degree": 8}
    if kind == "direct":
        return {"kind": kind, "points": int(_log(rng, 500, 30000)), "yukawa": rng.randint(1, 3)}
    if kind == "train":
        return {"kind": kind, "points": int(_log(rng, 20000, 10900000)), "hidden": rng.choice([64, 64, 32])}
    return {"kind": kind, "points": int(_log(rng, 1000, 2000000)), "hidden": rng.choice([64, 32])}


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=4)
def _mesh_workload(mesh, size):
    if mesh == "hydrogen":
        return W.hydrogen_1s(seed=0, ncell=size)
    if mesh == "li":
        return W.lithium(seed=1, tol_m=size)
    if mesh == "h2":
        return W.hydrogen_molecule(1.4, tol_m=size)
    return W.carbon_monoxide_scf(tol_m=size)


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _smooth(rng, xyz, amp):
    a = rng.normal(size=3)
    a *= 0.5 / np.linalg.norm(a)
    return 1.0 + amp * np.sin(a @ xyz + rng.uniform(0, 2 * np.pi))


def _atoms(case, seed):
    """Mesh, potential, orbitals with a seeded smooth perturbation, density (host arrays)."""
    wl = _mesh_workload(case["mesh"], case.get("cells") or case["tol"])
    rng = np.random.default_rng(seed)
    xyz = wl.mesh.xyz
    psi = np.stack([p * _smooth(rng, xyz, 0.01) for p in wl.psi])
    eps = wl.eps + rng.uniform(-0.01, 0.01, size=wl.eps.size)
    return wl, xyz, wl.mesh.w, psi, eps, wl.rho * _smooth(rng, xyz, 0.01)


def _fields(case, seed):
    """Mesh, Yukawa sources f with decay rates k, Hartree source (host arrays)."""
    ny = case["yukawa"]
    rng = np.random.default_rng(seed)
    if case.get("mesh", "cube") == "cube":
        xyz, w = W.random_cube(case["points"], seed=seed)
        f = [1.0 + 0.3 * np.sin(3 * xyz[0] + o + rng.uniform()) * np.cos(2 * xyz[1]) for o in range(ny)]
        k = rng.uniform(0.7, 4.0, size=ny)
        rho = np.exp(-np.sum(xyz * xyz, axis=0)) * _smooth(rng, xyz, 0.1)
    else:
        wl, xyz, w, psi, eps, rho = _atoms(case, seed)
        v = wl.veff + wl.vshift
        f = [v * psi[o % len(psi)] * (1.0 if o < len(psi) else _smooth(rng, xyz, 0.2)) for o in range(ny)]
        k = [math.sqrt(-2.0 * (eps[o % len(eps)] + wl.vshift)) for o in range(ny)]
    return xyz, w, (np.stack(f) if ny else None), list(k), rho if case.get("hartree") else None


@functools.lru_cache(maxsize=1)
def _h2_points():
    m = W.hydrogen_molecule(1.4).mesh
    return _t(m.xyz), _t(m.w)


def _geometries(case, seed):
    """Points of as many H2 geometries as the case's size takes: the mesh of
    bond length 1.4 scaled to seeded bond lengths.  Yields (R, xyz, w)."""
    xyz, w = _h2_points()
    left = case["points"]
    for R in np.random.default_rng(seed).uniform(1.0, 2.0, size=-(-left // w.numel())):
        m = min(left, w.numel())
        g = float(R) / 1.4
        yield float(R), (xyz[:, :m] * g).contiguous(), w[:m] * g ** 3
        left -= m


def _superposition(R, xyz, w):
    """Normalised superposition of the two 1s functions, and a correction as a converged orbital has it."""
    r = [torch.sqrt((xyz[0] - s * 0.5 * R) ** 2 + xyz[1] ** 2 + xyz[2] ** 2) for s in (-1.0, 1.0)]
    s = torch.exp(-r[0]) + torch.exp(-r[1])
    s = s / torch.sqrt(torch.sum(s * s * w))
    return s, 0.2 * torch.exp(-r[0] * r[1]) - 0.1 * torch.tanh(0.3 * (r[0] + r[1]) - R)


def _nuclei(R):
    return [[-0.5 * R, 0.0, 0.0], [0.5 * R, 0.0, 0.0]]


def _network(case, seed):
    return W.mlp_init(seed=seed, hidden=case["hidden"])


def _prec(case):
    return T.TAGI_FP64 if case.get("prec") == "fp64" else T.TAGI_FP32C


def _tree(case, xyz, w):
    return T.Tree(xyz, w, theta=case["theta"], degree=case["degree"], leaf_size=case["leaf"], prec=_prec(case),
                  ss=case.get("ss", True))


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind in ("conv", "direct"):
        xyz, w, f, k, rho = _fields(case, seed)
        st.update(xyz=_t(xyz), w=_t(w), f=None if f is None else _t(f), k=k, rho=None if rho is None else _t(rho))
        st["u"] = None if f is None else torch.empty_like(st["f"])
        st["vh"] = None if rho is None else torch.empty_like(st["rho"])
        if kind == "conv":
            st["tree"] = _tree(case, st["xyz"], st["w"])
    elif kind in ("step", "iterate", "scf"):
        wl, xyz, w, psi, eps, rho = _atoms(case, seed)
        st.update(xyz=_t(xyz), w=_t(w), psi0=_t(psi), eps=eps, rho0=_t(rho), vshift=wl.vshift, veff=_t(wl.veff),
                  vext=_t(wl.vext), n_elec=wl.n_elec)
        st["psi"], st["rho"] = torch.empty_like(st["psi0"]), torch.empty_like(st["rho0"])
        st["vh"], st["rho_out"] = torch.empty_like(st["rho0"]), torch.empty_like(st["rho0"])
        if kind != "step":
            st["tree"] = _tree(case, st["xyz"], st["w"])
    else:
        st["net"] = T.Mlp(_network(case, seed), hidden=case["hidden"])
        if kind == "warm":
            (R, xyz, w), = list(_geometries({"points": min(case["points"], 192000)}, seed))
            reps = -(-case["points"] // w.numel())  # a finer mesh: the same points shrunk a little each time
            xyz = torch.cat([xyz * (1.0 - 0.01 * q / reps) for q in range(reps)], dim=1)[:, :case["points"]]
            st.update(R=R, xyz=xyz.contiguous(), w=w.repeat(reps)[:case["points"]].contiguous())
            st["s"] = _superposition(R, st["xyz"], st["w"])[0].contiguous()
        else:
            feat, target, wt = [], [], []
            for R, xyz, w in _geometries(case, seed):
                s, t = _superposition(R, xyz, w)
                feat.append(T.tagi_mlp_features(xyz, _nuclei(R)))
                target.append(t.float())
                wt.append((w * s * s).float())
            st.update(feat=torch.cat(feat), target=torch.cat(target), wt=torch.cat(wt))
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "conv":
        h = st["tree"].handle
        if st["rho"] is None:
            T.tagi_yukawa_conv(h, st["f"], st["k"], st["u"])
        elif st["f"] is None:
            T.tagi_coulomb_conv(h, st["rho"], st["vh"])
        else:
            T.tagi_fields_conv(h, st["f"], st["k"], st["u"], rho=st["rho"], vh=st["vh"])
        return [t for t in (st["u"], st["vh"]) if t is not None]
    if kind == "direct":
        T.tagi_yukawa_direct_noalloc(st["xyz"], st["w"], st["f"], st["k"], st["u"])
        return [st["u"]]
    if kind == "step":
        st["psi"].copy_(st["psi0"])
        with _tree(case, st["xyz"], st["w"]) as tree:
            eps, resid, eh = T.tagi_green_step(tree.handle, st["veff"], st["vshift"], st["psi"], st["eps"],
                                               rho=st["rho0"], vh=st["vh"])
        return [st["psi"], st["vh"], eps, resid, eh]
    if kind == "iterate":
        st["psi"].copy_(st["psi0"])
        r = T.tagi_green_iterate(st["tree"].handle, st["veff"], st["vshift"], st["psi"], st["eps"], 0.0,
                                 case["steps"])
        return [st["psi"], r["eps"], r["resid"]]
    if kind == "scf":
        st["psi"].copy_(st["psi0"])
        st["rho"].copy_(st["rho0"])
        with T.Scf(st["tree"].handle, st["n_elec"], kT=KT, tol_gi_first=1e-12, gi_max_iter=case["steps"]) as scf:
            r = scf.step(st["vext"], st["vshift"], st["rho"], st["psi"], st["eps"], rho_out=st["rho_out"])
        return [st["psi"], st["rho"], st["rho_out"], r["eps"], r["residual"], r["e_total"]]
    net = st["net"]
    if kind == "train":
        loss = net.train_step(st["feat"], st["target"], st["wt"], 3e-3, want_loss=True)
        return [loss, net.params()]
    if kind == "gradient":
        loss, grad = net.gradient(st["feat"], st["target"], st["wt"])
        return [loss, grad]
    feat = T.tagi_mlp_features(st["xyz"], _nuclei(st["R"]))
    return [feat, net.warm_start(feat, st["s"], st["w"])]


# ------------------------------------------------------------------ work
def work(case):
    """Interactions are the treecode's own (near sources and proxies of the
    lists at the case's theta, degree and leaf size): 8 operations of geometry
    a pair and 8 a field and pair.  The network: 2 a weight and point forward,
    6 with the gradient, 10 a tanh."""
    kind = case["kind"]
    if kind in ("conv", "step", "iterate", "scf"):
        if case["mesh"] == "cube":
            xyz, w = W.random_cube(case["points"], seed=0)
            nw = 0
        else:
            wl = _mesh_workload(case["mesh"], case.get("cells") or case["tol"])
            xyz, w, nw = wl.mesh.xyz, wl.mesh.w, len(wl.psi)
        with _tree(case, _t(xyz), _t(w)) as tree:
            info = tree.info()
        n, pairs = info["n_points"], info["near_pairs"] + info["far_pairs"]
        if kind == "conv":
            nf = case["yukawa"] + bool(case["hartree"])
            return {"bytes": 8 * n * 2 * nf, "flops": pairs * (8 + 8 * nf)}
        if kind == "step":  # points, potential, orbitals and density in; orbitals and potential out
            return {"bytes": 8 * n * (4 + 1 + 2 * nw + 2), "flops": pairs * (8 + 8 * (nw + 1))}
        flops = case["steps"] * pairs * (8 + 8 * nw)
        if kind == "scf":
            return {"bytes": 8 * n * (2 * nw + 4), "flops": flops + pairs * 16}
        return {"bytes": 8 * n * (2 * nw + 1), "flops": flops}
    n = case["points"]
    if kind == "direct":
        return {"bytes": 8 * n * (4 + 2 * case["yukawa"]), "flops": n * n * case["yukawa"] * 16}
    H = case["hidden"]
    weights = 8 * H + H * H + H
    if kind == "warm":
        return {"bytes": n * (24 + 16 + 16 + 8), "flops": n * (2 * weights + 20 * H + 60)}
    return {"bytes": n * 24, "flops": n * (6 * weights + 20 * H)}


# ------------------------------------------------------------------ exact
def _direct(xyz, w, f, k, rho, ss, alpha=1.0):
    """Direct sums with the singularity subtraction, float64, in blocks of targets."""
    n = w.numel()
    ny = 0 if f is None else f.shape[0]
    u = torch.empty((ny, n), dtype=torch.float64, device=DEV)
    vh = None if rho is None else torch.empty(n, dtype=torch.float64, device=DEV)
    step = max(1, int(2e8) // n)
    for i in range(0, n, step):
        j = slice(i, min(n, i + step))
        r2 = sum((xyz[d][j, None] - xyz[d][None, :]) ** 2 for d in range(3))
        r = torch.sqrt(r2)
        g = torch.where(r2 > 0, w[None, :] / r, 0.0)  # w_j / r, the pair r = 0 left out
        for o in range(ny):
            e = torch.exp(-k[o] * r) * g
            s = e @ f[o]
            if ss:
                s = ((f[o][None, :] - f[o][j, None]) * e).sum(dim=1)
            u[o][j] = s / (4 * math.pi) + (f[o][j] / k[o] ** 2 if ss else 0.0)
        if rho is not None:
            s = g @ rho
            if ss:
                s = s - rho[j] * (torch.exp(-r2 / alpha ** 2) * g).sum(dim=1) + 2 * math.pi * alpha ** 2 * rho[j]
            vh[j] = s
    return u, vh


def _green(xyz, w, veff, vshift, psi, eps, rho=None):
    """One Green step: new orbitals, eigenvalues, residuals, Hartree potential."""
    f = (veff + vshift)[None, :] * psi
    k = [math.sqrt(-2.0 * (float(e) + vshift)) for e in eps]
    u, vh = _direct(xyz, w, f, k, rho, True)
    new, out = [], []
    for o in range(len(psi)):
        v = -2.0 * u[o]
        out.append(float(eps[o]) - float((f[o] * (psi[o] - v) * w).sum() / (v * v * w).sum()))
        for q in new:
            v = v - (v * q * w).sum() * q
        new.append(v / torch.sqrt((v * v * w).sum()))
    new = torch.stack(new)
    resid = torch.sqrt(((new - psi) ** 2 * w).sum(dim=1)).cpu().numpy()
    return new, np.array(out), resid, vh


def _anderson(hist, dot, beta):
    """Next iterate from pairs (x, F), newest last."""
    x, F = hist[-1]
    d = [F - g for _, g in hist[:-1]]
    th = np.zeros(0)
    if d:
        th = np.linalg.solve([[dot(a, b) for b in d] for a in d], [dot(a, F) for a in d])
    nx, nF = x, F
    for t, (y, g) in zip(th, hist[:-1]):
        nx = nx - t * (x - y)
        nF = nF - t * (F - g)
    return nx + beta * nF


def _iterate(xyz, w, veff, vshift, psi, eps, steps, beta=0.5):
    n = w.numel()
    wt = torch.cat([w, torch.ones(1, dtype=torch.float64, device=DEV)])  # the eigenvalue is the last component

    def dot(a, b):
        return float((a * b * wt).sum())

    hist = [[] for _ in psi]
    for _ in range(steps):
        new, e, resid, _ = _green(xyz, w, veff, vshift, psi, eps)
        nxt = []
        for o in range(len(psi)):
            x = torch.cat([psi[o], _t([eps[o]])])
            hist[o].append((x, torch.cat([new[o], _t([e[o]])]) - x))
            nxt.append(_anderson(hist[o], dot, beta))
        psi = torch.stack([v[:n] for v in nxt])
        eps = np.array([float(v[n]) for v in nxt])
    return psi, eps, resid


def _scf(st, steps):
    xyz, w, rho = st["xyz"], st["w"], st["rho0"]
    vh = _direct(xyz, w, None, [], rho, True)[1]
    exc, vxc = (_t(a) for a in _lda(rho.cpu().numpy()))
    veff = st["vext"] + vh + vxc
    psi, eps, _ = _iterate(xyz, w, veff, st["vshift"], st["psi0"], st["eps"], steps)
    psi = psi / torch.sqrt((psi * psi * w).sum(dim=1))[:, None]
    lo, hi = eps.min() - 60 * KT, eps.max() + 60 * KT
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        occ = 1.0 / (1.0 + np.exp((eps - mu) / KT))
        lo, hi = (mu, hi) if 2 * occ.sum() < st["n_elec"] else (lo, mu)
    out = 2.0 * (_t(occ)[:, None] * psi * psi).sum(dim=0)
    resid = float(torch.sqrt(((out - rho) ** 2 * w).sum()))
    e = 2.0 * float((occ * eps).sum()) + float(((exc - vxc - 0.5 * vh) * rho * w).sum())
    return [psi, rho + 0.5 * (out - rho), out, eps, resid, e]


def _lda(rho):
    """Slater exchange and Perdew-Zunger correlation: energy per electron and potential."""
    r = np.maximum(rho, 1e-30)
    x = np.cbrt(3 * r / np.pi)
    rs = np.cbrt(3 / (4 * np.pi * r))
    q, ln = np.sqrt(rs), np.log(rs)
    den = 1 + 1.0529 * q + 0.3334 * rs
    e1 = -0.1423 / den
    v1 = e1 * (1 + 7 / 6 * 1.0529 * q + 4 / 3 * 0.3334 * rs) / den
    e2 = 0.0311 * ln - 0.048 + 0.002 * rs * ln - 0.0116 * rs
    v2 = 0.0311 * ln - (0.048 + 0.0311 / 3) + 0.004 / 3 * rs * ln - (0.0232 + 0.002) / 3 * rs
    live = rho > 1e-30
    return (np.where(live, -0.75 * x + np.where(rs >= 1, e1, e2), 0.0),
            np.where(live, -x + np.where(rs >= 1, v1, v2), 0.0))


def _features64(R, xyz):
    a, b = (torch.sqrt((xyz[0] - s * 0.5 * R) ** 2 + xyz[1] ** 2 + xyz[2] ** 2) for s in (-1.0, 1.0))
    r1, r2 = torch.minimum(a, b), torch.maximum(a, b)
    f = [torch.exp(-r1), torch.exp(-r2), torch.tanh(r1), torch.tanh(r2), (r2 - r1) / R,
         torch.tanh((r1 + r2) / R - 1.0), torch.full_like(r1, R - 1.5), torch.exp(-(r1 + r2 - R))]
    return torch.stack(f, dim=1).bfloat16().double()  # the inputs are bfloat16


def _network64(case, seed):
    """Weights as the products take them (bfloat16), biases, all as float64 leaves."""
    p, H, at = _t(_network(case, seed)), case["hidden"], 0
    parts = []
    for shape in ((H, 8), (H,), (H, H), (H,), (H,), (1,)):
        m = int(np.prod(shape))
        parts.append(p[at:at + m].reshape(shape))
        at += m
    return [(q.bfloat16().double() if i in (0, 2, 4) else q).requires_grad_() for i, q in enumerate(parts)]


def _forward64(net, x):
    h1 = torch.tanh(x @ net[0].T + net[1])
    h2 = torch.tanh(h1 @ net[2].T + net[3])
    return h2 @ net[4] + net[5]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("conv", "direct"):
        xyz, w, f, k, rho = _fields(case, seed)
        nf = case["yukawa"] + (rho is not None)
        if w.size ** 2 * float(nf) > EXACT_PAIRS:
            return None
        u, vh = _direct(_t(xyz), _t(w), None if f is None else _t(f), k, None if rho is None else _t(rho),
                        case.get("ss", True))
        return [t for t in (u if len(u) else None, vh) if t is not None]
    if kind in ("step", "iterate", "scf"):
        wl, xyz, w, psi, eps, rho = _atoms(case, seed)
        nf = len(psi) + 1 if kind == "step" else len(psi) * case["steps"] + (kind == "scf")
        if w.size ** 2 * float(nf) > EXACT_PAIRS:
            return None
        xyz, w, psi, rho, veff = _t(xyz), _t(w), _t(psi), _t(rho), _t(wl.veff)
        if kind == "step":
            new, e, resid, vh = _green(xyz, w, veff, wl.vshift, psi, eps, rho)
            return [new, vh, e, resid, 0.5 * float((vh * rho * w).sum())]
        if kind == "iterate":
            return list(_iterate(xyz, w, veff, wl.vshift, psi, eps, case["steps"]))
        return _scf({"xyz": xyz, "w": w, "rho0": rho, "psi0": psi, "eps": eps, "vext": _t(wl.vext),
                     "vshift": wl.vshift, "n_elec": wl.n_elec}, case["steps"])
    net = _network64(case, seed)
    if kind == "warm":
        st = prepare(case, seed)
        with torch.no_grad():
            psi = st["s"] * (1.0 + _forward64(net, _features64(st["R"], st["xyz"])))
            return [None, psi / torch.sqrt((psi * psi * st["w"]).sum())]
    loss = 0.0
    for R, xyz, w in _geometries(case, seed):
        s, t = _superposition(R, xyz, w)
        wt = (w * s * s).float().double()
        part = (wt * (_forward64(net, _features64(R, xyz)) - t.float().double()) ** 2).sum()
        part.backward()
        loss += float(part)
    grad = torch.cat([q.grad.reshape(-1) for q in net])
    if kind == "gradient":
        return [loss, grad]
    return [loss, _t(_network(case, seed)) - 3e-3 * grad / (grad.abs() + 1e-8)]
