"""The cases by which this framework's speed is measured.

Each case is work that a user of the library has it do through its Python entry points:
the one-call step of a design iteration (K(rho), dc and c) on every kind of mesh, the
backward of the compliance, the constrained solve of the optimisation loop, and the
grouped step of many small designs.  Sizes are those of the benchmark (bench.py), its
serving stream and the paper's cantilever; ``draw`` spreads over the same ranges with
other cells, orders and odd sizes.  ``exact`` evaluates the same definitions by plain
Gauss quadrature in 64 bits with torch and numpy alone.
"""
import itertools
import math
import random

import numpy as np
import torch

import paper_2505_02438_gb300 as soptx
from paper_2505_02438_gb300.autograd import Compliance

E0, EMIN, NU, P = 1.0, 1e-9, 0.3, 3.0          # the paper's material; plane stress in 2D
DIM = {"tri": 2, "quad": 2, "tet": 3, "hex": 3}
JITTER = {"tri": 0.2, "quad": 0.2, "tet": 0.15, "hex": 0.15}   # of the grid spacing, as in workloads.py
RTOL, MAX_ITER, CHECK = 1e-12, 200000, 50      # CG: the loop's settings, to the tolerance of the solve tests


def _case(name, op, cell, order, n, jitter=False, prec="fp64", count=1):
    return {"name": name, "op": op, "cell": cell, "order": order, "nx": n[0], "ny": n[1],
            "nz": n[2] if len(n) > 2 else 0, "jitter": jitter, "prec": prec, "count": count}


def listed():
    return [
        # the paper's MBB beam: the smallest design in use, one step is launches and latency
        _case("step quad q1 60x20", "step", "quad", 1, (60, 20)),
        # the benchmark's default: a structured 3D design, every design iteration's step
        _case("step hex q1 120x40x40", "step", "hex", 1, (120, 40, 40)),
        # unstructured triangles of high order, in both precisions of the element matrices
        _case("step tri p3 400x200", "step", "tri", 3, (400, 200), True),
        _case("step tri p3 400x200 fp32", "step", "tri", 3, (400, 200), True, "fp32"),
        # unstructured tetrahedra, the usual mesh of a 3D part, in both precisions
        _case("step tet p2 60x20x20", "step", "tet", 2, (60, 20, 20), True),
        _case("step tet p2 60x20x20 fp32", "step", "tet", 2, (60, 20, 20), True, "fp32"),
        # distorted hexahedra (a mapped mesh of a curved part)
        _case("step hex q1 120x40x40 distorted", "step", "hex", 1, (120, 40, 40), True),
        # a structured box with quadratic elements
        _case("step hex q2 40x14x14", "step", "hex", 2, (40, 14, 14)),
        # the compliance in a differentiable program: forward and both gradients
        _case("backward hex q1 120x40x40", "backward", "hex", 1, (120, 40, 40)),
        _case("backward tet p2 60x20x20", "backward", "tet", 2, (60, 20, 20), True),
        # the equilibrium solve of the paper's 3D cantilever, most of an optimisation loop's time
        _case("solve hex q1 60x20x4", "solve", "hex", 1, (60, 20, 4)),
        # many small designs served together in one call (16 to 64 cells a side)
        _case("group of 16 quads q1", "group", "quad", 1, (64, 64), count=16),
    ]


# nonzeros a cell of a large mesh adds to K, to aim a drawn mesh at a size
_PER_CELL = {("tri", 1): 14, ("tri", 2): 92, ("tri", 3): 306, ("quad", 1): 36, ("quad", 2): 256, ("quad", 3): 900,
             ("tet", 1): 23, ("tet", 2): 353, ("tet", 3): 1900, ("hex", 1): 243, ("hex", 2): 4608, ("hex", 3): 29600}
_SPLIT = {"tri": 2, "quad": 1, "tet": 6, "hex": 1}


def draw(rng):
    op = rng.choice(["step"] * 7 + ["backward"] * 2 + ["solve", "group"])
    if op == "group":
        side = rng.randint(20, 64)
        return _drawn("group", "quad", 1, (side, rng.randint(16, 64)), False, "fp64", rng.randint(2, 16))
    if op == "solve":
        nz = rng.randint(1, 6)
        ny = rng.randint(5, 24)
        return _drawn("solve", "hex", 1, (rng.randint(10, max(11, min(80, 6000 // ((ny + 1) * (nz + 1))))), ny, nz),
                      False, "fp64", 1)
    cell = rng.choice(["tri", "quad", "tet", "hex", "hex"])
    order = rng.randint(1, 3)
    cells = math.exp(rng.uniform(math.log(4e4), math.log(4.5e7))) / (_PER_CELL[cell, order] * _SPLIT[cell])
    d = DIM[cell]
    side = max(cells, 1.0) ** (1.0 / d)
    skew = [math.exp(rng.uniform(-0.6, 0.6)) for _ in range(d - 1)]
    n = [max(1, round(side * s)) for s in skew]
    n.append(max(1, round(cells / math.prod(n))))
    return _drawn(op, cell, order, n[::-1], cell in ("tri", "tet") or rng.random() < 0.5,
                  rng.choice(["fp64", "fp64", "fp32"]), 1)


def _drawn(*a):
    c = _case("", *a)
    del c["name"]
    return c


def _group_sizes(case):
    """The box of each small design: sides log-uniform from 16 to the case's."""
    g = random.Random(case["count"])
    side = lambda top: round(16 * (max(top, 16) / 16) ** g.random())
    return [(side(case["nx"]), side(case["ny"])) for _ in range(case["count"])]


# ------------------------------------------------------------------ meshes and inputs

def _grid(cell, n, amount, g):
    """Vertices (x fastest) and cells of a unit-spaced grid, simplices split along the
    main diagonal; interior vertices moved by U(-amount, amount) per coordinate."""
    d = len(n)
    dims = [k + 1 for k in n]
    lat = np.stack([x.ravel() for x in np.meshgrid(*[np.arange(k) for k in dims[::-1]], indexing="ij")][::-1], 1)
    stride = np.cumprod([1] + dims[:-1])
    x = lat.astype(np.float64)
    if amount:
        inner = np.all((lat > 0) & (lat < np.array(n)), axis=1)
        x = x + inner[:, None] * g.uniform(-amount, amount, x.shape)
    org = np.stack([c.ravel() for c in np.meshgrid(*[np.arange(k) for k in n[::-1]], indexing="ij")][::-1], 1)
    first = org @ stride
    if cell in ("quad", "hex"):
        corner = [sum(((v >> m) & 1) * stride[m] for m in range(d)) for v in range(1 << d)]
        cells = first[:, None] + np.array(corner)[None]
    elif cell == "tri":
        s0, s1 = stride
        cells = (first[:, None, None] + np.array([[0, s0, s0 + s1], [0, s0 + s1, s1]])[None]).reshape(-1, 3)
    else:
        paths = [np.cumsum([0] + [stride[a] for a in p]) for p in itertools.permutations(range(3))]
        cells = (first[:, None, None] + np.array(paths)[None]).reshape(-1, 4)
    return x, np.ascontiguousarray(cells, dtype=np.int32)


def _inputs(case, seed):
    """Host coordinates, cells, density and displacement (and, for the solve, the clamped
    dofs and the load) of each mesh of the case."""
    out = []
    sizes = _group_sizes(case) if case["op"] == "group" else [tuple(case[k] for k in ("nx", "ny", "nz") if case[k])]
    for k, n in enumerate(sizes):
        g = np.random.default_rng([seed, k])
        cell, d = case["cell"], DIM[case["cell"]]
        x, cells = _grid(cell, n, JITTER[cell] if case["jitter"] else 0.0, g)
        nodes = _counts(cell, case["order"], n)[0]
        s = {"x": x, "cells": cells}
        if case["op"] == "solve":
            # an early design of the loop: volume fraction 0.3, clamped at x = 0, loaded at the far lower edge
            s["rho"] = np.clip(0.3 + g.uniform(-0.1, 0.1, len(cells)), 0.001, 1.0)
            s["fixed"] = np.repeat(x[:, 0] < 1e-9, d)
            s["f"] = np.zeros(d * len(x))
            s["f"][d * np.nonzero((x[:, 0] > n[0] - 1e-9) & (x[:, 1] < 1e-9))[0] + 1] = -1.0
            s["f"] *= 1.0 + 0.1 * g.uniform(-1, 1)
        else:
            s["rho"] = np.clip(0.5 + g.uniform(-0.1, 0.1, len(cells)), 0.001, 1.0) if (cell, case["order"]) == \
                ("quad", 1) else g.uniform(0.001, 1.0, len(cells))
            s["u"] = g.standard_normal(d * nodes)
        out.append(s)
    return out


def prepare(case, seed):
    state = {"op": case["op"], "m": []}
    for s in _inputs(case, seed):
        mesh = soptx.Mesh(case["cell"], case["order"], s["x"], s["cells"], E0, EMIN, NU, P, elem_prec=case["prec"])
        m = {"mesh": mesh}
        for k in ("rho", "u", "f"):
            if k in s:
                m[k] = torch.as_tensor(s[k], device="cuda")
        if case["op"] == "solve":
            m["fixed"] = torch.as_tensor(s["fixed"], device="cuda").to(torch.uint8)
            m["vals"] = mesh.assemble_K(m["rho"])
        if case["op"] == "backward":
            m["rho"].requires_grad_(True)
            m["u"].requires_grad_(True)
        state["m"].append(m)
    return state


def run(state):
    op, m = state["op"], state["m"][0]
    if op == "step":
        vals, dc, c = m["mesh"].step(m["rho"], m["u"])
        return {"vals": vals, "dc": dc, "c": c}
    if op == "backward":
        c = Compliance.apply(m["rho"], m["u"], m["mesh"])
        g_rho, g_u = torch.autograd.grad(c, (m["rho"], m["u"]))
        return {"c": c.detach(), "g_rho": g_rho, "g_u": g_u}
    if op == "solve":
        u, _ = m["mesh"].solve(m["vals"], m["fixed"], m["f"], rtol=RTOL, max_iter=MAX_ITER, check_every=CHECK)
        return {"u": u}
    outs = soptx.step_group([k["mesh"] for k in state["m"]], [k["rho"] for k in state["m"]],
                            [k["u"] for k in state["m"]])
    return {"vals": [o[0] for o in outs], "dc": [o[1] for o in outs], "c": [o[2] for o in outs]}


# ------------------------------------------------------------------ what a pass cannot do without

def _counts(cell, k, n):
    """(nodes, node pairs that share a cell, cells, vertices) of a grid with elements of order k."""
    pl = [q + 1 for q in n]
    v = math.prod(pl)
    box = math.prod(n)
    axis = sum(n[m] * math.prod(pl[:m] + pl[m + 1:]) for m in range(len(n)))
    if cell in ("quad", "tri"):
        ents = [v, axis + (box if cell == "tri" else 0), box * (2 if cell == "tri" else 1)]
    else:
        squares = sum(pl[m] * math.prod(n[:m] + n[m + 1:]) for m in range(3))
        if cell == "hex":
            ents = [v, axis, squares, box]
        else:
            e = axis + squares + box
            ents = [v, e, 1 - v + e + 6 * box, 6 * box]
    d = DIM[cell]
    if cell in ("tri", "tet"):
        closure = [math.comb(k + q, q) for q in range(d + 1)]           # nodes on a closed entity of dimension q
        faces = lambda q, r: math.comb(q + 1, r + 1)                      # its faces of dimension r
    else:
        closure = [(k + 1) ** q for q in range(d + 1)]
        faces = lambda q, r: math.comb(q, r) * 2 ** (q - r)
    inner, pairs = [], []
    for q in range(d + 1):
        inner.append(closure[q] - sum(faces(q, r) * inner[r] for r in range(q)))
        pairs.append(closure[q] ** 2 - sum(faces(q, r) * pairs[r] for r in range(q)))
    return (sum(e * i for e, i in zip(ents, inner)), sum(e * p for e, p in zip(ents, pairs)), ents[-1], v)


def work(case):
    d, k, cell = DIM[case["cell"]], case["order"], case["cell"]
    nb = math.comb(k + d, d) if cell in ("tri", "tet") else (k + 1) ** d
    nbytes = flops = 0.0
    sizes = _group_sizes(case) if case["op"] == "group" else [tuple(case[q] for q in ("nx", "ny", "nz") if case[q])]
    for n in sizes:
        n = list(n)
        nodes, pairs, nc, nv = _counts(cell, k, n)
        nnz, ndof = d * d * pairs, d * nodes
        # an unstructured mesh's connectivity and coordinates; a box is its sizes
        mesh = 4 * nc * {"tri": 3, "quad": 4, "tet": 4, "hex": 8}[cell] + 8 * d * nv if case["jitter"] else 0
        if case["op"] == "solve":
            nbytes += 8 * nnz + 4 * pairs + 8 * ndof * 2 + ndof        # K once, its pattern, f, u, the mask
            flops += 2 * nnz
        elif case["op"] == "backward":
            nbytes += mesh + 16 * nc + 16 * ndof + 8                   # rho, u and their gradients, c
            flops += 4 * nc * (nb * d) ** 2
        else:
            nbytes += mesh + 16 * nc + 8 * ndof + 8 * nnz + 8          # rho, u, K, dc, c
            flops += 4 * nc * (nb * d) ** 2
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the definitions in 64 bits

def _lattice(cell, k):
    """Lattice points (multiples of 1/k) of the reference cell's nodes, x fastest."""
    d = DIM[cell]
    pts = [p[::-1] for p in itertools.product(range(k + 1), repeat=d)]
    return [p for p in pts if cell in ("quad", "hex") or sum(p) <= k]


def _lagrange(cell, k, pts):
    """Gradients [q][b][m] at pts of the order-k basis on _lattice's points: products of 1D
    bases on squares and cubes, else by inverting the Vandermonde matrix of monomials."""
    d = DIM[cell]
    if cell in ("quad", "hex"):
        inv = np.linalg.inv(np.vander(np.arange(k + 1) / k, increasing=True))
        val = [np.vander(pts[:, m], k + 1, increasing=True) @ inv for m in range(d)]
        der = [np.vander(pts[:, m], k, increasing=True) * np.arange(1, k + 1) @ inv[1:] for m in range(d)]
        return np.stack([np.stack([math.prod((der if o == m else val)[o][:, a[o]] for o in range(d))
                                   for a in _lattice(cell, k)], 1) for m in range(d)], 2)
    lat = np.array(_lattice(cell, k), np.float64) / k
    powers = _lattice(cell, k)
    mono = lambda x: np.stack([np.prod([x[:, m] ** a[m] for m in range(d)], axis=0) for a in powers], 1)
    coef = np.linalg.inv(mono(lat))
    out = np.zeros((len(pts), len(lat), d))
    for m in range(d):
        dm = np.stack([a[m] * pts[:, m] ** max(a[m] - 1, 0) *
                       np.prod([pts[:, o] ** a[o] for o in range(d) if o != m], axis=0) for a in powers], 1)
        out[:, :, m] = dm @ coef
    return out


def _rule(cell, k):
    """Gauss points and weights of the reference cell: (k + 1)^d on squares and cubes (the
    definition on distorted cells), the collapsed rule of that many points on simplices."""
    d = DIM[cell]
    t, w = np.polynomial.legendre.leggauss(k + 1 if cell in ("quad", "hex") else k + 2)
    t, w = (t + 1) / 2, w / 2
    pts = np.array(list(itertools.product(t, repeat=d)))
    wt = np.array([math.prod(c) for c in itertools.product(w, repeat=d)])
    if cell in ("tri", "tet"):
        left, x = np.ones(len(pts)), np.zeros_like(pts)
        for m in range(d):
            x[:, m] = pts[:, m] * left
            wt = wt * left
            left = left - x[:, m]
        pts = x
    return pts, wt


def _numbering(cell, k, nv, cells):
    """Global node of every (cell, lattice point): vertices, then edges by (min id, max id)
    from the smaller id, faces by their sorted ids (a square's frame starts at its smallest
    vertex, first axis toward the smaller-id neighbour), then interiors cell by cell."""
    d, nc = DIM[cell], len(cells)
    cells = cells.astype(np.int64)
    lat = _lattice(cell, k)
    simplex = cell in ("tri", "tet")
    out = np.zeros((nc, len(lat)), np.int64)
    groups = {1: [], 2: []}
    n_in = 0
    for b, p in enumerate(lat):
        if simplex:
            bary = (k - sum(p),) + tuple(p)
            on = [v for v in range(d + 1) if bary[v]]
            dim = len(on) - 1
        else:
            free = [m for m in range(d) if 0 < p[m] < k]
            on = [v for v in range(1 << d) if all(m in free or ((v >> m) & 1) == (p[m] == k) for m in range(d))]
            dim, bary = len(free), None
        if dim == 0:
            out[:, b] = cells[:, on[0]]
        elif dim == d:
            out[:, b] = -1 - n_in
            n_in += 1
        else:
            groups[dim].append((b, p, bary, on))
    base = nv
    for dim in (1, 2):
        if not groups[dim]:
            continue
        keys = []
        for _, _, _, on in groups[dim]:
            ids = np.sort(cells[:, on], axis=1)
            key = ids[:, 0]
            for c in range(1, len(on)):
                key = key * nv + ids[:, c]
            keys.append(key)
        uniq, inv = np.unique(np.stack(keys, 1), return_inverse=True)
        inv = inv.reshape(nc, -1)
        per = k - 1 if dim == 1 else (math.comb(k - 1, 2) if simplex else (k - 1) ** 2)
        for c, (b, p, bary, on) in enumerate(groups[dim]):
            if dim == 1:
                lo_first = cells[:, on[0]] < cells[:, on[1]]
                if simplex:
                    steps = np.where(lo_first, bary[on[1]], bary[on[0]])       # from the smaller id
                else:
                    m = (on[0] ^ on[1]).bit_length() - 1
                    steps = np.where(lo_first, p[m], k - p[m])                 # on[0] is the low end
                idx = steps - 1
            elif simplex:
                idx = 0
            else:
                ax = [m for m in range(d) if 0 < p[m] < k]
                ids = cells[:, on]
                low = np.array(on)[np.argmin(ids, axis=1)]
                row = np.arange(nc)
                dist = [np.where((low >> a) & 1, k - p[a], p[a]) for a in ax]
                swap = cells[row, low ^ (1 << ax[0])] > cells[row, low ^ (1 << ax[1])]
                a0, a1 = np.where(swap, dist[1], dist[0]), np.where(swap, dist[0], dist[1])
                idx = (a0 - 1) + (k - 1) * (a1 - 1)
            out[:, b] = base + inv[:, c] * per + idx
        base += len(uniq) * per
    inner = out < 0
    out = np.where(inner, base + np.arange(nc)[:, None] * n_in + (-1 - out), out)
    return out, base + nc * n_in


def _elements(cell, k, x, cells, dev):
    """Chunks (start, K_e^0 [c][ldof][ldof]) of the element matrices at unit modulus."""
    d = DIM[cell]
    pts, wt = _rule(cell, k)
    dphi = torch.as_tensor(_lagrange(cell, k, pts), device=dev)
    dgeo = torch.as_tensor(_lagrange(cell, 1, pts), device=dev)
    # order-1 lattice points of a simplex are its vertices in another order: origin, then the unit vectors
    order1 = _lattice(cell, 1)
    vert = [0 if sum(p) == 0 else 1 + p.index(1) for p in order1] if cell in ("tri", "tet") else range(len(order1))
    w = torch.as_tensor(wt, device=dev)
    lam = NU / (1 - NU * NU) if d == 2 else NU / ((1 + NU) * (1 - 2 * NU))
    mu = 1 / (2 * (1 + NU))
    nb, nq = dphi.shape[1], len(wt)
    xc = torch.as_tensor(x, device=dev)[torch.as_tensor(cells, device=dev).long()]
    xc = (xc - xc[:, :1])[:, list(vert)]
    chunk = max(1, int(2e8) // (8 * (nb * d) ** 2 + 8 * nq * nb * d * 3))
    for s in range(0, len(cells), chunk):
        jac = torch.einsum("cvi,qvm->cqim", xc[s:s + chunk], dgeo)
        grad = torch.einsum("qbm,cqmi->cqbi", dphi, torch.linalg.inv(jac))
        g = grad.reshape(len(jac), nq, nb * d)
        pm = torch.bmm((g * (w * torch.linalg.det(jac).abs())[:, :, None]).transpose(1, 2), g)
        pm = pm.reshape(-1, nb, d, nb, d)
        ke = lam * pm + mu * pm.transpose(2, 4)
        ke += mu * torch.einsum("cambm->cab", pm)[:, :, None, :, None] * \
            torch.eye(d, device=dev, dtype=torch.float64)[None, None, :, None, :]
        yield s, ke.reshape(-1, nb * d, nb * d)


def _one(case, s, dev):
    """K's values in CSR order, its block pattern, dc, c and 2 K u of one mesh."""
    cell, k, d = case["cell"], case["order"], DIM[case["cell"]]
    nodes, nn = _numbering(cell, k, len(s["x"]), s["cells"])
    nodes = torch.as_tensor(nodes, device=dev)
    nb = nodes.shape[1]
    rho = torch.as_tensor(s["rho"], device=dev)
    e = EMIN + rho ** P * (E0 - EMIN)
    de = P * rho ** (P - 1) * (E0 - EMIN)
    want_k = case["op"] != "backward"
    u = torch.as_tensor(s["u"], device=dev) if "u" in s else None
    dof = (d * nodes[:, :, None] + torch.arange(d, device=dev)).reshape(len(nodes), -1)
    res = {}
    if want_k:
        keys = torch.unique((nodes[:, :, None] * nn + nodes[:, None, :]).reshape(-1))
        off = torch.searchsorted(keys, torch.arange(nn + 1, device=dev) * nn)
        deg = off[1:] - off[:-1]
        res["vals"] = torch.zeros(d * d * len(keys), dtype=torch.float64, device=dev)
        res["keys"], res["off"], res["nn"] = keys, off, nn
    energy = torch.zeros(len(nodes), dtype=torch.float64, device=dev)
    ku = torch.zeros(d * nn, dtype=torch.float64, device=dev)
    comp = torch.arange(d, device=dev)
    for c0, ke in _elements(cell, k, s["x"], s["cells"], dev):
        sl = slice(c0, c0 + len(ke))
        if want_k:
            a = nodes[sl]
            p = torch.searchsorted(keys, (a[:, :, None] * nn + a[:, None, :]).reshape(-1)).reshape(-1, nb, nb)
            p = p - off[a][:, :, None]
            at = (d * d * off[a])[:, :, None, None, None] + (d * deg[a])[:, :, None, None, None] * \
                comp[None, None, :, None, None] + d * p[:, :, None, :, None] + comp
            res["vals"].index_add_(0, at.reshape(-1), (e[sl][:, None, None] * ke).reshape(-1))
        if u is not None:
            ue = u[dof[sl]]
            fe = torch.bmm(ke, ue[:, :, None])[:, :, 0]
            energy[sl] = (ue * fe).sum(1)
            ku.index_add_(0, dof[sl].reshape(-1), (e[sl][:, None] * fe).reshape(-1))
    if u is not None:
        res.update(dc=-de * energy, c=(e * energy).sum().reshape(1), ku2=2 * ku)
    return res


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ins = _inputs(case, seed)
    parts = [_one(case, s, dev) for s in ins]
    if case["op"] == "step":
        return {k: parts[0][k] for k in ("vals", "dc", "c")}
    if case["op"] == "group":
        return {k: [p[k] for p in parts] for k in ("vals", "dc", "c")}
    r = parts[0]
    if case["op"] == "backward":
        return {"c": r["c"].reshape(()), "g_rho": -r["dc"], "g_u": r["ku2"]}
    # the solve: K of the free dofs, dense, by Cholesky and two steps of refinement
    d, nn = DIM[case["cell"]], r["nn"]
    rows, cols = r["keys"] // nn, r["keys"] % nn
    if d * nn > 21000:
        return None
    p = torch.arange(len(r["keys"]), device=dev) - r["off"][rows]
    deg = r["off"][1:] - r["off"][:-1]
    dense = torch.zeros(d * nn, d * nn, dtype=torch.float64, device=dev)
    for i in range(d):
        for j in range(d):
            dense[d * rows + i, d * cols + j] = r["vals"][d * d * r["off"][rows] + i * d * deg[rows] + d * p + j]
    free = torch.as_tensor(~ins[0]["fixed"], device=dev)
    f = torch.as_tensor(ins[0]["f"], device=dev)[free]
    kf = dense[free][:, free]
    del dense
    low = torch.linalg.cholesky(kf)
    x = torch.cholesky_solve(f[:, None], low)
    for _ in range(2):
        x = x + torch.cholesky_solve(f[:, None] - kf @ x, low)
    u = torch.zeros(d * nn, dtype=torch.float64, device=dev)
    u[free] = x[:, 0]
    return {"u": u}
