"""The sensitivities of general quadrilaterals and hexahedra with FP64 element matrices
(strain_general.cu): each cell against the oracle to the tolerance of the FP64 form, and
the error of all cells together against an evaluation in extended precision, which shows a
few lost bits.

Bounds of the latter, from the arithmetic: order 1 in float pairs (u rounded to 2^-48, some
ten operations of 2^-48 a value, averaged over a cell's points) 4.5e-15 of dc; orders 2 and
3 in FP64 3e-15 (1D tables rounded to 2^-53 whose sums cancel to about a tenth)."""
import itertools

import numpy as np
import pytest
import torch

import oracle
from helpers import TOL64
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng
MAT = (1.0, 1e-9, 0.3, 3.0, 0)
# one block of threads and ragged ones, both block sizes of k_strain_quad
MESHES = {
    "quad q1 3x2": ("quad", 1, lambda: W.quad_grid(3, 2, 0.2, g(1))),
    "quad q1": ("quad", 1, lambda: W.quad_grid(71, 47, 0.2, g(2))),
    "quad q2 5x3": ("quad", 2, lambda: W.quad_grid(5, 3, 0.2, g(3))),
    "quad q2": ("quad", 2, lambda: W.quad_grid(53, 45, 0.2, g(4))),
    "quad q2 large": ("quad", 2, lambda: W.quad_grid(173, 115, 0.2, g(4))),
    "quad q3": ("quad", 3, lambda: W.quad_grid(41, 35, 0.2, g(5))),
    "hex q1 2x2x2": ("hex", 1, lambda: W.hex_grid(2, 2, 2, 0.15, g(7))),
    "hex q1": ("hex", 1, lambda: W.hex_grid(19, 13, 11, 0.15, g(8))),
    "hex q2": ("hex", 2, lambda: W.hex_grid(9, 7, 5, 0.15, g(9))),
    "hex q3": ("hex", 3, lambda: W.hex_grid(5, 5, 4, 0.15, g(10))),
}
L = np.longdouble


def gauss(k):
    """Points and weights on [0, 1] of the (k + 1)-point rule."""
    r = lambda v: np.sqrt(L(v))
    if k == 1:
        t, w = [-1 / r(3), 1 / r(3)], [L(1), L(1)]
    elif k == 2:
        t, w = [-r(L(3) / 5), L(0), r(L(3) / 5)], [L(5) / 9, L(8) / 9, L(5) / 9]
    else:
        a, b = r(L(3) / 7 - L(2) / 7 * r(L(6) / 5)), r(L(3) / 7 + L(2) / 7 * r(L(6) / 5))
        wa, wb = (18 + r(30)) / 36, (18 - r(30)) / 36
        t, w = [-b, -a, a, b], [wb, wa, wa, wb]
    return (np.array(t) + 1) / 2, np.array(w) / 2


def basis(k, t):
    """Values and derivatives [q][j] of the 1D Lagrange basis on 0, 1/k, .., 1."""
    nodes = [L(j) / k for j in range(k + 1)]
    val, der = np.ones((len(t), k + 1), L), np.zeros((len(t), k + 1), L)
    for j in range(k + 1):
        for o in range(k + 1):
            if o != j:
                der[:, j] = der[:, j] * (t - nodes[o]) / (nodes[j] - nodes[o]) + val[:, j] / (nodes[j] - nodes[o])
                val[:, j] = val[:, j] * (t - nodes[o]) / (nodes[j] - nodes[o])
    return val, der


def energies(cell, k, x, cells, cell_nodes, lattice, u):
    """u_e^T K_e^0 u_e in extended precision."""
    d = x.shape[1]
    t, w = gauss(k)
    (v1, d1), (vg, dg) = basis(k, t), basis(1, t)
    lam, mu = (L(0.3) / (1 - L(0.3) ** 2) if d == 2 else L(0.3) / ((1 + L(0.3)) * (1 - 2 * L(0.3)))), 1 / (2 * (1 + L(0.3)))
    corner = np.array([[(v >> m) & 1 for m in range(d)] for v in range(1 << d)])
    ue = u.reshape(-1, d)[cell_nodes].astype(L)
    xe = (x[cells] - x[cells][:, :1]).astype(L)
    s = np.zeros(len(cells), L)
    for q in itertools.product(range(k + 1), repeat=d):
        def grads(val, der, idx):   # [local node][axis]
            out = np.ones((len(idx), d), L)
            for m in range(d):
                for o in range(d):
                    out[:, m] = out[:, m] * (der if o == m else val)[q[o], idx[:, o]]
            return out
        J = np.einsum("evi,vm->eim", xe, grads(vg, dg, corner))
        U = np.einsum("ebi,bm->eim", ue, grads(v1, d1, lattice))
        if d == 2:
            det = J[:, 0, 0] * J[:, 1, 1] - J[:, 0, 1] * J[:, 1, 0]
            adj = np.stack([J[:, 1, 1], -J[:, 0, 1], -J[:, 1, 0], J[:, 0, 0]], 1).reshape(-1, 2, 2)
        else:
            c = [[J[:, (i + 1) % 3, (m + 1) % 3] * J[:, (i + 2) % 3, (m + 2) % 3] -
                  J[:, (i + 1) % 3, (m + 2) % 3] * J[:, (i + 2) % 3, (m + 1) % 3] for i in range(3)] for m in range(3)]
            adj = np.stack([c[m][i] for m in range(3) for i in range(3)], 1).reshape(-1, 3, 3)
            det = (J[:, 0, :] * adj[:, :, 0]).sum(1)
        gu = np.einsum("eim,emj->eij", U, adj) / det[:, None, None]
        tr = np.einsum("eii->e", gu)
        dens = lam * tr * tr + mu * (gu * (gu + gu.swapaxes(1, 2))).sum((1, 2))
        s += np.prod([w[o] for o in q]) * abs(det) * dens
    return s


@pytest.mark.parametrize("name", MESHES)
def test_error_against_64_bits(lib, name):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    d = x.shape[1]
    m = lib.Mesh(cell, k, x, cells, *MAT)
    assert m.routes["sensitivity"] == "strain"
    rho = g(11).uniform(0.001, 1.0, len(cells))
    u = g(12).standard_normal(m.ndof)
    dc, c = m.sensitivity(torch.as_tensor(rho, device="cuda"), torch.as_tensor(u, device="cuda"))
    dc = dc.cpu().numpy()
    dco, _, _, sabs = oracle.sensitivity(cell, k, x, cells, MAT, rho, u, with_abs=True)
    assert np.all(np.abs(dc - dco) <= TOL64 * 3 * rho ** 2 * (1 - 1e-9) * sabs)
    # the reference cell's nodes give the local order
    one = np.array([[(v >> a) & 1 for a in range(d)] for v in range(1 << d)], np.float64)
    oc = np.arange(1 << d, dtype=np.int32)[None]
    local = oracle.node_coords(cell, k, one, oc)[lib.Mesh(cell, k, one, oc, *MAT).cell_nodes().cpu().numpy()[0]]
    r = rho.astype(L)
    s = energies(cell, k, x, cells, m.cell_nodes().cpu().numpy(), np.rint(k * local).astype(int), u)
    ref = -3 * r * r * (1 - L(1e-9)) * s
    err = (dc - ref).astype(np.float64)
    assert np.linalg.norm(err) <= (4.5e-15 if k == 1 else 3e-15) * float(np.sqrt((ref * ref).sum()))
    co = ((L(1e-9) + r ** 3 * (1 - L(1e-9))) * s).sum()
    assert abs(float(c.item() - co)) <= 3e-15 * float(co)


@pytest.mark.parametrize("h", [1e-12, 1e9])
@pytest.mark.parametrize("name", ["quad q1 3x2", "quad q2 5x3", "hex q1 2x2x2", "hex q2"])
def test_cells_of_any_size(lib, name, h):
    """|det J| of 1e-36 and 1e27: the weights are FP64, so no point loses its tail."""
    cell, k, mk = MESHES[name]
    x, cells = mk()
    m = lib.Mesh(cell, k, x * h, cells, *MAT)
    rho = np.full(len(cells), 0.7)
    u = h * g(12).standard_normal(m.ndof)
    dc, _ = m.sensitivity(torch.as_tensor(rho, device="cuda"), torch.as_tensor(u, device="cuda"))
    dco, _, _, sabs = oracle.sensitivity(cell, k, x * h, cells, MAT, rho, u, with_abs=True)
    assert np.all(np.abs(dc.cpu().numpy() - dco) <= TOL64 * 3 * rho ** 2 * (1 - 1e-9) * sabs)
