"""The solve with K in shared memory (cgresident.cu) against the oracle's direct solve:
2D and 3D, shuffled node numbers (halos over the whole mesh), prescribed values, an
untouched constrained node (an empty row), a few nodes, a warm start, several
launches, and a matrix too large for it beside those that fit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MAT = (1.0, 1e-9, 0.3, 3.0, 0)
g = np.random.default_rng


def shuffled(mesh):
    x, cells = mesh
    p = g(3).permutation(len(x))
    inv = np.empty_like(p)
    inv[p] = np.arange(len(p))
    return x[p], inv[np.asarray(cells)]


def with_loose_node(mesh):
    x, cells = mesh
    return np.vstack([x, x.max(axis=0) + 1.0]), cells


MESHES = {
    "quad 3x2": ("quad", 1, lambda: W.structured_quad(3, 2)),
    "quad 33x21": ("quad", 1, lambda: W.structured_quad(33, 21)),
    "quad shuffled": ("quad", 1, lambda: shuffled(W.quad_grid(24, 20, 0.2, g(1)))),
    "tri p3": ("tri", 3, lambda: W.triangle_grid(10, 8, 0.2, g(2))),
    "hex 7x4x3": ("hex", 1, lambda: W.structured_hex(7, 4, 3)),
    "hex shuffled": ("hex", 1, lambda: shuffled(W.hex_grid(9, 7, 6, 0.15, g(4)))),
    "hex q2": ("hex", 2, lambda: W.hex_grid(5, 3, 2, 0.1, g(5))),
    "tet p2 loose node": ("tet", 2, lambda: with_loose_node(W.kuhn_tets(5, 3, 3, 0.15, g(6)))),
    "hex too large": ("hex", 1, lambda: W.structured_hex(52, 17, 17)),
}


@pytest.mark.parametrize("name", MESHES)
def test_solution_matches_direct_solve(lib, name):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    m = lib.Mesh(cell, k, x, cells, *MAT)
    d = m.dim
    rho = g(7).uniform(0.3, 1.0, len(cells))
    vals = m.assemble_K(torch.as_tensor(rho, device="cuda"))
    xn = oracle.node_coords(cell, k, x, cells)
    lo = x[:, 0].min()
    fixed = np.repeat(xn[:, 0] < lo + 1e-9, d)
    if name.endswith("loose node"):
        fixed |= np.repeat(np.arange(len(xn)) == len(x) - 1, d)
    ub = np.where(fixed, 0.1 * g(8).standard_normal(m.ndof), 0.0)
    f = g(9).standard_normal(m.ndof)
    rp, ci, v, ndof = oracle.assemble(cell, k, x, cells, MAT, rho)
    t = lambda a: torch.as_tensor(a, device="cuda")
    kw = dict(u_fixed=t(ub), rtol=1e-12, max_iter=20000)
    u, info = m.solve(vals, t(fixed), t(f), check_every=7, **kw)
    assert info["converged"] and info["iterations"] % 7 == 0
    un = u.cpu().numpy()
    assert np.array_equal(un[fixed], ub[fixed])
    if name != "hex too large":
        ref = oracle.solve_dirichlet(rp, ci, v, fixed, f, ub)
        assert np.linalg.norm(un - ref) <= 1e-8 * np.linalg.norm(ref)
    else:   # a direct solve of 52k dofs is slow: the residual
        r = (f - oracle.spmv(rp, ci, v, un))[~fixed]
        b = (f - oracle.spmv(rp, ci, v, ub))[~fixed]
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)
    # the same bits again, and the same iterates whatever the check interval
    u2, _ = m.solve(vals, t(fixed), t(f), check_every=7, **kw)
    assert torch.equal(u, u2)
    kw.update(rtol=1e-300, max_iter=23)
    ua, ia = m.solve(vals, t(fixed), t(f), check_every=4, **kw)
    ub_, ib = m.solve(vals, t(fixed), t(f), check_every=100, **kw)
    assert ia["iterations"] == ib["iterations"] == 23 and torch.equal(ua, ub_)
    assert ia["rel_residual"] == ib["rel_residual"]
    # a warm start at the solution has nothing to do
    u3, i3 = m.solve(vals, t(fixed), t(f), u_fixed=t(ub), u0=u, rtol=1e-9, max_iter=100)
    assert i3["converged"] and i3["iterations"] <= 10


def test_more_iterations_than_one_launch(lib):
    """The state is carried from one launch (4096 iterations) to the next: 4101 iterations
    count to the cap and stay at the solution."""
    x, cells = W.structured_quad(12, 4)
    m = lib.Mesh("quad", 1, x, cells, *MAT)
    vals = m.assemble_K(torch.full((len(cells),), 0.5, dtype=torch.float64, device="cuda"))
    fixed = torch.as_tensor(np.repeat(x[:, 0] < 1e-9, 2), device="cuda")
    f = torch.ones(m.ndof, dtype=torch.float64, device="cuda")
    u, info = m.solve(vals, fixed, f, rtol=1e-12, max_iter=20000)
    assert info["converged"]
    ul, il = m.solve(vals, fixed, f, rtol=1e-300, max_iter=4101, check_every=4101)
    assert il["iterations"] == 4101
    assert float((ul - u).abs().max()) <= 1e-8 * float(u.abs().max())
