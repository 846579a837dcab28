"""Which way each call took (soptx_mesh_last_routes): the one-launch step of small lattices,
the backward from the cells' forces, the solve with K in shared memory and the block rows
are the ones that ran where they are meant to, and not beyond."""
import numpy as np
import pytest
import torch

from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng
MAT = (1.0, 1e-9, 0.3, 3.0, 0)


def mesh(lib, cell, k, xc, prec="fp64"):
    m = lib.Mesh(cell, k, *xc, *MAT, elem_prec=prec)
    r = torch.full((m.n_cells,), 0.5, dtype=torch.float64, device="cuda")
    u = torch.as_tensor(g(1).standard_normal(m.ndof), device="cuda")
    return m, r, u


@pytest.mark.parametrize("shape,route", [((60, 20), "one launch"), ((48, 32), "one launch"), ((49, 32), "launches"),
                                         ((16, 8, 8), "one launch"), ((5, 41, 5), "launches")], ids=str)
def test_lattice_step(lib, shape, route):
    d = len(shape)
    m, r, u = mesh(lib, "quad" if d == 2 else "hex", 1, W.structured_quad(*shape) if d == 2 else W.structured_hex(*shape))
    assert m.last_routes() == {"assembly": None, "step": None, "backward": None, "solve": None}
    m.step(r, u)
    assert m.last_routes()["step"] == route
    m.assemble_K(r)
    assert m.last_routes()["assembly"] == "lattice"


BACKWARD = {
    "lattice 2d": ("quad", 1, lambda: W.structured_quad(17, 9), "fp64", "forces"),
    "lattice 3d": ("hex", 1, lambda: W.structured_hex(13, 5, 4), "fp64", "forces"),
    "lattice fp32": ("hex", 1, lambda: W.structured_hex(13, 5, 4), "fp32", "product"),
    "tri p1": ("tri", 1, lambda: W.triangle_grid(13, 6, 0.2, g(1)), "fp64", "forces"),
    "tri p2": ("tri", 2, lambda: W.triangle_grid(9, 7, 0.2, g(2)), "fp64", "forces"),
    "tri p3 small": ("tri", 3, lambda: W.triangle_grid(60, 60, 0.2, g(3)), "fp64", "product"),
    "tri p3": ("tri", 3, lambda: W.triangle_grid(80, 60, 0.2, g(3)), "fp64", "forces"),
    "tet p1": ("tet", 1, lambda: W.kuhn_tets(5, 3, 2, 0.15, g(4)), "fp64", "forces"),
    "tet p2 small": ("tet", 2, lambda: W.kuhn_tets(8, 7, 6, 0.15, g(5)), "fp64", "product"),
    "tet p2": ("tet", 2, lambda: W.kuhn_tets(7, 7, 7, 0.15, g(5)), "fp64", "forces"),
    "quad q2 box": ("quad", 2, lambda: W.structured_quad(110, 80), "fp64", "forces"),
    "quad distorted": ("quad", 1, lambda: W.quad_grid(9, 7, 0.2, g(6)), "fp64", "product"),
}


@pytest.mark.parametrize("name", BACKWARD)
def test_backward(lib, name):
    from paper_2505_02438_gb300 import _native as N
    cell, k, mk, prec, route = BACKWARD[name]
    m, r, u = mesh(lib, cell, k, mk(), prec)
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    N.lib().soptx_debug_fail_alloc_after(1)
    try:
        m.compliance_vjp(r, u, one)
    finally:
        N.lib().soptx_debug_fail_alloc_after(0)
    assert m.last_routes()["backward"] == "element matrices"
    m.compliance_vjp(r, u, one)
    assert m.last_routes()["backward"] == route


@pytest.mark.parametrize("shape,route", [((33, 21), "resident"), ((7, 4, 3), "resident"), ((60, 20, 4), "resident"),
                                         ((52, 17, 17), "loop")], ids=str)
def test_solve(lib, shape, route):
    x, cells = W.structured_quad(*shape) if len(shape) == 2 else W.structured_hex(*shape)
    m, r, u = mesh(lib, "quad" if len(shape) == 2 else "hex", 1, (x, cells))
    fixed = torch.as_tensor(np.repeat(x[:, 0] < 1e-9, len(shape)), device="cuda")
    m.solve(m.assemble_K(r), fixed, u, max_iter=20)
    assert m.last_routes()["solve"] == route


def test_assembly(lib):
    for cell, k, xc, prec, route in (
            ("hex", 1, W.hex_grid(16, 16, 16, 0.15, g(1)), "fp64", "gather"),
            ("hex", 1, W.hex_grid(19, 18, 12, 0.15, g(2)), "fp64", "stream"),
            ("tet", 2, W.kuhn_tets(7, 3, 2, 0.15, g(3)), "fp64", "gather"),
            ("tet", 2, W.kuhn_tets(5, 3, 3, 0.15, g(4)), "fp64", "stream"),
            ("tet", 2, W.kuhn_tets(2, 1, 1, 0.0), "fp32", "contract"),
            ("hex", 2, W.structured_hex(3, 2, 2), "fp64", "pairs"),
            ("quad", 1, W.quad_grid(9, 7, 0.2, g(6)), "fp64", "gather")):
        m, r, u = mesh(lib, cell, k, xc, prec)
        m.assemble_K(r)
        assert m.last_routes()["assembly"] == route, (cell, k, prec)
        m.step(r, u)
        assert m.last_routes() == {"assembly": route, "step": "launches", "backward": None, "solve": None}
