"""The backward from the cells' forces (vjp.cu): no further from 64 bits than the product
over the assembled matrix that it replaced, on 2D cells of several points, on cells
whose |det J| is 1e-27, and on both sides of the cell counts from which P2 tetrahedra
and hexahedra take it.

The product itself (K assembled, then soptx_spmv) gives the bound of g_u for all rows
together, with 5% for the scatter of such a norm over some ten thousand rows."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL64
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng
MAT = (1.0, 1e-9, 0.3, 3.0, 0)


def sheared(mesh):
    c, cl = mesh
    c = c + 0.03 / c.max() * c[:, :1] ** 2 * np.eye(c.shape[1])[0]     # widths that grow along x
    return c @ (np.eye(c.shape[1]) + 0.2 * np.arange(c.shape[1] ** 2).reshape(c.shape[1], -1) / 9).T, cl


MESHES = {
    "tri p2": ("tri", 2, lambda: W.triangle_grid(80, 60, 0.2, g(2))),
    "tri p3": ("tri", 3, lambda: W.triangle_grid(80, 60, 0.2, g(3))),
    "quad q2 sheared": ("quad", 2, lambda: sheared(W.structured_quad(110, 80))),
    "tet p2 of 2016": ("tet", 2, lambda: W.kuhn_tets(8, 7, 6, 0.15, g(5))),
    "tet p2 of 2058": ("tet", 2, lambda: W.kuhn_tets(7, 7, 7, 0.15, g(5))),
    "hex q1 of 9975": ("hex", 1, lambda: sheared(W.structured_hex(25, 21, 19))),
    "hex q1 of 10120": ("hex", 1, lambda: sheared(W.structured_hex(23, 22, 20))),
}


def gradients(lib, name, h, us):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    m = lib.Mesh(cell, k, x * h, cells, *MAT)
    rho, u = g(8).uniform(0.001, 1.0, len(cells)), us * g(7).standard_normal(m.ndof)
    gr, gu = m.compliance_vjp(torch.as_tensor(rho, device="cuda"), torch.as_tensor(u, device="cuda"),
                              torch.ones(1, dtype=torch.float64, device="cuda"))
    gr_o, gu_o = oracle.compliance_vjp(cell, k, x * h, cells, MAT, rho, u, 1.0)
    _, _, _, sabs = oracle.sensitivity(cell, k, x * h, cells, MAT, rho, u, with_abs=True)
    rp, ci, va, _ = oracle.assemble(cell, k, x * h, cells, MAT, rho, absval=True)
    row = np.add.reduceat(va * np.abs(u[ci]), rp[:-1])
    product = 2 * m.spmv(m.assemble_K(torch.as_tensor(rho, device="cuda")), torch.as_tensor(u, device="cuda"))
    return gr.cpu().numpy(), gu.cpu().numpy(), gr_o, gu_o, 3 * rho ** 2 * sabs, 2 * row, product.cpu().numpy()


@pytest.mark.parametrize("name", MESHES)
def test_error_of_all_rows(lib, name):
    gr, gu, gr_o, gu_o, rs, us, product = gradients(lib, name, 1.0, 1.0)
    assert np.all(np.abs(gr - gr_o) <= TOL64 * rs)
    assert np.all(np.abs(gu - gu_o) <= TOL64 * us)
    assert np.linalg.norm(gu - gu_o) <= 1.05 * np.linalg.norm(product - gu_o)


@pytest.mark.parametrize("name", [n for n in MESHES if n.startswith(("tet", "hex"))])
def test_small_cells(lib, name):
    """Cells of 1e-9: the energies, near 1e-33, keep 2^-149 of absolute precision, some
    1e-12 a cell and 2e-13 together; a weight that had lost its tail left 4e-13 .. 8e-13."""
    gr, gu, gr_o, gu_o, _, us, _ = gradients(lib, name, 1e-9, 1e-12)
    assert np.linalg.norm(gr - gr_o) <= 2e-13 * np.linalg.norm(gr_o)
    assert np.all(np.abs(gu - gu_o) <= TOL64 * us)
