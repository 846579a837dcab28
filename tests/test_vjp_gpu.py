"""The backward from the cells' nodal forces (vjp.cu) against the oracle: box
lattices in 2D and 3D (one cell, ragged blocks), every affine cell it is compiled
for, an incoming gradient other than one, and moduli outside the float-pair range."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL64
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng


def sheared(mesh):
    c, cl = mesh
    c = c + 0.03 * c[:, :1] ** 2 * np.eye(c.shape[1])[0]     # widths that grow along x
    return c @ (np.eye(c.shape[1]) + 0.2 * np.arange(c.shape[1] ** 2).reshape(c.shape[1], -1) / 9).T, cl


MESHES = {
    "lattice 1x1": ("quad", 1, lambda: W.structured_quad(1, 1)),
    "lattice 17x9": ("quad", 1, lambda: W.structured_quad(17, 9)),
    "lattice 1x1x1": ("hex", 1, lambda: W.structured_hex(1, 1, 1)),
    "lattice 13x5x4": ("hex", 1, lambda: W.structured_hex(13, 5, 4)),
    "tri p1": ("tri", 1, lambda: W.triangle_grid(13, 6, 0.2, g(1))),
    "tri p2": ("tri", 2, lambda: W.triangle_grid(9, 7, 0.2, g(2))),
    "tri p3": ("tri", 3, lambda: W.triangle_grid(9, 8, 0.2, g(3))),
    "tet p1": ("tet", 1, lambda: W.kuhn_tets(5, 3, 2, 0.15, g(4))),
    "tet p2": ("tet", 2, lambda: W.kuhn_tets(4, 3, 2, 0.15, g(5))),
    "quad q1 sheared": ("quad", 1, lambda: sheared(W.structured_quad(11, 13))),
    "quad q2 box": ("quad", 2, lambda: W.structured_quad(9, 5)),
    "hex q1 sheared": ("hex", 1, lambda: sheared(W.structured_hex(5, 6, 5))),
}


@pytest.mark.parametrize("name", MESHES)
def test_gradients_match_oracle(lib, name):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    mat = (1.0, 0.0, 0.3, 3.0, 0)
    m = lib.Mesh(cell, k, x, cells, *mat)
    u = g(7).standard_normal(m.ndof)
    rho = g(8).uniform(0.001, 1.0, len(cells))
    scale = -1.75
    gout = torch.tensor([scale], dtype=torch.float64, device="cuda")
    for tiny in (False, True):
        if tiny:   # moduli of 1e-27 and zero
            rho[::5] = 1e-9
            rho[1::7] = 0.0
        gr, gu = m.compliance_vjp(torch.as_tensor(rho, device="cuda"), torch.as_tensor(u, device="cuda"), gout)
        gr_o, gu_o = oracle.compliance_vjp(cell, k, x, cells, mat, rho, u, scale)
        _, _, _, sabs = oracle.sensitivity(cell, k, x, cells, mat, rho, u, with_abs=True)
        rp, ci, va, _ = oracle.assemble(cell, k, x, cells, mat, rho, absval=True)
        row = np.add.reduceat(va * np.abs(u[ci]), rp[:-1])
        assert np.all(np.abs(gr.cpu().numpy() - gr_o) <= TOL64 * abs(scale) * 3 * rho ** 2 * sabs + 1e-300)
        assert np.all(np.abs(gu.cpu().numpy() - gu_o) <= TOL64 * 2 * abs(scale) * row + 1e-40)
