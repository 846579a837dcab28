"""Both sides of the cell counts from which Q1 hexahedra and P2 tetrahedra with cached FP64
matrices are assembled by the block rows (fewer: by the gather): K against the oracle, the
one-call step bitwise the separate calls, pairs of more cells than lanes, and an odd
8-byte address."""
import numpy as np
import pytest
import torch

from helpers import TOL64, oracle_csr
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng


def rings(n, layers):
    """Stacked rings of n tetrahedra around one axis."""
    t = 2 * np.pi * np.arange(n) / n
    axis = np.stack([np.zeros(layers + 1), np.zeros(layers + 1), np.arange(layers + 1.0)], 1)
    x = [axis] + [np.stack([np.cos(t), np.sin(t), 0 * t + k + 0.5], 1) for k in range(layers)]
    cells = [[k, k + 1, layers + 1 + k * n + j, layers + 1 + k * n + (j + 1) % n]
             for k in range(layers) for j in range(n)]
    return np.vstack(x), np.array(cells, np.int32)


def sheared(n):
    c, cl = W.structured_hex(*n)
    c = c + 0.03 * c[:, :1] ** 2 / n[0] * np.array([1.0, 0.0, 0.0])
    return c @ np.array([[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]]).T, cl


MESHES = {
    "hex q1 of 4096": ("hex", 1, lambda: W.hex_grid(16, 16, 16, 0.15, g(1))),
    "hex q1 of 4104": ("hex", 1, lambda: W.hex_grid(19, 18, 12, 0.15, g(2))),
    "hex q1 sheared": ("hex", 1, lambda: sheared((19, 18, 13))),
    "tet p2 of 252": ("tet", 2, lambda: W.kuhn_tets(7, 3, 2, 0.15, g(3))),
    "tet p2 of 270": ("tet", 2, lambda: W.kuhn_tets(5, 3, 3, 0.15, g(4))),
    "rings of 20 p2": ("tet", 2, lambda: rings(20, 14)),
}


@pytest.mark.parametrize("name", MESHES)
def test_both_sides(lib, name):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    mat = (1.0, 0.0, 0.3, 3.0, 0)
    m = lib.Mesh(cell, k, x, cells, *mat)
    rho = g(5).uniform(0.001, 1.0, len(cells))
    u = torch.as_tensor(g(6).standard_normal(m.ndof), device="cuda")
    for tiny in (False, True):
        if tiny:   # moduli of 1e-27 and zero
            rho[::4] = 1e-9
            rho[1::7] = 0.0
        r = torch.as_tensor(rho, device="cuda")
        vals = m.assemble_K(r)
        _, _, v, va, _ = oracle_csr(cell, k, x, cells, mat, rho)
        assert np.all(np.abs(vals.cpu().numpy() - v) <= TOL64 * va + 1e-15 * va.max() + 1e-300)
        sv, dc, _ = m.step(r, u)
        assert torch.equal(sv, vals) and torch.equal(dc, m.sensitivity(r, u)[0])
        odd = torch.full((m.nnz + 1,), np.nan, dtype=torch.float64, device="cuda")[1:]
        assert odd.data_ptr() % 16 == 8
        assert torch.equal(m.assemble_K(r, vals=odd), vals)
