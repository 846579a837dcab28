"""The block-row kernel of 3D meshes (k_block_rows) at its edges, against the
oracle: meshes of one cell and of many chunks, a pair shared by several lanes
(more cells than a lane walks) and by all 32 of them, every source of blocks
(contraction, one matrix, streamed cached matrices), moduli
outside the float-pair range on those pairs, and CSR values at an odd 8-byte
address (plain stores in place of the bulk copies)."""
import numpy as np
import pytest
import torch

from helpers import TOL32, TOL64, oracle_csr
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def ring(n):
    """n tetrahedra around one edge."""
    t = 2 * np.pi * np.arange(n) / n
    x = np.vstack([[0, 0, -1.0], [0, 0, 1.0], np.stack([np.cos(t), np.sin(t), 0 * t], axis=1)])
    return x, np.array([[0, 1, 2 + k, 2 + (k + 1) % n] for k in range(n)], np.int32)


def sheared(n):
    c, cl = W.structured_hex(*n)
    # widths that grow along x: parallelepipeds, no two layers alike
    c = c + 0.03 * c[:, :1] ** 2 * np.array([1.0, 0.0, 0.0])
    return c @ np.array([[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]]).T, cl


g = np.random.default_rng
MESHES = {
    "one tet p3": ("tet", 3, lambda: (np.array([[0, 0, 0], [1, 0.1, 0], [0.2, 0.9, 0], [0, 0.1, 1.0]]),
                                      np.array([[0, 1, 2, 3]], np.int32))),
    "ring of 9 p2": ("tet", 2, lambda: ring(9)),
    "ring of 40 p1": ("tet", 1, lambda: ring(40)),
    "ring of 40 p2": ("tet", 2, lambda: ring(40)),
    "tets p2": ("tet", 2, lambda: W.kuhn_tets(7, 5, 4, 0.15, g(1))),
    "tets p3": ("tet", 3, lambda: W.kuhn_tets(3, 2, 2, 0.15, g(2))),
    "hexes q1 distorted": ("hex", 1, lambda: W.hex_grid(9, 7, 5, 0.15, g(3))),
    "hexes q2 distorted": ("hex", 2, lambda: W.hex_grid(4, 3, 3, 0.1, g(4))),
    "hexes q1 sheared": ("hex", 1, lambda: sheared((8, 5, 4))),
    "hexes q2 sheared": ("hex", 2, lambda: sheared((4, 3, 2))),
    "box q2": ("hex", 2, lambda: W.structured_hex(5, 4, 3)),
    "box q3": ("hex", 3, lambda: W.structured_hex(3, 2, 2)),
}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", MESHES)
def test_rows_match_oracle(lib, name, prec):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    mat = (1.0, 0.0, 0.3, 3.0, 0)
    m = lib.Mesh(cell, k, x, cells, *mat, elem_prec=prec)
    # (distorted cells with FP32 element matrices take the row gather; one cell is a uniform mesh)
    assert m.routes["assembly"] == ("gather" if "distorted" in name and prec == "fp32" else "pairs" if m.path == "uniform"
                                    else "contract" if prec == "fp32" else "stream")
    tol, floor = (TOL64, 1e-15) if prec == "fp64" else (TOL32, 1e-7)
    rho = g(5).uniform(0.001, 1.0, len(cells))
    for tiny in (False, True):
        if tiny:   # moduli of 1e-27 and zero
            rho[::4] = 1e-9
            rho[1::7] = 0.0
        r = torch.as_tensor(rho, device="cuda")
        vals = m.assemble_K(r)
        _, _, v, va, _ = oracle_csr(cell, k, x, cells, mat, rho)
        assert np.all(np.abs(vals.cpu().numpy() - v) <= tol * va + floor * va.max() + 1e-300)
        assert torch.equal(m.assemble_K(r), vals)   # the counter of chunks was set back
        odd = torch.full((m.nnz + 1,), np.nan, dtype=torch.float64, device="cuda")[1:]
        assert odd.data_ptr() % 16 == 8
        assert torch.equal(m.assemble_K(r, vals=odd), vals)
