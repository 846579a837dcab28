"""Linear tetrahedra in the block-row kernel (chunks and CTAs of their own sizes): meshes
of one chunk, of a few and of many per CTA, and a vertex with more row blocks than a
chunk holds, against the oracle, both element precisions."""
import numpy as np
import pytest
import torch

from helpers import TOL32, TOL64, oracle_csr
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng


def star(n):
    """Tetrahedra from one vertex to the triangles of a sphere of n x 2n quadrilaterals."""
    th, ph = np.pi * (np.arange(n + 1)) / n, 2 * np.pi * np.arange(2 * n) / (2 * n)
    ring = lambda i: 1 + (i - 1) * 2 * n + np.arange(2 * n)
    x = [[0, 0, 0]] + [[np.sin(t) * np.cos(p), np.sin(t) * np.sin(p), np.cos(t)] for t in th[1:-1] for p in ph]
    x += [[0, 0, 1.0], [0, 0, -1.0]]
    top, bot = len(x) - 2, len(x) - 1
    cells = []
    for j in range(2 * n):
        k = (j + 1) % (2 * n)
        cells.append([0, top, ring(1)[j], ring(1)[k]])
        cells.append([0, bot, ring(n - 1)[k], ring(n - 1)[j]])
        for i in range(1, n - 1):
            a, b, c, d = ring(i)[j], ring(i)[k], ring(i + 1)[j], ring(i + 1)[k]
            cells += [[0, a, c, b], [0, b, c, d]]
    return np.array(x), np.array(cells, np.int32)


MESHES = {"1x1x1": lambda: W.kuhn_tets(1, 1, 1), "5x4x3": lambda: W.kuhn_tets(5, 4, 3, 0.15, g(1)),
          "31x23x19": lambda: W.kuhn_tets(31, 23, 19, 0.15, g(2)), "star of 288": lambda: star(9)}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", MESHES)
def test_rows_match_oracle(lib, name, prec):
    x, cells = MESHES[name]()
    mat = (1.0, 0.0, 0.3, 3.0, 0)
    m = lib.Mesh("tet", 1, x, cells, *mat, elem_prec=prec)
    assert m.routes["assembly"] == ("stream" if prec == "fp64" else "contract")
    tol, floor = (TOL64, 1e-15) if prec == "fp64" else (TOL32, 1e-7)
    rho = g(5).uniform(0.001, 1.0, len(cells))
    r = torch.as_tensor(rho, device="cuda")
    vals = m.assemble_K(r)
    _, _, v, va, _ = oracle_csr("tet", 1, x, cells, mat, rho)
    assert np.all(np.abs(vals.cpu().numpy() - v) <= tol * va + floor * va.max())
    assert torch.equal(m.assemble_K(r), vals)
