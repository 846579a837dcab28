"""CSR values of 3D meshes far from one (k_block_rows): values near 1e-18 .. 1e-30, where
the fast conversion of float pairs would be off by up to 2^-126 each, values beyond the
largest float, and meshes whose moduli are all outside the float-pair range (all cells
of a mesh alike, so the floor of 1e-15 of the largest value, which entries that vanish by
symmetry need, hides no block)."""
import numpy as np
import pytest
import torch

from helpers import TOL32, TOL64, oracle_csr
from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng
MESHES = {"tets p2": ("tet", 2, lambda: W.kuhn_tets(5, 4, 3, 0.15, g(1))),
          "hexes q2 distorted": ("hex", 2, lambda: W.hex_grid(3, 3, 2, 0.1, g(3))),
          "box q2": ("hex", 2, lambda: W.structured_hex(4, 3, 2))}
# modulus of the solid and grid spacing: values of about their product.  FP32 element
# matrices are contracted from FP32 geometry, whose |det J| of spacing^3 has to be a normal float.
SCALES = {"fp64": [(1e-9, 1e-9), (1e-12, 1e-12), (1e-12, 1e-15), (1e-12, 1e-18), (1e-17, 1e-9), (1e18, 1e25)],
          "fp32": [(1e-9, 1e-9), (1e-12, 1e-11), (1e-17, 1e-11)]}


@pytest.mark.parametrize("prec,E0,h", [(p, *s) for p in SCALES for s in SCALES[p]])
@pytest.mark.parametrize("name", MESHES)
def test_values_of_any_size(lib, name, prec, E0, h):
    cell, k, mk = MESHES[name]
    x, cells = mk()
    x = x * h
    mat = (E0, 0.0, 0.3, 3.0, 0)
    m = lib.Mesh(cell, k, x, cells, *mat, elem_prec=prec)
    rho = g(5).uniform(0.8, 1.0, len(cells))
    vals = m.assemble_K(torch.as_tensor(rho, device="cuda")).cpu().numpy()
    _, _, v, va, _ = oracle_csr(cell, k, x, cells, mat, rho)
    tol, floor = (TOL64, 1e-15) if prec == "fp64" else (TOL32, 1e-7)
    # (a float pair's own step is 2^-149 for each of a value's contributions, at most 24 here)
    assert np.all(np.abs(vals - v) <= tol * va + floor * va.max() + 24 * 2.0 ** -149)


@pytest.mark.parametrize("rho", [1e-9, 1e-7])
@pytest.mark.parametrize("name", MESHES)
def test_all_moduli_outside_the_pair_range(lib, name, rho):
    """Moduli of 1e-27 and 1e-21: every block is redone in FP64."""
    cell, k, mk = MESHES[name]
    x, cells = mk()
    mat = (1.0, 0.0, 0.3, 3.0, 0)
    m = lib.Mesh(cell, k, x, cells, *mat)
    r = np.full(len(cells), rho)
    vals = m.assemble_K(torch.as_tensor(r, device="cuda")).cpu().numpy()
    _, _, v, va, _ = oracle_csr(cell, k, x, cells, mat, r)
    assert np.all(np.abs(vals - v) <= TOL64 * va + 1e-15 * va.max())
