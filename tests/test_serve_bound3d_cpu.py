"""The serving admission bound of 3D and of general cells, checked without a GPU: it covers
the arrays of mesh creation as it sizes them on the host -- element matrices, CSR indices,
positions, the block rows' chunk records and streamed blocks (soptx_host_block_tables),
the geometry of the Gauss points -- and is at most twice them (on meshes large enough that
its constants do not count), so that no job throws out meshes that it could share the device
with."""
import numpy as np
import pytest

from paper_2505_02438_gb300 import build, workloads as W

g = np.random.default_rng


@pytest.fixture(scope="module", autouse=True)
def native():
    build.build_library()


def sheared(mesh):
    c, cl = mesh
    return c + 0.01 * c[:, :1] ** 2 * np.array([1.0, 0.0, 0.0]), cl


def delaunay(n):
    spatial = pytest.importorskip("scipy.spatial")
    p = g(0).random((n, 3))
    t = spatial.Delaunay(p).simplices
    e = p[t[:, 1:]] - p[t[:, :1]]
    return p, np.ascontiguousarray(t[np.abs(np.linalg.det(e)) > 1e-9], np.int32)


def shells(n, layers):
    """Rings of n tetrahedra around one axis (n cells and more at a pair)."""
    t = 2 * np.pi * np.arange(n) / n
    x = [np.stack([0 * t, 0 * t, 0 * t], 1)[:1] + [[0, 0, k]] for k in range(layers + 1)]
    ring = np.stack([np.cos(t), np.sin(t), 0 * t], 1)
    x += [ring + [0, 0, k + 0.5] for k in range(layers)]
    base = layers + 1
    cells = [[k, k + 1, base + k * n + j, base + k * n + (j + 1) % n] for k in range(layers) for j in range(n)]
    return np.vstack(x), np.array(cells, np.int32)


MESHES = {
    "tet 1": ("tet", 1, lambda: W.kuhn_tets(20, 14, 12, 0.15, g(1))),
    "tet 2": ("tet", 2, lambda: W.kuhn_tets(14, 8, 7, 0.15, g(2))),
    "tet 3": ("tet", 3, lambda: W.kuhn_tets(8, 5, 4, 0.15, g(3))),
    "tet 1 random": ("tet", 1, lambda: delaunay(4000)),
    "tet 2 random": ("tet", 2, lambda: delaunay(1000)),
    "tet 2 shells of 40": ("tet", 2, lambda: shells(40, 60)),
    "hex 1 distorted": ("hex", 1, lambda: W.hex_grid(24, 16, 14, 0.15, g(4))),
    "hex 2 distorted": ("hex", 2, lambda: W.hex_grid(12, 8, 7, 0.1, g(5))),
    "hex 3 distorted": ("hex", 3, lambda: W.hex_grid(8, 6, 5, 0.1, g(6))),
    "hex 1 sheared": ("hex", 1, lambda: sheared(W.structured_hex(24, 16, 14))),
    "hex 2 sheared": ("hex", 2, lambda: sheared(W.structured_hex(12, 8, 7))),
    "hex 3 sheared": ("hex", 3, lambda: sheared(W.structured_hex(8, 6, 5))),
    "box 1": ("hex", 1, lambda: W.structured_hex(24, 16, 14)),
    "box 2": ("hex", 2, lambda: W.structured_hex(14, 10, 8)),
    "box 3": ("hex", 3, lambda: W.structured_hex(9, 7, 6)),
    "quad 1 distorted": ("quad", 1, lambda: W.quad_grid(150, 100, 0.2, g(7))),
    "quad 2 distorted": ("quad", 2, lambda: W.quad_grid(90, 70, 0.2, g(8))),
    "quad 3 distorted": ("quad", 3, lambda: W.quad_grid(60, 50, 0.2, g(9))),
}


def arrays(cell, k, coords, cells, prec):
    """Bytes of the large device arrays of the mesh."""
    from paper_2505_02438_gb300.api import host_block_tables, host_plan
    pl = host_plan(cell, k, coords, cells)
    d, nc, nb = coords.shape[1], len(cells), pl["nb"]
    own = nc if pl["path"] == "cached" else 1
    esz = 8 if prec == "fp64" else 4
    b = own * (d * nb) ** 2 * esz + 4 * pl["nnz"] + 2 * nc * nb * nb + 25 * nc * nb + 24 * pl["ndof"]
    T = host_block_tables(cell, k, coords, cells, prec)
    if T is not None:
        b += T["table_bytes"]
        b += T["n_rows"] * 32 * 72 if prec == "fp64" and pl["path"] == "cached" else 0
    if cell in ("quad", "hex") and pl["path"] == "cached":
        x = coords[cells] - coords[cells][:, :1]
        corner = np.array([[(v >> m) & 1 for m in range(d)] for v in range(1 << d)])
        affine = np.einsum("vm,emi->evi", corner, x[:, [1 << m for m in range(d)]])
        if np.abs(x - affine).max() > 1e-9:
            b += nc * ((1 << d) * d * 8 + (nb * (d * d + 1) * 8 if prec == "fp64" else 0))
    return b, T


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", MESHES)
def test_bound_is_between_the_arrays_and_twice_them(name, prec):
    from paper_2505_02438_gb300.serve import mesh_bytes_bound
    cell, k, mk = MESHES[name]
    coords, cells = mk()
    bound = mesh_bytes_bound(W.Workload("t", cell, k, coords, cells, elem_prec=prec))
    b, T = arrays(cell, k, coords, cells, prec)
    assert bound >= b
    # (a box of order 1 has no tables if its numbering makes it a lattice, which the bound
    # does not look at)
    assert bound <= (3 if name == "box 1" else 2) * b + 4 * 2 ** 20, (bound / b, T)
    # no tables: FP32 matrices of distorted cells, and of order 3, whose integrals fill the shared memory
    if name[:3] in ("tet", "hex") and not (prec == "fp32" and name in ("hex 1 distorted", "hex 2 distorted",
                                                                      "hex 3 distorted", "hex 3 sheared")):
        assert T is not None and T["n_chunks"] > 0


def test_large_job_leaves_room():
    """The benchmark's P2 tetrahedra: the bound is far below the 14 GB that it once was."""
    from paper_2505_02438_gb300.serve import mesh_bytes_bound
    coords, cells = W.kuhn_tets(60, 20, 20, 0.15, g(1))
    assert mesh_bytes_bound(W.Workload("t", "tet", 2, coords, cells, elem_prec="fp64")) < 4.5e9
