"""The step of a small box lattice in one launch of two clusters (lattice.cu): K, dc
and c bitwise those of the separate assembly and sensitivity calls, on one cell, rows,
ragged chunks, both sides of the node count where its CTAs widen and of the largest
sizes it serves, with moduli outside the float-pair range, and replayed in a graph."""
import numpy as np
import pytest
import torch

from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MAT = (1.0, 0.0, 0.3, 3.0, 0)
SHAPES = [(1, 1), (1, 9), (7, 1), (15, 23), (31, 11), (16, 23), (60, 20), (48, 32), (53, 29), (1536, 1),
          (1, 1, 1), (2, 3, 1), (8, 8, 8), (16, 8, 8), (1, 1, 1024), (5, 41, 5)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_step_is_bitwise_the_separate_calls(lib, shape):
    d = len(shape)
    x, cells = W.structured_quad(*shape) if d == 2 else W.structured_hex(*shape)
    m = lib.Mesh("quad" if d == 2 else "hex", 1, x, cells, *MAT)
    assert m.path == "lattice"
    g = np.random.default_rng(sum(shape))
    rho = g.uniform(0.001, 1.0, m.n_cells)
    u = torch.as_tensor(g.standard_normal(m.ndof + 1), device="cuda")[1:]   # off 16-byte alignment
    graph = torch.cuda.CUDAGraph()
    for bad in (False, True):
        if bad:   # moduli of 1e-27 and zero
            rho[::5], rho[1::7] = 1e-9, 0.0
        r = torch.as_tensor(rho, device="cuda")
        vals, dc, c = m.step(r, u)
        want = m.assemble_K(r), *m.sensitivity(r, u)
        assert all(torch.equal(a, b) for a, b in zip((vals, dc, c), want))
    with torch.cuda.graph(graph):
        out = m.step(r, u)
    for t in out:
        t.fill_(float("nan"))
    graph.replay()
    assert all(torch.equal(a, b) for a, b in zip(out, want))
