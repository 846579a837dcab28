"""The one-call step runs its two parts beside each other: it takes no longer than the
assembly and the sensitivities one after the other (linear cells on FP32 matrices, whose
short sensitivities once ran on so few blocks that they outlasted both)."""
import numpy as np
import pytest
import torch

from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def best(f, reps=10):
    t = []
    for _ in range(6):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        for _ in range(reps):
            f()
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b) / reps)
    return min(t[1:])


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_step_of_linear_triangles(lib, prec):
    x, cells = W.triangle_grid(1200, 600, 0.2, np.random.default_rng(1))
    m = lib.Mesh("tri", 1, x, cells, 1.0, 1e-9, 0.3, 3.0, 0, elem_prec=prec)
    r = torch.full((m.n_cells,), 0.5, dtype=torch.float64, device="cuda")
    u = torch.as_tensor(np.random.default_rng(2).standard_normal(m.ndof), device="cuda")
    vals, dc, c = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (m.nnz, m.n_cells, 1))
    apart = best(lambda: m.assemble_K(r, vals)) + best(lambda: m.sensitivity(r, u, dc, c))
    assert best(lambda: m.step(r, u, vals, dc, c)) <= 1.2 * apart
