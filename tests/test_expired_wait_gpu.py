"""A wait inside the block-row kernel that runs out (its limit set to none): the kernel
returns, the next call on the mesh reports it once, and the mesh works again."""
import numpy as np
import pytest
import torch

from paper_2505_02438_gb300 import workloads as W

pytestmark = pytest.mark.gpu

g = np.random.default_rng
MESHES = {"stream": ("tet", 2, lambda: W.kuhn_tets(9, 7, 6, 0.15, g(1)), "fp64"),
          "contract": ("tet", 2, lambda: W.kuhn_tets(9, 7, 6, 0.15, g(1)), "fp32"),
          "pairs": ("hex", 2, lambda: W.structured_hex(7, 6, 5), "fp64")}


@pytest.mark.parametrize("route", MESHES)
def test_reported_by_the_next_call(lib, route):
    from paper_2505_02438_gb300 import _native as N
    cell, k, mk, prec = MESHES[route]
    x, cells = mk()
    m = lib.Mesh(cell, k, x, cells, elem_prec=prec)
    assert m.routes["assembly"] == route
    t = lambda a: torch.as_tensor(a, device="cuda")
    rho, u = t(g(2).uniform(0.1, 1.0, len(cells))), t(g(3).standard_normal(m.ndof))
    want = m.step(rho, u)
    fixed = torch.zeros(m.ndof, dtype=torch.bool, device="cuda")
    fixed[:9] = True
    gout = torch.ones(1, dtype=torch.float64, device="cuda")
    calls = {"assemble": lambda: m.assemble_K(rho), "sensitivity": lambda: m.sensitivity(rho, u),
             "step": lambda: m.step(rho, u), "vjp": lambda: m.compliance_vjp(rho, u, gout),
             "spmv": lambda: m.spmv(want[0], u),
             "step_host": lambda: m.step_host(rho.cpu().pin_memory(), u.cpu().pin_memory())}
    for name, call in calls.items():
        N.lib().soptx_debug_mesh_wait_tries(m._h, 0)
        m.step(rho, u)                   # gives up; nothing has been waited for, so it cannot say so yet
        torch.cuda.synchronize()
        N.lib().soptx_debug_mesh_wait_tries(m._h, -1)
        with pytest.raises(N.SoptxError, match="incomplete") as e:
            call()
        assert e.value.code == 3
        got = m.step(rho, u)             # reported once, the counters are back at zero
        assert all(torch.equal(a, b) for a, b in zip(got, want)), name
    # the solve waits for the stream first, so it reports an assembly just before it
    N.lib().soptx_debug_mesh_wait_tries(m._h, 0)
    vals = m.assemble_K(rho, vals=want[0].clone())
    N.lib().soptx_debug_mesh_wait_tries(m._h, -1)
    with pytest.raises(N.SoptxError, match="incomplete"):
        m.solve(vals, fixed, u, max_iter=10)
    torch.cuda.synchronize()
    assert torch.equal(m.assemble_K(rho), want[0])
