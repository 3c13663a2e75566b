"""Set-up of the element blocks: the unit-vector columns of the operator kernel (MODE_PROBE).

On a mesh of one element A is its own diagonal block, so the FP64 block
preconditioner inverts it.  With A from the plain applies to every unit vector
(an independent path), n eps bounds the relative rounding of its entries, of
the factor and of each product, so that z = M^{-1} A u differs from u by at
most 4 n eps cond(A) |u|.
"""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10])
@pytest.mark.parametrize("kind", ["laplace", "scalar"])
def test_block_of_one_element(kind, W):
    from paper_1110_2316_gb300 import api
    pb = wl.laplace_sinh(n=1, W=W) if kind == "laplace" else wl.varcoef_manufactured(n=(1, 1, 1), W=W)
    n = (W + 1) ** 3
    m = api.Mesh(pb.mesh, n_rhs=1, coef_kind=api.COEF_SCALAR if pb.a is not None else api.COEF_LAPLACE)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    A = torch.empty(n, n, dtype=torch.float64, device="cuda")
    u = torch.zeros(n, dtype=torch.float64, device="cuda")
    for j in range(n):
        u.zero_()
        u[j] = 1.0
        m.apply_operator(u, A[j])
    ev = torch.linalg.eigvalsh(0.5 * (A + A.T))
    cond = float(ev[-1] / ev[0])
    u = torch.tensor(wl.random_dofs(n, 3), device="cuda")
    z = torch.empty_like(u)
    m.apply_preconditioner(A @ u, z)
    bound = 4 * n * 2.0 ** -53 * cond
    assert float((z - u).norm()) <= bound * float(u.norm())
    m.close()
