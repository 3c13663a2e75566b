"""One-pass products of the element-block preconditioner (bj_pass.cuh, bj_mma.cuh) against the dense block.

Block sizes from one ragged 16-row block (W = 1, n = 8) to the largest
(W = 10, n = 1331), right-hand-side counts at the edges of the tiles (1, 4, 8,
16 per CTA) and three elements (the row blocks shared by a cluster).  The
dense inverse comes from the FP64 application to every unit vector; with
X = L^{-1} of its inverse the products' rounding is bounded, per element and
right-hand side, by 2 n eps |X|^T (|X| |r|) (two sums of at most n terms; the
FP32 factor's own rounding is one eps of |X| in each).
"""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1110_2316_gb300 import api as a
    return a


@pytest.mark.parametrize("W", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10])
@pytest.mark.parametrize("n_rhs", [1, 4, 7, 9, 31])
def test_one_pass_products(api, W, n_rhs):
    base = wl.varcoef_manufactured(n=(3, 1, 1), W=W)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    n, E = (W + 1) ** 3, 3
    # FP64 inverse blocks, column by column (a tile of k_bj_tri: variant 7 for one right-hand side)
    if n_rhs == 1:
        m.set_block_tile(W, api.FP64, 7)
    inv = torch.zeros(E, n, n, dtype=torch.float64, device="cuda")
    r = torch.zeros(n_rhs, E, n, dtype=torch.float64, device="cuda")
    z = torch.empty_like(r)
    for j0 in range(0, n, n_rhs):
        r.zero_()
        c = min(n_rhs, n - j0)
        for q in range(c):
            r[q, :, j0 + q] = 1.0
        m.apply_preconditioner(r, z)
        inv[:, :, j0:j0 + c] = z[:c].permute(1, 2, 0)
    inv = 0.5 * (inv + inv.transpose(1, 2))
    X = torch.linalg.inv(torch.linalg.cholesky(torch.linalg.inv(inv)))
    for prec, dt, eps, variant in ((api.FP64, torch.float64, 2.0 ** -53, 5 if n_rhs == 1 else 3),
                                   (api.FP32, torch.float32, 2.0 ** -24, 6 if n_rhs == 1 else 4)):
        m.set_block_tile(W, prec, variant)
        r = torch.tensor(wl.random_dofs(n_rhs * m.ndof, 5), dtype=dt, device="cuda")
        z = torch.full_like(r, float("nan"))
        m.apply_preconditioner(r, z)
        R, Z = (v.double().reshape(n_rhs, E, n).permute(1, 2, 0) for v in (r, z))
        ref = X.transpose(1, 2) @ (X @ R)
        bound = 2 * n * eps * (X.abs().transpose(1, 2) @ (X.abs() @ R.abs())).norm(dim=1)
        # the reference itself carries the FP64 rounding of the inverse it was formed from
        slack = 0.0 if prec == api.FP32 else 4 * n * 2.0 ** -53 * float(torch.linalg.cond(X).max()) ** 2
        err = (Z - ref).norm(dim=1)
        assert bool((err <= bound + slack * ref.norm(dim=1)).all()), (W, n_rhs, prec, float((err / bound).max()))
    m.close()
