"""hpse_block_tile reports what a CTA works on: a tile, or for the one-pass variants the whole block."""
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,n_rhs,f32,f64", [(3, 1, 1, 1), (3, 4, 4, 4), (5, 16, 4, 8), (6, 8, 8, 8), (6, 9, 16, 8),
                                             (10, 5, 8, 4)])
def test_tile_of_the_variants(W, n_rhs, f32, f64):
    from paper_1110_2316_gb300 import api
    base = wl.varcoef_manufactured(n=(1, 1, 1), W=W)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    for prec, v, rhs in ((api.FP32, 6 if n_rhs == 1 else 4, f32), (api.FP64, 5 if n_rhs == 1 else 3, f64)):
        m.set_block_tile(W, prec, v)
        assert m.block_tile(W, prec)[:2] == (v, ((W + 1) ** 3, rhs))
        m.set_block_tile(W, prec, 0)
        assert m.block_tile(W, prec)[:2] == (0, (64, 64))
    m.close()


@pytest.mark.parametrize("boxes,n_rhs,offered", [((5, 4, 4), 9, True), ((5, 4, 4), 8, False), ((2, 2, 2), 9, False),
                                                 ((2, 1, 1), 1, True)])
def test_fp64_tiles_beside_the_pass(boxes, n_rhs, offered):
    # many large blocks can be faster as tiles in FP64 (128 rows x 8 right-hand sides, 128 x 1):
    # they are timed there, and give the products of the one-pass variant to 1e-10 of the norm
    # (n eps = 8e-14 per sum, times the cancellation of X^T X against |X|^T |X|, below 1e3)
    from paper_1110_2316_gb300 import api
    base = wl.varcoef_manufactured(n=boxes, W=8)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    v, one_pass, shape = (6, 5, (128, 1)) if n_rhs == 1 else (4, 3, (128, 8))
    assert (m.block_tile(8, api.FP64)[2][v] > 0) == offered
    r = torch.tensor(wl.random_dofs(n_rhs * m.ndof, 4), device="cuda")
    z = {}
    for k in (v, one_pass):
        m.set_block_tile(8, api.FP64, k)
        z[k] = torch.full_like(r, float("nan"))
        m.apply_preconditioner(r, z[k])
    assert float((z[v] - z[one_pass]).norm()) <= 1e-10 * float(z[one_pass].norm())
    m.set_block_tile(8, api.FP64, v)
    assert m.block_tile(8, api.FP64)[:2] == (v, shape)
    m.close()
