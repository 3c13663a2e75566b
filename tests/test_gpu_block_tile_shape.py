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
