"""Expired device waits of the element-block products (hpse_set_block_wait).

The one-pass variants wait for their copies, the tensor-core one for its matrix
instructions; every wait is bounded.  With a limit of 0 polls the first wait of
every CTA gives up at once (what is in flight still lands before the CTA ends):
z is NaN throughout, the next application and solve report it, the solve in
which it happens reports it, and a new set-up keeps to the variants without
waits and works.
"""
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CUDA = 7  # HPSE_ERR_CUDA


def _waits(prec, v, api):
    return v in ((2, 4, 6, 8) if prec == api.FP32 else (3, 5))


# one element row (clusters of CTAs per element) and 6^3 elements (a CTA per element)
@pytest.mark.parametrize("W,boxes", [(1, (3, 1, 1)), (3, (3, 1, 1)), (5, (3, 1, 1)), (4, (6, 6, 6))])
@pytest.mark.parametrize("n_rhs", [1, 4, 8, 16, 40])
def test_expired_wait(W, boxes, n_rhs):
    from paper_1110_2316_gb300 import api
    from paper_1110_2316_gb300._lib import HpseError
    base = wl.varcoef_manufactured(n=boxes, W=W)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    x = torch.zeros(n_rhs * m.ndof, dtype=torch.float64, device="cuda")
    for prec, dt, tol in ((api.FP64, torch.float64, 1e-12), (api.FP32, torch.float32, 1e-4)):
        m.setup_block_preconditioner()
        r = torch.tensor(wl.random_dofs(n_rhs * m.ndof, 3), dtype=dt, device="cuda")
        z0, z = torch.empty_like(r), torch.empty_like(r)
        m.apply_preconditioner(r, z0)
        for v in range(9):
            try:
                m.set_block_tile(W, prec, v)
            except HpseError:
                continue
            m.set_block_wait(0)
            m.apply_preconditioner(r, z)  # asynchronous: it cannot know yet
            torch.cuda.synchronize()
            if not _waits(prec, v, api):
                assert float((z - z0).abs().max()) <= tol * float(z0.abs().max())
                continue
            assert bool(torch.isnan(z).all()), (prec, v)
            for call in (lambda: m.apply_preconditioner(r, z), lambda: m.pcg_solve(x, prec=prec)):
                with pytest.raises(HpseError) as ei:
                    call()
                assert ei.value.status == CUDA
            # the set-up drops what gives up and clears the report
            m.setup_block_preconditioner()
            assert not _waits(api.FP64, m.block_tile(W, api.FP64)[0], api)
            assert not _waits(api.FP32, m.block_tile(W, api.FP32)[0], api)
            m.apply_preconditioner(r, z)
            assert float((z - z0).abs().max()) <= tol * float(z0.abs().max())
            # the solve in which it happens
            m.set_block_tile(W, prec, v)
            rep = m.pcg_solve(x, tol=1e-8, prec=prec, max_iter=64, raise_on_error=False)
            assert rep["status"] == CUDA, rep
            m.set_block_wait(2 ** 22)
            m.setup_block_preconditioner()
    m.apply_preconditioner(r, z)
    assert float((z - z0).abs().max()) <= tol * float(z0.abs().max())
    x.zero_()
    rep = m.pcg_solve(x, tol=1e-8, prec=api.FP32, max_iter=20000)
    assert rep["status"] == 0 and rep["rel_residual"] <= 1e-8
    m.close()


def test_limit_range():
    from paper_1110_2316_gb300 import api
    from paper_1110_2316_gb300._lib import HpseError
    pb = wl.poisson_sine(n=1, W=2)
    m = api.Mesh(pb.mesh, n_rhs=1, coef_kind=api.COEF_LAPLACE)
    for bad in (-1, 2 ** 22 + 1):
        with pytest.raises(HpseError) as ei:
            m.set_block_wait(bad)
        assert ei.value.status == 1
    m.close()
