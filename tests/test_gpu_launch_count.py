"""hpse_kernel_launch_count of the block products: one launch per degree group for the one-pass variants, two otherwise."""
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rhs", [1, 5, 40])
def test_launches_of_an_application(n_rhs):
    from paper_1110_2316_gb300 import api
    from paper_1110_2316_gb300._lib import HpseError
    base = wl.varcoef_manufactured(n=(2, 1, 1), W=3)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    for prec, dt, one_pass in ((api.FP64, torch.float64, (3, 5)), (api.FP32, torch.float32, (2, 4, 6))):
        r = torch.tensor(wl.random_dofs(n_rhs * m.ndof, 3), dtype=dt, device="cuda")
        z = torch.empty_like(r)
        for v in range(9):
            try:
                m.set_block_tile(3, prec, v)
            except HpseError:
                continue
            api.kernel_launch_count(reset=True)
            m.apply_preconditioner(r, z)
            assert api.kernel_launch_count() == (1 if v in one_pass else 2), (prec, v)
    m.close()
