"""Non-finite entries in the element-block preconditioner: z = X^T (X r).

X^T X has no zero structure to rely on (row n - 1 of X reaches every column), so
a NaN or an infinity anywhere in an element's r makes that element's whole z
non-finite, for that right-hand side and no other: the other right-hand sides
and elements keep their values, bit for bit.  NaN comes in the bit patterns of
GPU arithmetic (0x7fffffff), of its negative and of the host (0x7fc00000); the
splits into TF32 parts work on those bits.
"""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PATTERNS = (0x7FFFFFFF, 0xFFFFFFFF, 0x7FC00000, 0x7F800000, 0xFF800000)


@pytest.mark.parametrize("n_rhs", [1, 4, 8, 31, 33, 64])
@pytest.mark.parametrize("W", [1, 3, 5, 6])
def test_nonfinite_entry_reaches_its_block(W, n_rhs):
    from paper_1110_2316_gb300 import api
    from paper_1110_2316_gb300._lib import HpseError
    base = wl.varcoef_manufactured(n=(2, 1, 1), W=W)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    n, k = (W + 1) ** 3, n_rhs // 2
    for prec, dt in ((api.FP32, torch.float32), (api.FP64, torch.float64)):
        for v in range(9):
            try:
                m.set_block_tile(W, prec, v)
            except HpseError:
                continue  # a variant that does not exist here
            clean = torch.tensor(wl.random_dofs(n_rhs * m.ndof, 5), dtype=dt, device="cuda")
            z0 = torch.empty_like(clean)
            m.apply_preconditioner(clean, z0)
            assert torch.isfinite(z0).all()
            for bits in PATTERNS:
                for at in (0, n // 3, n - 1):
                    r, z = clean.clone(), torch.empty_like(clean)
                    bad = torch.from_numpy(np.array([bits], dtype=np.uint32).view(np.int32)).view(torch.float32)
                    if prec == api.FP32:  # the pattern itself
                        r.view(torch.int32)[k * m.ndof + n + at] = int(bad.view(torch.int32)[0])
                    else:
                        r[k * m.ndof + n + at] = float(bad[0])
                    m.apply_preconditioner(r, z)
                    z, want = z.view(n_rhs, 2, n), z0.clone().view(n_rhs, 2, n)
                    assert not torch.isfinite(z[k, 1]).any(), (prec, v, hex(bits), at)
                    z[k, 1] = want[k, 1] = 0.0
                    assert torch.equal(z, want), (prec, v, hex(bits), at)
    m.close()
