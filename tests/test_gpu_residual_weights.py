"""Rounding of the residual map's weights: z = sqrt(w J) (L u - f) at u = 0.

There L u is zero exactly, so z = -sqrt(w J) f takes one rounding of sqrt(w J),
one of f (FP32; FP64 holds it exactly) and one of the product: at most 3 units
in FP32 and 2 in FP64 (u = 2^-24, 2^-53), point by point, against the product
in long doubles.  Every degree, both coefficient kinds, elements of unequal
sides (their Jacobian is no power of two).
"""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", list(range(1, 11)))
@pytest.mark.parametrize("kind", ["laplace", "scalar"])
def test_residual_weights(W, kind):
    from paper_1110_2316_gb300 import api
    pb = wl.varcoef_manufactured(n=(3, 1, 2), W=W)
    scalar = kind == "scalar"
    m = api.Mesh(pb.mesh, n_rhs=1, coef_kind=api.COEF_SCALAR if scalar else api.COEF_LAPLACE)
    d = api.problem_data_arrays(m, pb)
    rng = np.random.default_rng(100 + W)
    f = rng.standard_normal(m.nquad)
    m.set_data(f=f, g=d["g"], **({k: d[k] for k in ("a", "grad_a")} if scalar else {}))
    w = torch.empty(m.nquad, dtype=torch.float64, device="cuda")
    m.quad_weights(w)
    ref = -np.sqrt(w.cpu().numpy().astype(np.longdouble)) * f.astype(np.longdouble)
    for dt, unit, most in ((torch.float32, 2.0 ** -24, 3.0), (torch.float64, 2.0 ** -53, 2.0)):
        u = torch.zeros(m.ndof, dtype=dt, device="cuda")
        z = torch.empty(m.nquad, dtype=dt, device="cuda")
        m.apply_residual(u, z)
        err = np.abs(z.cpu().numpy().astype(np.longdouble) - ref) / np.abs(ref)
        assert float(err.max()) <= most * unit * (1 + 4 * unit), (W, kind, dt, float(err.max()) / unit)
    m.close()
