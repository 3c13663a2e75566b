"""Residual map at every degree, against the oracle (FP64) and the FP64 result (FP32).

FP64: 1e-12 of max|z| (the operator tests' bound) against the oracle's
sqrt(w J)(L u - f) element by element.  FP32: 2e-5 of max|z| against FP64 (about
1e3 unit roundoffs of the contraction chain).  Two right-hand sides, both
coefficient kinds.  (The transpose: test_gpu_adjoint.py, test_gpu_ibp.py.)
"""
import numpy as np
import pytest
import torch

import workloads as wl
from oracle.functional import Discretisation

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1110_2316_gb300 import api as A
    return A


@pytest.mark.parametrize("W", list(range(1, 11)))
@pytest.mark.parametrize("coef", ["laplace", "scalar"])
def test_residual_map_every_degree(api, W, coef):
    if coef == "scalar":
        base = wl.varcoef_manufactured(n=(2, 1, 1), W=W)
        pb = wl.Problem(base.mesh, base.f * 2, base.g * 2, base.a, base.grad_a)
        kind = api.COEF_SCALAR
    else:
        base = wl.laplace_sinh(n=(1, 2, 1), W=W)
        pb = wl.Problem(base.mesh, base.f * 2, base.g * 2)
        kind = api.COEF_LAPLACE
    disc = Discretisation(pb)
    m = api.Mesh(pb.mesh, n_rhs=2, coef_kind=kind)
    m.set_data(**api.problem_data_arrays(m, pb))
    U = wl.random_dofs(2 * disc.ndof, 40 + W)
    u = torch.tensor(U, device="cuda")
    z = torch.full((2, m.nquad), float("nan"), dtype=torch.float64, device="cuda")
    m.apply_residual(u, z)
    for r in range(2):
        ref = np.concatenate([(np.sqrt(disc.vol_weight(e)) * (
            disc.L_apply(disc.block(U[r * disc.ndof:(r + 1) * disc.ndof], e), e) - disc.f_at(e, r))).ravel()
            for e in range(disc.E)])
        assert np.max(np.abs(z[r].cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref)), (W, coef, r)
    z32 = torch.full((2, m.nquad), float("nan"), dtype=torch.float32, device="cuda")
    m.apply_residual(u.float(), z32)
    m.apply_residual(u.float().double(), z)
    assert float((z32.double() - z).abs().max()) <= 2e-5 * float(z.abs().max()), (W, coef)
    m.close()
