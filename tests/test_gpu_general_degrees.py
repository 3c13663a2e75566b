"""The general operator's kernel at every degree it is built for (FP64 and FP32, W = 1..9) against the oracle.

All ten terms of eq. (5.45) with coefficients that vary from point to point
(so that no field or coefficient slot can stand for another), anisotropic
elements, one interior face.  Bounds: those of the operator tests, 1e-12 (FP64)
and 2e-5 (FP32, about 1e3 unit roundoffs of the contraction chain) of max|y|.
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


def _problem(W):
    mesh = wl.box_mesh((2, 1, 1), lo=(-1, 0, 0), hi=(1, 1, 0.5), W=W)

    def op(xs, ys, zs):
        x, y, z = wl._grid(xs, ys, zs)
        A = [[-1 - 0.2 * np.cos(x), 0.3 * np.sin(y + z), -0.2 * np.cos(x * z)],
             [0.3 * np.sin(y + z), -2 - 0.1 * y * z, 0.15 * np.cos(x - y)],
             [-0.2 * np.cos(x * z), 0.15 * np.cos(x - y), -1.5 + 0.3 * np.sin(x + z)]]
        return A, [0.4 * np.cos(y), -0.7 * np.sin(x), 0.25 + z], 1.3 + np.sin(x * y)

    one = lambda xs, ys, zs: wl._full(1.0, xs, ys, zs)  # noqa: E731
    return wl.Problem(mesh, [one], [one], op=op)


@pytest.mark.parametrize("W", list(range(1, 10)))
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
def test_general_apply_every_degree(api, W, prec, tol):
    pb = _problem(W)
    disc = Discretisation(pb)
    m = api.Mesh(pb.mesh, n_rhs=1, coef_kind=api.COEF_GENERAL)
    m.set_data(**api.problem_data_arrays(m, pb))
    U = wl.random_dofs(disc.ndof, 3 + W)
    dt = torch.float64 if prec == "fp64" else torch.float32
    u = torch.tensor(U, dtype=dt, device="cuda")
    y = torch.full_like(u, float("nan"))
    m.apply_operator(u, y)
    ref = disc.apply_A(u.double().cpu().numpy())
    assert np.max(np.abs(y.double().cpu().numpy() - ref)) <= tol * np.max(np.abs(ref)), (W, prec)
    m.close()
