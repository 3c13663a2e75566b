"""The two FP64 launch shapes of the apply kernels give the same results.

Which one a launch takes depends on the item count (one item per SM or fewer,
more), so the same element block is applied alone and as one of many copies:
the contractions run in the same order in both, so the results are equal bit
for bit.  Degrees with a second shape (2..7) and their neighbours, both
coefficient kinds, 8 elements and enough copies for several items per SM.
"""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1110_2316_gb300 import api as A
    return A


@pytest.mark.parametrize("W", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("coef", ["laplace", "scalar"])
def test_few_and_many_items(api, W, coef):
    copies = 80
    kind = api.COEF_LAPLACE if coef == "laplace" else api.COEF_SCALAR
    one = wl.box_mesh(2, W=W)
    many = wl.concat_meshes([wl.box_mesh(2, W=W) for _ in range(copies)])
    U = wl.random_dofs(8 * (W + 1) ** 3, 11 + W)
    outs = []
    for mesh, k in ((one, 1), (many, copies)):
        m = api.Mesh(mesh, n_rhs=1, coef_kind=kind)
        nq = m.nquad // k
        rng = np.random.default_rng(5)
        f, a, ga = rng.standard_normal(nq), 1 + rng.random(nq), rng.standard_normal((3, nq))
        d = dict(f=np.tile(f, k)[None])
        if coef == "scalar":
            d.update(a=np.tile(a, k), grad_a=np.tile(ga, (1, k)))
        m.set_data(**d)
        u = torch.tensor(np.tile(U, k), device="cuda")
        y = torch.full_like(u, float("nan"))
        m.apply_operator(u, y)
        z = torch.full((1, m.nquad), float("nan"), dtype=torch.float64, device="cuda")
        m.apply_residual(u, z)
        t = torch.full_like(u, float("nan"))
        m.apply_transpose(z, t)
        outs.append([v.reshape(k, -1).cpu().numpy() for v in (y, z, t)])
        m.close()
    for few, lots in zip(*outs):
        assert np.isfinite(few).all()
        assert np.array_equal(lots, np.broadcast_to(few, lots.shape)), (W, coef)
