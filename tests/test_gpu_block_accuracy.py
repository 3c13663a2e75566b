"""Accuracy of the FP32 element-block products against the FP64 factor.

The one-pass products (variant 4 at 2 to 31 right-hand sides) took the place of
tiles that are chains of FP32 multiply-adds (variant 3): on the same factor and
right-hand sides their error against the FP64 products (variant 0, a tile that
shares no code with the one-pass kernels) may not be larger.  Norms over all
elements and right-hand sides of four random r; 10 % for what is left of the
sampling noise.
"""
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1110_2316_gb300 import api as a
    return a


def _mesh(api, W, boxes, n_rhs):
    base = wl.varcoef_manufactured(n=boxes, W=W)
    pb = wl.Problem(base.mesh, base.f * n_rhs, base.g * n_rhs, base.a, base.grad_a)
    m = api.Mesh(pb.mesh, n_rhs=n_rhs, coef_kind=api.COEF_SCALAR)
    m.set_data(**api.problem_data_arrays(m, pb))
    m.setup_block_preconditioner()
    m.set_block_tile(W, api.FP64, 0)
    return m


def _errors(api, m, W, r, variants):
    """Relative error against the FP64 products per variant."""
    ref = torch.empty(r.shape, dtype=torch.float64, device="cuda")
    m.apply_preconditioner(r.double(), ref)
    out = {}
    for v in variants:
        m.set_block_tile(W, api.FP32, v)
        z = torch.full_like(r, float("nan"))
        m.apply_preconditioner(r, z)
        out[v] = (z.double() - ref, ref)
    return out


# three elements (a cluster of CTAs per element), and enough of them for a CTA per element
@pytest.mark.parametrize("W,boxes", [(W, (3, 1, 1)) for W in range(1, 11)] + [(4, (10, 8, 5)), (6, (7, 7, 6))])
@pytest.mark.parametrize("n_rhs", [7, 16, 31])
def test_error_no_larger_than_the_tiles(api, W, boxes, n_rhs):
    m = _mesh(api, W, boxes, n_rhs)
    g = torch.Generator(device="cuda").manual_seed(5)
    acc = {3: 0.0, 4: 0.0}
    for _ in range(4):
        r = torch.randn(n_rhs * m.ndof, generator=g, device="cuda")
        for v, (d, ref) in _errors(api, m, W, r, acc).items():
            acc[v] += float(d.norm() / ref.norm()) ** 2
    m.close()
    assert acc[4] ** 0.5 <= 1.1 * acc[3] ** 0.5, (acc[4] / acc[3]) ** 0.5
