"""Accuracy of the FP32 element-block products against the FP64 factor.

The one-pass products (variant 4 at 2 to 31 right-hand sides) took the place of
tiles that are chains of FP32 multiply-adds (variant 3): on the same factor and
right-hand sides their error against the FP64 products (variant 0, a tile that
shares no code with the one-pass kernels) may not be larger.  Norms over all
elements and right-hand sides of four random r; 10 % for what is left of the
sampling noise.

The factor and the products also stand against the operator itself: on a mesh of
one element A is its own block, read here from applies to unit vectors, with
X = L^{-1} of A = L L^T formed by torch in FP64.
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


def _one_element(api, W, n_rhs):
    """A mesh of one element, its A and X = L^{-1} (FP64)."""
    m = _mesh(api, W, (1, 1, 1), n_rhs)
    n = (W + 1) ** 3
    A = torch.empty(n, n, dtype=torch.float64, device="cuda")
    u = torch.zeros(n_rhs, n, dtype=torch.float64, device="cuda")
    y = torch.empty_like(u)
    for j in range(0, n, n_rhs):
        u.zero_()
        c = min(n_rhs, n - j)
        u[torch.arange(c), j + torch.arange(c)] = 1.0
        m.apply_operator(u, y)
        A[j:j + c] = y[:c]
    A = 0.5 * (A + A.T)
    L = torch.linalg.cholesky(A)
    return m, A, torch.linalg.solve_triangular(L, torch.eye(n, dtype=torch.float64, device="cuda"), upper=False)


@pytest.mark.parametrize("W", list(range(1, 11)))
@pytest.mark.parametrize("n_rhs", [1, 2, 5, 9, 31])
def test_fp64_products(api, W, n_rhs):
    # one-pass variant and tile against X^T X r: n eps bounds each of the two sums, the factor
    # 4 n eps cond(A); against each other (the same factor) 2 n eps |X|^T |X| |r| each
    m, A, X = _one_element(api, W, n_rhs)
    n, eps = A.shape[0], 2.0 ** -53
    ev = torch.linalg.eigvalsh(A)
    g = torch.Generator(device="cuda").manual_seed(8)
    r = torch.randn(n_rhs, n, dtype=torch.float64, generator=g, device="cuda")
    ref = r @ X.T @ X
    sums = 2 * n * eps * ((r.abs() @ X.abs().T) @ X.abs()).norm(dim=1)
    z = {}
    for v in ((5, 7) if n_rhs == 1 else (3, 0)):
        m.set_block_tile(W, api.FP64, v)
        z[v] = torch.full_like(r, float("nan"))
        m.apply_preconditioner(r, z[v])
        bound = sums + 4 * n * eps * float(ev[-1] / ev[0]) * ref.norm(dim=1)
        assert bool(((z[v] - ref).norm(dim=1) <= bound).all()), v
    a, b = z.values()
    assert bool(((a - b).norm(dim=1) <= 2 * sums).all())
    m.close()


def _tf32(v):
    return ((v.view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32)


@pytest.mark.parametrize("W", list(range(4, 11)))
@pytest.mark.parametrize("n_rhs", [1, 4, 8, 16, 31, 40])
def test_fp32_parts_are_kept(api, W, n_rhs):
    # against 64-bit products of the FP32 factor: one TF32 part per operand (up to 2^-11 of each entry)
    # must be at least 64 times as far off as any variant (FP32 sums: 2^-24 of growing partial
    # sums, at most sqrt(n) = 36 of them in effect), 4 times for the long sums on the tensor
    # cores (variant 8); a product that drops a part of an operand comes within 2
    from paper_1110_2316_gb300._lib import HpseError
    m, _, X = _one_element(api, W, n_rhs)
    X = X.float()
    g = torch.Generator(device="cuda").manual_seed(9)
    r = torch.randn(n_rhs, X.shape[0], generator=g, device="cuda")
    ref = r.double() @ X.double().T @ X.double()
    t = _tf32(r).double() @ _tf32(X).double().T
    tf32 = float((_tf32(t.float()).double() @ _tf32(X).double() - ref).norm() / ref.norm())
    seen = []
    for v in range(9):
        try:
            m.set_block_tile(W, api.FP32, v)
        except HpseError:
            continue
        z = torch.full_like(r, float("nan"))
        m.apply_preconditioner(r, z)
        err = float((z.double() - ref).norm() / ref.norm())
        assert err <= tf32 / (4 if v == 8 else 64), (v, err, tf32)
        seen.append(v)
    assert seen == [0, 1, 2, 3, 4, 5, 6, 7] + ([8] if n_rhs >= 32 else [])
    m.close()
