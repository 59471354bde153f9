"""The blocked Cholesky of lgw_fit_factors (csrc/k_static.cu) around its block (64) and panel
(8) edges, and at pivots whose square root leaves the range of the quick form.

With C the identity B is R itself.  Bound: |A - R R^T| <= (n + 1) u |R| |R^T| elementwise for
any order of the sums (u = 2^-53), the square roots and divisions here each within two units
instead of half, so 4 (n + 4) u sqrt(a_ii a_jj); the product with the identity adds a unit of
R's largest element in the column, inside the same factor."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def L():
    from paper_2310_20103_gb300.build import build
    build()
    from paper_2310_20103_gb300 import lgw
    return lgw


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -480, 2.0 ** 480])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 63, 64, 65, 72, 127, 129, 200])
def test_factor_reproduces_the_metric(L, n, scale):
    g = torch.Generator(device=DEV).manual_seed(n)
    X = torch.randn(n, n + 3, generator=g, device=DEV, dtype=torch.float64)
    A = X @ X.T / n + 0.1 * torch.eye(n, device=DEV, dtype=torch.float64)
    A = 0.5 * (A + A.T)
    A = A * scale * scale            # pivots near 2^-960 and 2^960: exact scalings
    B = torch.zeros(n, n, device=DEV, dtype=torch.float64)
    h = L.lgw_create(0)
    L.lgw_fit_factors(h, torch.eye(n, device=DEV, dtype=torch.float64), A.contiguous(), B)
    torch.cuda.synchronize()
    L.lgw_destroy(h)
    R = (B / scale).cpu().numpy().astype(np.longdouble)
    ref = (A / scale / scale).cpu().numpy().astype(np.longdouble)
    d = np.sqrt(np.diag(ref))
    assert np.abs(np.triu(B.cpu().numpy(), 1)).max(initial=0.0) == 0.0
    assert np.abs(R @ R.T - ref).max() <= 4 * (n + 4) * 2.0 ** -53 * np.outer(d, d).max()
