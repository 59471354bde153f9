"""FP64 products of graded operands: auxiliary functions and pairs of very different scales.

The digits of a sliced product are a fixed point relative to a row's largest element, so what
is graded along the contraction has to be balanced first.  Yardstick: numpy's own FP64
evaluation against extended precision; over all outputs, each relative to the typical
magnitude of the terms it sums, the largest error may be 4 times numpy's (plus 2^-50: digits
of 2^-56 of the largest of a few hundred terms)."""
import numpy as np
import pytest

import gw_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LD = np.longdouble


@pytest.fixture(scope="module")
def L():
    from paper_2310_20103_gb300.build import build
    build()
    from paper_2310_20103_gb300 import lgw
    return lgw


def _factor(n, rng):
    """A lower triangular factor of small integers with 16 on its diagonal: R R^T and every
    step of its Cholesky factorisation are exact in FP64, so that what a fit errs by is the
    product's own."""
    R = np.tril(rng.integers(-3, 4, (n, n)), -1).astype(np.float64)
    np.fill_diagonal(R, 16.0)
    return R


def _fit(L, C, metric):
    B = np.zeros_like(C)
    h = L.lgw_create(0)
    try:
        L.lgw_fit_factors(h, C, metric, B)
    finally:
        L.lgw_destroy(h)
    return B


@pytest.mark.parametrize("order", ["random", "falling", "rising"])
@pytest.mark.parametrize("coeffs", ["inverse", "flat", "same"])
@pytest.mark.parametrize("decades", [0, 8, 12, 16, 24])
@pytest.mark.parametrize("n_pairs,n", [(200, 64), (150, 200)])
def test_fit_factors_of_a_graded_metric(L, n_pairs, n, decades, coeffs, order):
    """metric = D R R^T D, R exact, with `decades` between the diagonal's ends, C as 1 / D (auxiliary
    functions of any normalisation), without, or as D."""
    rng = np.random.default_rng(n + decades)
    u = np.linspace(0, 1, n)
    u = {"random": rng.permutation(u), "falling": u[::-1], "rising": u}[order]
    d = 2.0 ** np.round(0.5 * decades * np.log2(10) * (u - 0.5))
    R = d[:, None] * _factor(n, rng)
    metric = R @ R.T
    C = rng.standard_normal((n_pairs, n)) * {"inverse": 1 / d, "flat": np.ones(n), "same": d}[coeffs]
    B = _fit(L, C, metric)
    ref = C.astype(LD) @ R.astype(LD)
    typical = np.abs(C).mean(0) @ np.abs(R)      # per column of B
    own = np.abs(C @ R - ref) / typical
    err = np.abs(B - ref) / typical
    assert np.isfinite(B).all()
    assert err.max() <= 4 * own.max() + 2.0 ** -50


@pytest.mark.parametrize("n_pairs,n", [(2200, 1024), (80, 4160)])
def test_large_fits_of_a_graded_metric(L, n_pairs, n):
    """Sizes that make the digits beside the factorisation, and rows too long for one block's
    single pass."""
    rng = np.random.default_rng(n)
    d = 2.0 ** rng.integers(-25, 26, n)
    R = d[:, None] * _factor(n, rng)
    C = rng.standard_normal((n_pairs, n)) / d
    B = _fit(L, C, R @ R.T)
    typical = np.abs(C).mean(0) @ np.abs(R)
    rows = np.linspace(0, n_pairs - 1, 12).astype(int)      # the extended products take long
    ref = C[rows].astype(LD) @ R.astype(LD)
    own = np.abs(C[rows] @ R - ref) / typical
    err = np.abs(B[rows] - ref) / typical
    assert err.max() <= 4 * own.max() + 2.0 ** -50
    assert np.abs((B - C @ R) / typical).max() <= 1e-13


def test_fit_factors_of_rows_with_gradings_of_their_own(L):
    """No scale per auxiliary function helps where every pair has its own: pairs on fragment
    a see a's functions at 1 and b's at 1e-12, pairs on b the other way round, and B's columns
    of b's functions come from the small ones."""
    rng = np.random.default_rng(1)
    n, n_pairs = 256, 120
    R = _factor(n, rng)
    R[128:, :128] *= 2.0 ** -20
    C = rng.standard_normal((n_pairs, n))
    C[:60, 128:] *= 1e-12
    C[60:, :128] *= 1e-12
    B = _fit(L, C, R @ R.T)
    ref = C.astype(LD) @ R.astype(LD)
    typical = np.empty_like(C)
    for rows in (slice(0, 60), slice(60, n_pairs)):
        typical[rows] = np.abs(C[rows]).mean(0) @ np.abs(R)
    own = np.abs(C @ R - ref) / typical
    err = np.abs(B - ref) / typical
    assert err.max() <= 4 * own.max() + 2.0 ** -50


def test_fit_factors_of_infinities(L):
    """A row of C with an infinity is not finite where it was not, the other rows are as
    without it."""
    rng = np.random.default_rng(2)
    C = rng.standard_normal((70, 96))
    W = rng.standard_normal((96, 96))
    metric = W @ W.T / 96 + np.eye(96)
    metric = 0.5 * (metric + metric.T)
    clean = _fit(L, C, metric)
    C[5, 95] = np.inf          # meets every column's last row of R
    B = _fit(L, C, metric)
    others = np.arange(70) != 5
    assert np.abs(B[others] - clean[others]).max() <= 1e-13 * np.abs(clean).max()
    assert not np.isfinite(B[5]).any()


@pytest.mark.parametrize("pairs,aux", [(0, 0), (10, 0), (0, 12), (10, 12), (16, 16)])
@pytest.mark.parametrize("x_scale", ["flat", "inverse"])
@pytest.mark.parametrize("n_v,n_c,A", [(8, 32, 96), (13, 80, 130)])
def test_apply_casida_of_a_graded_factor(L, n_v, n_c, A, pairs, aux, x_scale):
    """L = D1 K D2, vectors without grading or as 1 / D1."""
    rng = np.random.default_rng(pairs + aux + A)
    wl = gw_inputs.make_workload("p", n_v, n_c, A, [0], [0], 1, 3)
    N, n_vec = n_v * n_c, 20
    d1 = 10.0 ** (-pairs * rng.uniform(0, 1, N))
    d2 = 10.0 ** (-aux * rng.uniform(0, 1, A))
    Lm = rng.standard_normal((N, A)) * d1[:, None] * d2[None, :]
    X = rng.standard_normal((n_vec, N)) / (d1 if x_scale == "inverse" else 1.0)
    Y = np.zeros_like(X)
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, n_v, n_c, A, torch.from_numpy(wl.eps).to(DEV),
                                 torch.from_numpy(Lm).to(DEV))
        L.lgw_apply_casida(h, s, np.ascontiguousarray(X), Y, "fp64")
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)

    def apply(dt):
        e = wl.eps.astype(dt)
        D = (e[None, n_v:] - e[:n_v, None]).reshape(-1)
        y = (X.astype(dt) * np.sqrt(D)) @ Lm.astype(dt)
        return X.astype(dt) * D ** 2 + dt(4.0) * np.sqrt(D) * (y @ Lm.astype(dt).T), D, y

    ref, D, y = apply(LD)
    own, err = np.abs(apply(np.float64)[0] - ref), np.abs(Y - ref)
    D = D.astype(np.float64)
    # terms of the low-rank part, by their typical size over the vectors
    xt = (np.abs(X) * np.sqrt(D)).mean(0)
    scale = np.abs(X).mean(0) * D ** 2 + 4 * np.sqrt(D) * ((xt @ np.abs(Lm)) @ np.abs(Lm).T)
    assert (err / scale).max() <= 4 * (own / scale).max() + 2.0 ** -50


def test_coupling_vectors_of_a_graded_basis(L):
    """V = L M with auxiliary functions of any normalisation, L's columns as d and M as 1 / d:
    against the FP64 pipe (a handle with a byte limit), within the bounds of the ungraded
    comparison (1e-11 eV for E, 1e-9 of the largest self-energy)."""
    wl = gw_inputs.tiny(k=12)
    d = 10.0 ** (-12 * np.random.default_rng(5).uniform(0, 1, wl.n_aux))
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
    res = []
    for limit in (0, 1 << 40):
        h = L.lgw_create(0)
        try:
            L.lgw_set_workspace_limit(h, limit)
            s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, t(wl.eps), t(wl.L * d), 4.0)
            prob = L.Problem(targets=t(wl.targets), m_idx=t(wl.m_idx), omega=t(wl.omega),
                             delta=wl.delta, M=t(wl.M / d))
            sig = torch.zeros(wl.n_t, wl.omega.size, 2, dtype=torch.float64, device=DEV)
            e = torch.zeros(wl.n_t, dtype=torch.float64, device=DEV)
            L.lgw_sigma_c(h, s, prob, L.Options(k=12, precision="fp64", reorth="cgs2"), sig, e)
            torch.cuda.synchronize()
            res.append((sig.cpu().numpy(), e.cpu().numpy()))
            L.lgw_release_system(s)
        finally:
            L.lgw_destroy(h)
    (s0, e0), (s1, e1) = res
    assert np.abs(s0 - s1).max() <= 1e-9 * np.abs(s1).max()
    assert np.abs(e0 - e1).max() <= 1e-11
