"""Spectral map on tridiagonals whose Gauss rule degenerates: coefficients that are not
numbers, and nodes that coincide.

A coefficient of T (or the start norm) that is Inf or NaN makes the vector's self-energy NaN
and the call fail, as the sums over it would in any order.  Coincident nodes share their
weight, so sums over a cluster are those of numpy's eigensolver: few eps ||T|| / (2 Omega
delta) relative, below 1e-10 for the norms used here (||T|| ~ 1e3, Omega >= 1, delta 0.05)."""
import numpy as np
import pytest

import gw_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def L():
    from paper_2310_20103_gb300.build import build
    build()
    from paper_2310_20103_gb300 import lgw
    return lgw


M_IDX = np.array([0, 8, 39], dtype=np.int32)


def _run(L, a, b, b0, raises=None):
    """Two targets of three summed orbitals each; (sigma, E) on the host."""
    wl = gw_inputs.tiny(k=64)
    k = a.shape[1]
    k_eff = np.full(6, k, dtype=np.int32)
    t = wl.targets[:2].copy()
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, torch.from_numpy(wl.eps).to(DEV),
                                 torch.from_numpy(wl.L).to(DEV))
        prob = L.Problem(targets=t, m_idx=M_IDX, omega=wl.omega, delta=wl.delta,
                         M=np.zeros((2, 3, wl.n_aux)))
        sig = torch.zeros(2, wl.omega.size, 2, dtype=torch.float64, device=DEV)
        e = torch.zeros(2, dtype=torch.float64, device=DEV)
        args = [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (a, b, b0, k_eff)]
        if raises is None:
            L.lgw_sigma_from_coeffs(h, s, prob, L.Options(k=k), *args, sig, e)
        else:
            with pytest.raises(L.LgwError) as err:
                L.lgw_sigma_from_coeffs(h, s, prob, L.Options(k=k), *args, sig, e)
            assert raises in str(err.value)
        torch.cuda.synchronize()
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)
    return sig.cpu().numpy(), e.cpu().numpy()


def _random(k):
    rng = np.random.default_rng(k)
    return (500 + 20 * rng.uniform(-1, 1, (6, k)), 240 * rng.uniform(0.9, 1.0, (6, k)),
            rng.uniform(0.1, 0.2, 6))


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["alpha", "beta", "beta0"])
@pytest.mark.parametrize("k", [1, 2, 40, 256])
def test_non_finite_coefficients_end_in_an_error(L, k, where, value):
    a, b, b0 = _random(k)
    clean, e = _run(L, a, b, b0)
    last = k - 1 if where == "alpha" else k - 2
    rows = [0] if where == "beta0" else sorted({0, last // 2, last} if last >= 0 else set())
    for i in rows:
        x = [a.copy(), b.copy(), b0.copy()]
        if where == "beta0":
            x[2][4] = value
        else:
            x[0 if where == "alpha" else 1][4, i] = value
        sig, e2 = _run(L, *x, raises="onverge")
        assert np.isnan(sig[1]).all() and np.isnan(e2[1])
        assert np.array_equal(sig[0], clean[0]) and e2[0] == e[0]


def test_the_unused_last_beta_is_not_read(L):
    """beta_k couples nothing inside T_k: whatever it is, the result is the same."""
    a, b, b0 = _random(40)
    clean = _run(L, a, b, b0)
    b[:, -1] = np.nan
    got = _run(L, a, b, b0)
    assert np.array_equal(got[0], clean[0]) and np.array_equal(got[1], clean[1])


def _reference(a, b, b0, wl):
    out = np.zeros((2, wl.omega.size), dtype=complex)
    for v in range(6):
        k = a.shape[1]
        th, U = np.linalg.eigh(np.diag(a[v]) + np.diag(b[v, :k - 1], 1) + np.diag(b[v, :k - 1], -1))
        m = M_IDX[v % 3]
        eta = 1.0 if m < wl.n_v else -1.0
        z = wl.omega - wl.eps[m] - 1j * eta * wl.delta
        Om = np.sqrt(th)
        out[v // 3] += (b0[v] ** 2 * U[0] ** 2 / Om / (z[:, None] + eta * Om)).sum(1)
    return out


@pytest.mark.parametrize("kind", ["constant", "copies 1e-7", "copies 1e-30", "copies 0",
                                  "one in the middle"])
@pytest.mark.parametrize("m,n", [(2, 9), (3, 11), (4, 25), (7, 36)])
def test_coincident_nodes_share_their_weight(L, kind, m, n):
    """m weakly coupled copies of one n-row tridiagonal: every node m times."""
    wl = gw_inputs.tiny(k=64)
    rng = np.random.default_rng(10 * m + n)
    k = m * n
    a, b, b0 = np.zeros((6, k)), np.zeros((6, k)), rng.uniform(0.1, 0.2, 6)
    for v in range(6):
        if kind == "constant":
            a[v] = 500.0
            continue
        x, y = 500 + 20 * rng.uniform(-1, 1, n), 200 * rng.uniform(0.9, 1.0, n)
        for c in range(m):
            # every second copy upside down, so that the first row meets its image
            a[v, c * n:(c + 1) * n] = x if c % 2 == 0 else x[::-1]
            b[v, c * n:c * n + n - 1] = y[:n - 1] if c % 2 == 0 else y[:n - 1][::-1]
            b[v, (c + 1) * n - 1] = 0.0 if kind == "one in the middle" else float(kind.split()[1])
        if kind == "one in the middle":      # an isolated row at an eigenvalue of the first copy
            a[v, k // 2] = np.linalg.eigvalsh(np.diag(x) + np.diag(y[:n - 1], 1)
                                              + np.diag(y[:n - 1], -1))[n // 2]
            b[v, k // 2 - 1] = b[v, k // 2] = 0.0
    sig, _ = _run(L, a, b, b0)
    ref = _reference(a, b, b0, wl)
    assert np.abs(sig[..., 0] + 1j * sig[..., 1] - ref).max() <= 1e-10 * np.abs(ref).max()
