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
