"""Spectral map, pole sums and QP solve at the depths and spectra where they can go wrong:
warp and block edges of the eigenvalue-per-thread kernel, clustered and ghosted spectra,
graded tridiagonals, against numpy's eigensolver.

Tolerance: the nodes carry a few roundings of ||T||, so with Omega = sqrt(theta) and the
broadening delta a pole's term changes by d Omega / delta = few eps ||T|| / (2 Omega delta)
relative: below 1e-10 for the norms used here (||T|| ~ 1e3, Omega >= 1, delta = 0.05)."""
import numpy as np
import pytest
import torch

import gw_inputs
from paper_2310_20103_gb300 import lgw as L

pytestmark = pytest.mark.gpu




def _tridiagonals(kind, B, k, rng):
    if kind == "random":
        return 500 + 20 * rng.uniform(-1, 1, (B, k)), 240 * rng.uniform(0.9, 1.0, (B, k))
    if kind == "graded":          # off-diagonals that fall by 1e-10 over the depth
        b = 200.0 * 10.0 ** (-10 * np.arange(k) / max(1, k - 1))
        return 700 + 250 * rng.uniform(-1, 1, (B, k)), np.tile(b, (B, 1))
    # "ghost": two weakly coupled copies of one tridiagonal, eigenvalues in close pairs
    a, b = np.zeros((B, k)), np.zeros((B, k))
    h = max(1, k // 2)
    for v in range(B):
        x, y = 500 + 20 * rng.uniform(-1, 1, h), 200 * rng.uniform(0.9, 1.0, h)
        a[v, :h], b[v, :h] = x, y
        if k > h:
            a[v, h:2 * h], b[v, h:2 * h] = x[::-1], np.roll(y[::-1], -1)
            a[v, 2 * h:], b[v, 2 * h:] = 500, 200
            b[v, h - 1] = 1e-7
    return a, b


def _reference(a, b, b0, k_eff, eps, n_v, m_idx, omega, delta, n_t):
    B = a.shape[0]
    n_m = B // n_t
    out = np.zeros((n_t, omega.size), dtype=complex)
    for v in range(B):
        n = int(k_eff[v])
        if n == 0:
            continue
        T = np.diag(a[v, :n]) + np.diag(b[v, : n - 1], 1) + np.diag(b[v, : n - 1], -1)
        th, U = np.linalg.eigh(T)
        Om = np.sqrt(th)
        m = m_idx[v % n_m]
        eta = 1.0 if m < n_v else -1.0
        z = omega - eps[m] - 1j * eta * delta
        w = b0[v] ** 2 * U[0] ** 2 / Om
        out[v // n_m] += (w / (z[:, None] + eta * Om)).sum(1)
    return out


@pytest.mark.parametrize("kind", ["random", "graded", "ghost"])
@pytest.mark.parametrize("k", [1, 2, 7, 8, 9, 31, 32, 33, 63, 200, 255, 256])
def test_poles_against_numpy(kind, k):
    rng = np.random.default_rng(17 * k + len(kind))
    wl = gw_inputs.tiny(k=64)
    n_t, n_m = 2, 5
    B = n_t * n_m
    a, b = _tridiagonals(kind, B, k, rng)
    b0 = rng.uniform(0.1, 0.2, B)
    k_eff = np.full(B, k, dtype=np.int32)
    k_eff[0], k_eff[B - 1] = 0, max(1, k - 1)      # an empty and a shortened recurrence
    dev = torch.device("cuda:0")
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, torch.from_numpy(wl.eps).to(dev),
                                 torch.from_numpy(wl.L).to(dev))
        t, m = wl.targets[:n_t].copy(), np.array([0, 7, 8, 20, 39], dtype=np.int32)
        prob = L.Problem(targets=t, m_idx=m, omega=wl.omega, delta=wl.delta,
                         M=np.zeros((n_t, n_m, wl.n_aux)))
        sig, e, z = np.zeros((n_t, wl.omega.size, 2)), np.zeros(n_t), np.zeros(n_t)
        L.lgw_sigma_from_coeffs(h, s, prob, L.Options(k=k), a, b, b0, k_eff, sig, e, z)
        got = sig[..., 0] + 1j * sig[..., 1]
        ref = _reference(a, b, b0, k_eff, wl.eps, wl.n_v, m, wl.omega, wl.delta, n_t)
        assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()
        # E solves the QP equation of the reference sum, Z is its slope there
        for i in range(n_t):
            d = 1e-5
            x = np.array([e[i], e[i] - d, e[i] + d])
            S = _reference(a, b, b0, k_eff, wl.eps, wl.n_v, m, x, wl.delta, n_t)[i].real
            slope = (S[2] - S[1]) / (2 * d)
            # Newton ends at |dE| <= 1e-10 max(1, |E|)
            assert abs(x[0] - wl.eps[t[i]] - S[0]) <= 1e-9 * max(1.0, abs(x[0])) * abs(1 - slope)
            assert abs(z[i] - 1 / (1 - slope)) <= 1e-4 * max(1.0, abs(z[i]) ** 2)
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)


@pytest.mark.parametrize("n_m", [1, 31, 65, 300])
def test_many_summed_orbitals(n_m):
    """More summed orbitals than the QP cluster has warps, and fewer."""
    rng = np.random.default_rng(n_m)
    wl = gw_inputs.custom(16, 400, 64, 1, n_m, 64, seed=3, k=40)
    k, dev = 40, torch.device("cuda:0")
    a, b = _tridiagonals("random", n_m, k, rng)
    b0 = rng.uniform(0.05, 0.1, n_m)
    k_eff = np.full(n_m, k, dtype=np.int32)
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, torch.from_numpy(wl.eps).to(dev),
                                 torch.from_numpy(wl.L).to(dev))
        prob = L.Problem(targets=wl.targets, m_idx=wl.m_idx, omega=wl.omega, delta=wl.delta,
                         M=wl.M)
        sig, e, z = np.zeros((1, 64, 2)), np.zeros(1), np.zeros(1)
        L.lgw_sigma_from_coeffs(h, s, prob, L.Options(k=k), a, b, b0, k_eff, sig, e, z)
        ref = _reference(a, b, b0, k_eff, wl.eps, wl.n_v, wl.m_idx, wl.omega, wl.delta, 1)
        got = sig[..., 0] + 1j * sig[..., 1]
        assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()
        S = _reference(a, b, b0, k_eff, wl.eps, wl.n_v, wl.m_idx, e, wl.delta, 1)[0].real
        assert abs(e[0] - wl.eps[wl.targets[0]] - S[0]) <= 1e-8
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)
