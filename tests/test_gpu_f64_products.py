"""FP64 products on the tensor cores: C X = Delta^2 X + c_K Delta^1/2 L (L^T (Delta^1/2 X))
through lgw_apply_casida, B = C chol(metric) through lgw_fit_factors, against extended
precision (numpy longdouble), at the sizes where tiles, K blocks, 1024-term chunks and
digits can go wrong.

Tolerances.  An FP64 dot product of K terms errs by a few 2^-53 of its terms' root sum of
squares times sqrt(K); eight 7-bit digits resolve 2^-56 of a row's largest element, which
for these distributions (largest element at most 10 times the root mean square, or sums
carried by the largest elements) stays below that.  So over all outputs of a case the root
mean square error may be at most 4 times that of numpy's own FP64 evaluation of the same
formula, and no output may be further off than the a-priori bound of the digits."""
import numpy as np
import pytest
import torch

import gw_inputs
from paper_2310_20103_gb300 import lgw as L

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _case(n_v, n_c, A, n_vec, kind, seed):
    rng = np.random.default_rng(seed)
    wl = gw_inputs.make_workload("p", n_v, n_c, A, [0], [0], 1, seed)
    N = n_v * n_c
    Lm, X = wl.L.copy(), rng.standard_normal((n_vec, N))
    if kind == "wide":        # twelve decades within each vector and each row of L
        X *= 10.0 ** rng.uniform(-12, 0, X.shape)
        Lm *= 10.0 ** rng.uniform(-6, 0, Lm.shape)
    elif kind == "coherent":  # every product positive, no cancellation, all digits alike
        X = np.full_like(X, 1.0 / 3.0)
        Lm = np.full_like(Lm, 0.7)
    elif kind == "spike":     # one element carries a vector, zero rows and columns
        X *= 1e-9
        X[:, N // 2] = 1.0
        Lm[:, 0] = 0.0
        Lm[N - 1] = 0.0
    elif kind == "tiny":      # far from 1, so the row scales must be carried exactly
        X *= 1e-120
        Lm *= 1e-60
    return wl.eps, Lm, X


def _apply(eps, n_v, Lm, X, dt):
    e = eps.astype(dt)
    D = (e[None, n_v:] - e[:n_v, None]).reshape(-1)
    d = np.sqrt(D)
    Lx = Lm.astype(dt)
    y = (X.astype(dt) * d) @ Lx
    return X.astype(dt) * D ** 2 + dt(4.0) * d * (y @ Lx.T), D, d, y


@pytest.mark.parametrize("kind", ["normal", "wide", "coherent", "spike", "tiny"])
@pytest.mark.parametrize("n_v,n_c,A,n_vec", [
    (3, 37, 20, 1),        # one K block short, one vector
    (8, 32, 128, 16),      # exact tiles
    (13, 80, 130, 17),     # K just over 1024, A just over a tile
    (16, 65, 64, 33),
    (24, 100, 200, 65),    # three chunks, a second column tile
    (8, 64, 1100, 40),     # GEMM2 over two chunks
])
def test_apply_casida_against_extended_precision(n_v, n_c, A, n_vec, kind):
    eps, Lm, X = _case(n_v, n_c, A, n_vec, kind, seed=n_v * n_c + A)
    dev = torch.device("cuda:0")
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, n_v, n_c, A, torch.from_numpy(eps).to(dev),
                                 torch.from_numpy(Lm).to(dev))
        Y = np.zeros_like(X)
        L.lgw_apply_casida(h, s, np.ascontiguousarray(X), Y, "fp64")
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)
    ref, D, d, y = _apply(eps, n_v, Lm, X, LD)
    cpu = _apply(eps, n_v, Lm, X, np.float64)[0]
    err, own = np.abs(Y - ref), np.abs(cpu - ref)
    scale = np.abs(ref).max(1, keepdims=True)
    rms = np.sqrt(np.mean((err / scale) ** 2))
    rms_cpu = np.sqrt(np.mean((own / scale) ** 2))
    assert rms <= 4 * rms_cpu + 2.0 ** -56
    # digits: K 2^-54 of the largest products, twice, and FP64's own roundings
    N = n_v * n_c
    xd = np.abs(X * d.astype(np.float64))
    aL = np.abs(Lm)
    ey = N * 2.0 ** -54 * xd.max(1)[:, None] * aL.max(0)[None] + 2.0 ** -52 * np.abs(y)
    eu = A * 2.0 ** -54 * np.abs(y).max(1)[:, None] * aL.max(1)[None] + ey @ aL.T
    bound = 4 * d * eu + 2.0 ** -50 * (np.abs(X) * D ** 2 + 4 * d * (np.abs(y) @ aL.T))
    assert np.all(err <= bound.astype(np.float64) + 1e-300)


def test_non_finite_inputs_stay_visible():
    """Inf and NaN in L or in one vector: that vector's result is not finite, and with a
    finite L the other vectors' results are untouched."""
    eps, Lm, X = _case(8, 40, 96, 20, "normal", 5)
    dev = torch.device("cuda:0")
    h = L.lgw_create(0)
    try:
        out = {}
        for name, (a, b) in {"clean": (None, None), "x": (None, np.inf), "L": (np.nan, None)}.items():
            L2, X2 = Lm.copy(), X.copy()
            if a is not None:
                L2[7, 3] = a
            if b is not None:
                X2[4, 9] = b
            s = L.lgw_prepare_system(h, 8, 40, 96, torch.from_numpy(eps).to(dev),
                                     torch.from_numpy(L2).to(dev))
            Y = np.zeros_like(X)
            L.lgw_apply_casida(h, s, X2, Y, "fp64")
            out[name] = Y
            L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)
    others = np.arange(20) != 4
    assert np.array_equal(out["x"][others], out["clean"][others])
    assert not np.isfinite(out["x"][4]).any()
    assert not np.isfinite(out["L"]).any()


@pytest.mark.parametrize("n_pairs,n_aux", [(1, 1), (5, 63), (17, 64), (100, 65), (300, 130),
                                           (70, 1030)])
def test_fit_factors_against_extended_precision(n_pairs, n_aux):
    rng = np.random.default_rng(n_pairs + n_aux)
    C = rng.standard_normal((n_pairs, n_aux))
    W = rng.standard_normal((n_aux, n_aux))
    metric = W @ W.T / n_aux + np.eye(n_aux)
    metric = 0.5 * (metric + metric.T)
    B = np.zeros_like(C)
    h = L.lgw_create(0)
    try:
        L.lgw_fit_factors(h, C, metric, B)
    finally:
        L.lgw_destroy(h)
    R = np.linalg.cholesky(metric)
    ref = C.astype(LD) @ R.astype(LD)
    # R itself carries the factorisation's roundings: a few 2^-53 cond(metric) ||R||
    scale = np.abs(ref).max()
    assert np.abs(B - ref).max() <= 64 * 2.0 ** -53 * np.linalg.cond(metric) * scale


def test_workspace_limit_runs_on_the_cuda_cores():
    """A handle with a workspace limit keeps it for the buffers every call needs: the products
    run without digits, in no more memory than that, with the same results to rounding."""
    wl = gw_inputs.tiny(k=16)
    dev = torch.device("cuda:0")
    res, held = {}, {}
    for limit in (0, 1 << 40):
        h = L.lgw_create(0)
        try:
            L.lgw_set_workspace_limit(h, limit)
            s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, torch.from_numpy(wl.eps).to(dev),
                                     torch.from_numpy(wl.L).to(dev))
            prob = L.Problem(targets=torch.from_numpy(wl.targets).to(dev),
                             m_idx=torch.from_numpy(wl.m_idx).to(dev),
                             omega=torch.from_numpy(wl.omega).to(dev), delta=wl.delta,
                             M=torch.from_numpy(wl.M).to(dev))
            sig = torch.zeros(wl.n_t, wl.omega.size, 2, dtype=torch.float64, device=dev)
            e = torch.zeros(wl.n_t, dtype=torch.float64, device=dev)
            opt = L.Options(k=16, precision="fp64", reorth="cgs2")
            L.lgw_sigma_c(h, s, prob, opt, sig, e)
            torch.cuda.synchronize()
            res[limit] = (sig.cpu().numpy(), e.cpu().numpy())
            held[limit] = L.lgw_workspace_bytes(h)
            if limit:      # exactly what it held is enough
                L.lgw_release_workspace(h)
                L.lgw_set_workspace_limit(h, held[limit])
                L.lgw_sigma_c(h, s, prob, opt, sig, e)
                torch.cuda.synchronize()
                assert np.array_equal(sig.cpu().numpy(), res[limit][0])
            L.lgw_release_system(s)
        finally:
            L.lgw_destroy(h)
    assert held[1 << 40] < held[0]
    (s0, e0), (s1, e1) = res[0], res[1 << 40]
    assert np.abs(e0 - e1).max() <= 1e-11
    assert np.abs(s0 - s1).max() <= 1e-9 * np.abs(s0).max()
