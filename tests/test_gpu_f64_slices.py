"""FP64 contractions of more than 1024 vectors: slices of 1024 and a shorter last one, whose
own split count needs more partial rows than the first slice's.

Tolerances: apply_casida against FP64 matrix products, elementwise within the a-priori bound
of the digits (2^-54 of the largest factors per term, twice) and of FP64's own roundings; a
gradient against the CUDA-core products of a handle with a byte limit, whose sums differ in
rounding only (1e-8 of the largest element, as for the gradients against the oracle)."""
import numpy as np
import pytest

import gw_inputs as gi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def L():
    from paper_2310_20103_gb300.build import build
    build()
    from paper_2310_20103_gb300 import lgw
    return lgw


def _t(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


@pytest.mark.parametrize("n_v,n_c,A,n_vec", [(16, 256, 384, 1920), (16, 128, 1024, 1040)])
def test_apply_casida_with_a_short_last_slice(L, n_v, n_c, A, n_vec):
    wl = gi.make_workload("p", n_v, n_c, A, [0], [0], 1, 3, aux_scaled=True)
    X = torch.randn(n_vec, n_v * n_c, dtype=torch.float64, device=DEV,
                    generator=torch.Generator(device=DEV).manual_seed(5))
    Y = torch.zeros_like(X)
    Lm, eps = _t(wl.L), _t(wl.eps)
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, n_v, n_c, A, eps, Lm, 4.0)
        L.lgw_apply_casida(h, s, X, Y, "fp64")
        torch.cuda.synchronize()
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)
    D = (eps[None, n_v:] - eps[:n_v, None]).reshape(-1)
    d = D.sqrt()
    x = X * d
    y = x @ Lm
    ref = X * D ** 2 + 4.0 * d * (y @ Lm.T)
    aL, N = Lm.abs(), n_v * n_c
    ey = N * 2.0 ** -54 * x.abs().amax(1)[:, None] * aL.amax(0)[None] \
        + N * 2.0 ** -53 * (x.abs() @ aL)
    eu = A * 2.0 ** -54 * y.abs().amax(1)[:, None] * aL.amax(1)[None] \
        + A * 2.0 ** -53 * (y.abs() @ aL.T) + ey @ aL.T
    bound = 4.0 * d * eu + 2.0 ** -50 * (X.abs() * D ** 2 + 4.0 * d * (y.abs() @ aL.T))
    assert bool(((Y - ref).abs() <= bound).all())
    # far inside the bound on the whole, and nowhere left over from another slice
    assert float((Y - ref).norm() / ref.norm()) <= 1e-14


@pytest.mark.parametrize("n_v,n_c,A,n_m,k", [
    (16, 256, 1024, 16, 84),     # 1344 rows, last slice 320
    (16, 128, 2048, 16, 89),     # 1424 rows, last slice 400
])
def test_gradient_with_a_short_last_slice(L, n_v, n_c, A, n_m, k):
    wl = gi.custom(n_v, n_c, A, 1, n_m, 32, seed=7, k=k)
    dE = _t(np.ones(wl.n_t))
    prob = L.Problem(targets=_t(wl.targets), m_idx=_t(wl.m_idx), omega=_t(wl.omega),
                     delta=wl.delta, M=_t(wl.M))
    out = {}
    for limit in (0, 1 << 40):
        h = L.lgw_create(0)
        try:
            L.lgw_set_workspace_limit(h, limit)
            s = L.lgw_prepare_system(h, n_v, n_c, A, _t(wl.eps), _t(wl.L), 4.0)
            dL = torch.zeros(n_v * n_c, A, dtype=torch.float64, device=DEV)
            de = torch.zeros(n_v + n_c, dtype=torch.float64, device=DEV)
            L.lgw_sigma_c_backward(h, s, prob, L.Options(k=k, precision="fp64", reorth="cgs2"),
                                   dE, dL, de)
            torch.cuda.synchronize()
            out[limit] = (dL, de)
            L.lgw_release_system(s)
        finally:
            L.lgw_destroy(h)
    for a, b in zip(out[0], out[1 << 40]):
        assert float((a - b).abs().max()) <= 1e-8 * float(b.abs().max())


@pytest.mark.parametrize("reorth", ["cgs2", "cgs1k"])
def test_sub_batches_on_a_fresh_handle(L, reorth):
    """A gradient in sub-batches on a handle whose buffers have not grown yet: the adjoint of
    one sub-batch contracts k times as many rows as the recurrence of the next, which must
    still find its own buffers.  Against the single pass, on a handle of its own."""
    wl = gi.tiny(k=40)
    dE = _t(np.random.default_rng(3).normal(size=wl.n_t))
    prob = L.Problem(targets=_t(wl.targets), m_idx=_t(wl.m_idx), omega=_t(wl.omega),
                     delta=wl.delta, M=_t(wl.M))
    out = []
    for b_sub in (48, 0):
        h = L.lgw_create(0)
        try:
            s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, _t(wl.eps), _t(wl.L), 4.0)
            dL = torch.zeros(wl.n_vc, wl.n_aux, dtype=torch.float64, device=DEV)
            de = torch.zeros(wl.n_v + wl.n_c, dtype=torch.float64, device=DEV)
            opt = L.Options(k=40, precision="fp64", reorth=reorth, b_sub=b_sub)
            L.lgw_sigma_c_backward(h, s, prob, opt, dE, dL, de)
            torch.cuda.synchronize()
            out.append((dL, de))
            L.lgw_release_system(s)
        finally:
            L.lgw_destroy(h)
    for a, b in zip(*out):
        assert float((a - b).abs().max()) <= 1e-12 * float(b.abs().max())


def test_one_split_needs_no_partials(L):
    """On a handle with a byte limit (CUDA-core products) a contraction of one split writes
    its result directly: vectors, results and y are all that a wide product holds."""
    n_v, n_c, A, n_vec = 8, 32, 1024, 1216       # 16 x 19 tiles: one split
    wl = gi.make_workload("p", n_v, n_c, A, [0], [0], 1, 3, aux_scaled=True)
    X = torch.randn(n_vec, n_v * n_c, dtype=torch.float64, device=DEV,
                    generator=torch.Generator(device=DEV).manual_seed(5))
    out = []
    for limit in (0, 8 * n_vec * (2 * n_v * n_c + A)):
        h = L.lgw_create(0)
        try:
            s = L.lgw_prepare_system(h, n_v, n_c, A, _t(wl.eps), _t(wl.L), 4.0)
            L.lgw_set_workspace_limit(h, limit)
            Y = torch.zeros_like(X)
            L.lgw_apply_casida(h, s, X, Y, "fp64")
            torch.cuda.synchronize()
            out.append(Y)
            L.lgw_release_system(s)
        finally:
            L.lgw_destroy(h)
    assert float((out[0] - out[1]).norm() / out[0].norm()) <= 1e-14
