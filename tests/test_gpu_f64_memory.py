"""When the digits of L that the FP64 products use are made, kept and given back (32 bytes per
element of L: 1 GiB at the size used here)."""
import numpy as np
import pytest

import gw_inputs as gi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GB = 1 << 30
N_V, N_C, A = 64, 512, 1024


@pytest.fixture(scope="module")
def L():
    from paper_2310_20103_gb300.build import build
    build()
    from paper_2310_20103_gb300 import lgw
    return lgw


@pytest.fixture(scope="module")
def inputs():
    g = torch.Generator(device=DEV).manual_seed(1)
    eps = torch.from_numpy(gi.make_workload("p", N_V, N_C, 1, [0], [0], 1, 3).eps).to(DEV)
    Lm = torch.randn(N_V * N_C, A, generator=g, device=DEV, dtype=torch.float64) * 0.05 / A ** 0.5
    X = torch.randn(16, N_V * N_C, generator=g, device=DEV, dtype=torch.float64)
    return eps, Lm, X, torch.empty_like(X)


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _apply(L, h, s, inputs):
    L.lgw_apply_casida(h, s, inputs[2], inputs[3], "fp64")
    torch.cuda.synchronize()
    return inputs[3].clone()


def test_a_limited_handle_makes_none(L, inputs):
    h = L.lgw_create(0)
    try:
        L.lgw_set_workspace_limit(h, 8 * GB)
        s = L.lgw_prepare_system(h, N_V, N_C, A, inputs[0], inputs[1], 4.0)
        before = _free()
        y0 = _apply(L, h, s, inputs)
        assert before - _free() < L.lgw_workspace_bytes(h) + GB // 8
        # with the limit lifted the next request makes them, and a new limit frees them
        L.lgw_set_workspace_limit(h, 0)
        y1 = _apply(L, h, s, inputs)
        assert before - _free() > GB
        L.lgw_set_workspace_limit(h, 8 * GB)
        assert before - _free() < L.lgw_workspace_bytes(h) + GB // 8
        assert torch.equal(_apply(L, h, s, inputs), y0)
        assert float((y0 - y1).norm() / y0.norm()) <= 1e-14
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)


def test_release_workspace_gives_them_back(L, inputs):
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, N_V, N_C, A, inputs[0], inputs[1], 4.0)
        before = _free()
        y0 = _apply(L, h, s, inputs)
        assert before - _free() > GB
        L.lgw_release_workspace(h)
        assert before - _free() < GB // 8
        assert torch.equal(_apply(L, h, s, inputs), y0)
        assert before - _free() > GB
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)


def test_made_again_once_memory_has_come_back(L, inputs):
    """A shortage at one request does not keep a system on the CUDA cores for good."""
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, N_V, N_C, A, inputs[0], inputs[1], 4.0)
        hog = torch.empty(_free() - 2 * GB, dtype=torch.uint8, device=DEV)
        before = _free()
        y0 = _apply(L, h, s, inputs)
        assert before - _free() < L.lgw_workspace_bytes(h) + GB // 8
        del hog
        before = _free()
        y1 = _apply(L, h, s, inputs)
        assert before - _free() > GB
        assert float((y0 - y1).norm() / y0.norm()) <= 1e-14
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_a_factor_with_infinities_is_asked_once(L, inputs, bad):
    """Inf or NaN in L: no digits, and none asked for again."""
    Lm = inputs[1].clone()
    Lm[5, 7] = bad
    h = L.lgw_create(0)
    try:
        s = L.lgw_prepare_system(h, N_V, N_C, A, inputs[0], Lm, 4.0)
        _apply(L, h, s, inputs)
        L.lgw_release_workspace(h)       # the block the attempt took
        before = _free()
        y = _apply(L, h, s, inputs)
        assert before - _free() < L.lgw_workspace_bytes(h) + GB // 8
        assert not torch.isfinite(y).any()
        L.lgw_release_system(s)
    finally:
        L.lgw_destroy(h)
