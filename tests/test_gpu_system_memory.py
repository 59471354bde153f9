"""Device memory of released systems that a handle keeps for the next one.

Results must not depend on what a reused block held before (bit for bit those of a handle
that starts with fresh memory), at sizes that reuse, partly reuse and outgrow the blocks,
and the blocks must go back when the header says so."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GB = 1 << 30


@pytest.fixture(scope="module")
def L():
    from paper_2310_20103_gb300.build import build
    build()
    from paper_2310_20103_gb300 import lgw
    return lgw


def _system(L, h, n_v, n_c, n_aux):
    g = torch.Generator(device=DEV).manual_seed(n_v * n_c + n_aux)
    eps = torch.cat([torch.linspace(-9, -6, n_v), torch.linspace(-3, 15, n_c)]).double().to(DEV)
    Lm = torch.randn(n_v * n_c, n_aux, generator=g, device=DEV).double() * 0.01
    return L.lgw_prepare_system(h, n_v, n_c, n_aux, eps, Lm, 4.0)


def _apply(L, h, sizes, precision):
    s = _system(L, h, *sizes)
    n = sizes[0] * sizes[1]
    X = torch.randn(3, n, generator=torch.Generator(device=DEV).manual_seed(1), device=DEV).double()
    Y = torch.empty_like(X)
    L.lgw_apply_casida(h, s, X, Y, precision)
    torch.cuda.synchronize()
    L.lgw_release_system(s)
    return Y


@pytest.mark.parametrize("precision", ["fp64", "bf16", "fp8"])
def test_reused_blocks_give_the_same_results(L, precision):
    sizes = [(9, 211, 200), (9, 211, 200), (9, 200, 190), (5, 100, 70), (12, 300, 300),
             (9, 211, 200)]
    h = L.lgw_create(0)
    got = [_apply(L, h, c, precision) for c in sizes]
    L.lgw_destroy(h)
    for c, y in zip(sizes, got):
        f = L.lgw_create(0)
        assert torch.equal(y, _apply(L, f, c, precision)), c
        L.lgw_destroy(f)


@pytest.mark.parametrize("how", ["release", "limit", "destroy"])
def test_blocks_are_bounded_and_given_back(L, how):
    h = L.lgw_create(0)
    L.lgw_release_system(_system(L, h, 4, 40, 64))
    L.lgw_release_workspace(h)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    big = [_system(L, h, 128, 1024, 1024) for _ in range(2)]     # 1.9 GB each
    for s in big:
        L.lgw_release_system(s)
    torch.cuda.empty_cache()
    assert before - torch.cuda.mem_get_info()[0] < 2 * GB + L.lgw_workspace_bytes(h) + GB // 8
    if how == "release":
        L.lgw_release_workspace(h)
    elif how == "limit":
        L.lgw_set_workspace_limit(h, 10 * GB)
    else:
        L.lgw_destroy(h)
    held = 0 if how == "destroy" else L.lgw_workspace_bytes(h)
    torch.cuda.empty_cache()
    assert before - torch.cuda.mem_get_info()[0] < held + GB // 8
    if how != "destroy":
        L.lgw_destroy(h)
