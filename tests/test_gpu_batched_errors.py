"""A batched call that fails at one of its systems has the others in flight on streams of its
own.  It may only return once they are done: the caller releases their systems and buffers
after synchronising the handle's stream, and their memory goes to the next system."""
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


@pytest.mark.parametrize("precision", ["fp64", "bf16"])
def test_work_in_flight_is_waited_for(L, precision):
    wl = gi.custom(32, 256, 512, 1, 32, 400, seed=3, k=60)
    opt = L.Options(k=60, precision=precision, reorth="cgs2")
    good = L.Problem(targets=_t(wl.targets), m_idx=_t(wl.m_idx), omega=_t(wl.omega),
                     delta=wl.delta, M=_t(wl.M))
    m = wl.m_idx.copy()
    m[3] = wl.n_v + wl.n_c + 5               # no such orbital
    bad = L.Problem(targets=_t(wl.targets), m_idx=_t(m), omega=_t(wl.omega), delta=wl.delta,
                    M=_t(wl.M))
    eps, Lm = _t(wl.eps), _t(wl.L)
    new = lambda: (torch.zeros(wl.n_t, wl.omega.size, 2, dtype=torch.float64, device=DEV),
                   torch.zeros(wl.n_t, dtype=torch.float64, device=DEV))
    h = L.lgw_create(0)
    try:
        systems = [L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, eps, Lm, 4.0)
                   for _ in range(2)]
        ref = [new(), new()]
        L.lgw_sigma_c_batched(h, systems, [good, good], opt, [x[0] for x in ref],
                              [x[1] for x in ref])
        torch.cuda.synchronize()
        got = [new(), new()]
        with pytest.raises(L.LgwError, match="LGW_ERR_SHAPE"):
            L.lgw_sigma_c_batched(h, systems, [good, bad], opt, [x[0] for x in got],
                                  [x[1] for x in got])
        # on the handle's stream, no other synchronisation: the first system's results
        sig, e = got[0][0].cpu(), got[0][1].cpu()
        torch.cuda.synchronize()
        assert torch.equal(sig, ref[0][0].cpu()) and torch.equal(e, ref[0][1].cpu())
        # and the handle goes on
        L.lgw_release_system(systems[0])
        s = L.lgw_prepare_system(h, wl.n_v, wl.n_c, wl.n_aux, eps, 0.5 * Lm, 4.0)
        last = [new(), new()]
        L.lgw_sigma_c_batched(h, [s, systems[1]], [good, good], opt, [x[0] for x in last],
                              [x[1] for x in last])
        torch.cuda.synchronize()
        assert torch.equal(last[1][0], ref[1][0])
        assert not torch.equal(last[0][0], ref[0][0])
        L.lgw_release_system(s)
        L.lgw_release_system(systems[1])
    finally:
        L.lgw_destroy(h)
