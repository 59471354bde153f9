"""The calls that users of the Lanczos GW library make, at the sizes they make them.

Each case is one pass through the public binding (``paper_2310_20103_gb300.lgw`` and its
``autograd`` module): self-energies and quasiparticle energies of one system or of
several, the paper's polynomial form, resuming from stored tridiagonals, the self-energy
matrix of a few targets, density-fitting factors, and gradients.  Inputs follow the recipe
of ``gw_inputs`` (energies U[-12, -5] and U[-3, 20] eV, normal L and M), drawn on the GPU.
"""
import math
import os

import numpy as np
import torch

# A run whose results must be the same from process to process fixes the contraction
# tiles: the autotuner's choice of a split count depends on its timings and changes the
# FP32 summation order of the tensor-core products.
os.environ.setdefault("LGW_AUTOTUNE", "0")

from paper_2310_20103_gb300 import autograd, lgw  # noqa: E402

F64 = torch.float64
DELTA, CK = 0.05, 4.0


def listed():
    sig = dict(kind="sigma", scaled=True, host=False, flags=0)
    return [
        # the smallest request: four states of a molecule in plain FP64, host arrays in and out
        dict(sig, name="tiny_fp64", n_v=8, n_c=32, n_aux=128, n_t=4, n_m=40, n_freq=200, k=64,
             precision="fp64", reorth="cgs2", scaled=False, host=True),
        # a small molecule on the tensor cores; no size is a multiple of a tile
        dict(sig, name="ragged_bf16", n_v=13, n_c=347, n_aux=200, n_t=2, n_m=50, n_freq=333, k=64,
             precision="bf16", reorth="dcgs"),
        # the plain FP64 path that mixed precision is checked against
        dict(sig, name="fp64_plain", n_v=64, n_c=512, n_aux=1024, n_t=1, n_m=64, n_freq=1000, k=24,
             precision="fp64", reorth="cgs2"),
        # one state of the mid-size system as the benchmark runs it (the largest call)
        dict(sig, name="mid_bf16_dcgs", n_v=128, n_c=1024, n_aux=2048, n_t=1, n_m=256, n_freq=1000,
             k=200, precision="bf16", reorth="dcgs"),
        # a cluster-sized pair space: 8-bit L, three-term recurrence only, no FP64 copy of L
        dict(sig, name="cluster_e4m3", n_v=200, n_c=2000, n_aux=4096, n_t=1, n_m=512, n_freq=2000,
             k=16, precision="fp8", reorth="none", flags=lgw.SYS_NO_FP64),
        # the paper's own form: short Lanczos on p_g(C)
        dict(name="poly_bf16", kind="poly", n_v=128, n_c=1024, n_aux=2048, n_t=1, n_m=256,
             n_freq=1000, k=8, g=8, precision="bf16"),
        # several small systems of uneven size in one call
        dict(name="batched_bf16", kind="batched", n_sys=4, shapes=7, n_t=2, n_m=128, n_freq=1000,
             k=100, precision="bf16", reorth="dcgs"),
        # training: energies and their gradient through torch.autograd, stored basis
        dict(name="grad_bf16", kind="grad", n_v=64, n_c=512, n_aux=1024, n_t=1, n_m=128, n_freq=200,
             k=120, precision="bf16", reorth="dcgs"),
        # the exact gradient of a short FP64 recurrence
        dict(name="grad_exact_fp64", kind="grad", n_v=64, n_c=512, n_aux=1024, n_t=1, n_m=32,
             n_freq=200, k=8, precision="fp64", reorth="none"),
        # resuming from stored tridiagonals: spectral map, fractions, QP solve
        dict(name="from_coeffs", kind="coeffs", n_v=128, n_c=1024, n_t=2, n_m=256, n_freq=1000,
             k=200),
        # density-fitting front end: factors of the pairs from a Coulomb metric
        dict(name="fit_factors", kind="fit", n_pairs=16384, n_aux=1024),
        # the self-energy matrix of four frontier orbitals by band Lanczos
        dict(name="band_bf16", kind="band", n_v=64, n_c=512, n_aux=512, n_t=4, n_m=64, n_freq=400,
             k=48, precision="bf16"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pairs(rng, lo, hi):
    """n_v, n_c with n_v n_c spread over [lo, hi] and n_c / n_v about 8."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    n_v = max(4, int(round(math.sqrt(n / 8) * rng.uniform(0.8, 1.25))))
    return n_v, max(8, int(round(n / n_v)))


def draw(rng):
    kind = rng.choice(["sigma_fp64", "sigma_bf16", "sigma_bf16", "sigma_fp8", "poly", "batched",
                       "grad_bf16", "grad_fp64", "coeffs", "fit", "band"])
    n_freq = _logint(rng, 50, 2000)
    if kind in ("sigma_fp64", "sigma_bf16", "sigma_fp8"):
        c = dict(kind="sigma", scaled=True, host=rng.random() < 0.3, flags=0)
        if kind == "sigma_fp64":
            n_v, n_c = _pairs(rng, 256, 32768)
            c.update(n_aux=_logint(rng, 64, 1024), n_t=rng.randint(1, 4), n_m=rng.randint(12, 64),
                     k=rng.randint(8, 24), precision="fp64",
                     reorth=rng.choice(["cgs2", "cgs1k", "none"]))
        elif kind == "sigma_bf16":
            n_v, n_c = _pairs(rng, 1024, 131072)
            c.update(n_aux=_logint(rng, 128, 2048), n_t=rng.randint(1, 2),
                     n_m=_logint(rng, 16, 128), k=_logint(rng, 24, 160), precision="bf16",
                     reorth=rng.choice(["dcgs", "dcgs", "cgs2", "cgs1k"]))
        else:
            n_v, n_c = _pairs(rng, 8192, 400000)
            c.update(n_aux=_logint(rng, 512, 4096), n_t=1, n_m=_logint(rng, 64, 512),
                     k=rng.randint(8, 16), precision=rng.choice(["fp8", "fp8", "fp8_deq", "bf16"]),
                     reorth="none", flags=lgw.SYS_NO_FP64)
        c["n_m"] = min(c["n_m"], n_v + n_c)
        return dict(c, n_v=n_v, n_c=n_c, n_freq=n_freq)
    if kind == "poly":
        n_v, n_c = _pairs(rng, 8192, 131072)
        return dict(kind="poly", n_v=n_v, n_c=n_c, n_aux=_logint(rng, 256, 2048), n_t=1,
                    n_m=_logint(rng, 32, 256), n_freq=n_freq, k=rng.randint(4, 12),
                    g=rng.randint(3, 9), precision="bf16")
    if kind == "batched":
        return dict(kind="batched", n_sys=rng.randint(2, 6), shapes=rng.randint(0, 1 << 20),
                    n_t=rng.randint(1, 2), n_m=_logint(rng, 32, 128), n_freq=n_freq,
                    k=rng.randint(32, 100), precision="bf16", reorth=rng.choice(["dcgs", "cgs1k"]))
    if kind in ("grad_bf16", "grad_fp64"):
        n_v, n_c = _pairs(rng, 1024, 32768)
        c = dict(kind="grad", n_v=n_v, n_c=n_c, n_aux=_logint(rng, 128, 1024), n_t=rng.randint(1, 2),
                 n_freq=200)
        if kind == "grad_bf16":
            c.update(n_m=_logint(rng, 16, 64), k=rng.randint(40, 120), precision="bf16",
                     reorth="dcgs")
        else:
            c.update(n_m=_logint(rng, 8, 16), k=rng.randint(4, 10), precision="fp64",
                     reorth="none")
        return c
    if kind == "coeffs":
        return dict(kind="coeffs", n_v=128, n_c=1024, n_t=rng.randint(1, 4),
                    n_m=_logint(rng, 16, 256), n_freq=n_freq, k=_logint(rng, 8, 300))
    if kind == "fit":
        return dict(kind="fit", n_pairs=_logint(rng, 512, 16384), n_aux=_logint(rng, 64, 1024))
    n_v, n_c = _pairs(rng, 1024, 32768)
    return dict(kind="band", n_v=n_v, n_c=n_c, n_aux=_logint(rng, 128, 512),
                n_t=rng.randint(2, 4), n_m=rng.randint(8, 64), n_freq=_logint(rng, 50, 400),
                k=rng.randint(16, 48), precision=rng.choice(["bf16", "fp64"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _System:
    """A prepared system, released with its last reference."""

    def __init__(self, n_v, n_c, n_aux, eps, L, flags=0):
        self.s = lgw.lgw_prepare_system(_handle(), n_v, n_c, n_aux, eps, L, CK, flags)

    def __del__(self):
        lgw.lgw_release_system(self.s)


_H = {}


def _handle():
    """The one handle that a program keeps (workspace and stream)."""
    if "h" not in _H:
        _H["h"] = lgw.lgw_create(0)
    return _H["h"]


def _dev():
    return torch.device("cuda", 0)


def _gen(seed, part):
    return torch.Generator(device=_dev()).manual_seed(1000003 * int(seed) + part)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=_dev(), dtype=torch.float32).double()


def _eps(c, seed):
    g = _gen(seed, 1)
    u = torch.rand(c["n_v"] + c["n_c"], generator=g, device=_dev(), dtype=F64)
    ev = torch.sort(-12.0 + 7.0 * u[:c["n_v"]])[0]
    ec = torch.sort(-3.0 + 23.0 * u[c["n_v"]:])[0]
    return torch.cat([ev, ec])


def _factor(c, seed):
    s = 0.05 / (math.sqrt(c["n_aux"]) if c.get("scaled", True) else 1.0)
    return _normal(_gen(seed, 2), c["n_v"] * c["n_c"], c["n_aux"]).mul_(s)


def _orbitals(c):
    """Targets on both sides of the gap, and the lowest n_m orbitals that hold them."""
    lo = max(0, c["n_v"] - (c["n_t"] + 1) // 2)
    t = list(range(lo, lo + c["n_t"]))
    first = max(0, c["n_v"] - c["n_m"] // 2)
    m = list(range(min(first, c["n_v"] + c["n_c"] - c["n_m"]), c["n_v"] + c["n_c"]))[:c["n_m"]]
    return t, m


def _couplings(c, seed):
    t, m = _orbitals(c)
    s = 0.1 / (math.sqrt(c["n_aux"]) if c.get("scaled", True) else 1.0)
    M = _normal(_gen(seed, 3), len(t), len(m), c["n_aux"]).mul_(s)
    for i, a in enumerate(t):        # (tm| = (mt| for real orbitals
        for j, b in enumerate(t[:i]):
            if a in m and b in m:
                M[i, m.index(b)] = M[j, m.index(a)]
    return M


def _problem(c, seed, host=False, with_M=True):
    t, m = _orbitals(c)
    d = _dev()
    p = dict(targets=torch.tensor(t, dtype=torch.int32, device=d),
             m_idx=torch.tensor(m, dtype=torch.int32, device=d),
             omega=torch.linspace(-30.0, 30.0, c["n_freq"], dtype=F64, device=d))
    # a checkpoint's request names its couplings too; resuming does not read them
    p["M"] = _couplings(c, seed) if with_M else torch.zeros(
        len(t), len(m), c.get("n_aux", 128), dtype=F64, device=d)
    if host:
        p = {k: v.cpu().numpy() for k, v in p.items()}
    return lgw.Problem(delta=DELTA, **p)


def _outputs(c, host=False):
    shapes = [(c["n_t"], c["n_freq"], 2), (c["n_t"],), (c["n_t"],)]
    if host:
        return [np.zeros(s) for s in shapes]
    return [torch.zeros(s, dtype=F64, device=_dev()) for s in shapes]


def _system(c, seed):
    return _System(c["n_v"], c["n_c"], c["n_aux"], _eps(c, seed), _factor(c, seed),
                   c.get("flags", 0))


def _parts(c):
    """The systems of a batched request, uneven sizes from the case's own shape seed."""
    r = np.random.default_rng(c["shapes"])
    parts = []
    for _ in range(c["n_sys"]):
        n = math.exp(r.uniform(math.log(2048), math.log(24000)))
        n_v = max(8, int(round(math.sqrt(n / 8))))
        n_c = int(round(n / n_v))
        parts.append(dict(c, n_v=n_v, n_c=n_c, n_m=min(c["n_m"], n_v + n_c),
                          n_aux=64 * int(round(math.exp(r.uniform(math.log(4), math.log(16)))))))
    return parts


def _tridiagonals(c, seed):
    """Coefficients as the recurrence leaves them on a spectrum of C within [25, 1000] eV^2:
    they scatter about the constants of that interval."""
    g, B = _gen(seed, 4), c["n_t"] * c["n_m"]
    u = torch.rand(2, B, c["k"], generator=g, device=_dev(), dtype=F64)
    mid, quarter = 0.5 * (1000.0 + 25.0), 0.25 * (1000.0 - 25.0)
    alpha = mid + 15.0 * (2 * u[0] - 1)
    beta = quarter * (0.96 + 0.02 * (2 * u[1] - 1))
    beta0 = 0.15 * (0.8 + 0.4 * torch.rand(B, generator=g, device=_dev(), dtype=F64))
    k_eff = torch.full((B,), c["k"], dtype=torch.int32, device=_dev())
    return alpha, beta, beta0, k_eff


def _interval(c, eps):
    """[x_lo, x_hi] of C: min Delta^2 and max Delta^2 + c_K max Delta ||L||^2, with the norm
    of a normal matrix."""
    gap = float(eps[c["n_v"]] - eps[c["n_v"] - 1])
    top = float(eps[-1] - eps[0])
    norm = 0.05 / math.sqrt(c["n_aux"]) * (math.sqrt(c["n_v"] * c["n_c"]) + math.sqrt(c["n_aux"]))
    return gap * gap, top * top + 1.05 * CK * top * norm * norm


def _fit_inputs(c, seed):
    n = c["n_aux"]
    g = _gen(seed, 5)
    X = _normal(g, n, n)
    metric = X @ X.T / n + torch.eye(n, dtype=F64, device=_dev())
    return _normal(g, c["n_pairs"], n), 0.5 * (metric + metric.T).contiguous()


def prepare(case, seed):
    c, kind, h = case, case["kind"], _handle()
    st = dict(kind=kind, h=h, case=c)
    if kind in ("sigma", "poly", "band"):
        st.update(sys=_system(c, seed), problem=_problem(c, seed, c.get("host", False)))
        st["options"] = lgw.Options(k=c["k"], precision=c["precision"],
                                    reorth=c.get("reorth", "none"))
        if kind == "poly":
            st["interval"] = _interval(c, _eps(c, seed))
        if kind == "band":
            st["out"] = torch.zeros(c["n_t"], c["n_t"], c["n_freq"], 2, dtype=F64, device=_dev())
        else:
            st["out"] = _outputs(c, c.get("host", False))
    elif kind == "batched":
        parts = _parts(c)
        st["systems"] = [_system(p, 100 * seed + i) for i, p in enumerate(parts)]
        st["problems"] = [_problem(p, 100 * seed + i) for i, p in enumerate(parts)]
        st["out"] = [_outputs(p) for p in parts]
        st["options"] = lgw.Options(k=c["k"], precision=c["precision"], reorth=c["reorth"])
    elif kind == "grad":
        st["L"] = _factor(c, seed).requires_grad_()
        st["eps"] = _eps(c, seed).requires_grad_()
        st["problem"] = _problem(c, seed)
        st["options"] = lgw.Options(k=c["k"], precision=c["precision"], reorth=c["reorth"])
        st["dE"] = _weights(c, seed)
    elif kind == "coeffs":
        full = dict(c, n_aux=128)
        st["sys"] = _system(full, seed)
        st["problem"] = _problem(full, seed, with_M=False)
        st["coeffs"] = _tridiagonals(c, seed)
        st["options"] = lgw.Options(k=c["k"])
        st["out"] = _outputs(c)
    else:
        st["C"], st["metric"] = _fit_inputs(c, seed)
        st["out"] = torch.zeros_like(st["C"])
    return st


def _weights(c, seed):
    return 0.5 + torch.rand(c["n_t"], generator=_gen(seed, 6), device=_dev(), dtype=F64)


def run(st):
    kind, h = st["kind"], st["h"]
    if kind == "sigma":
        lgw.lgw_sigma_c(h, st["sys"].s, st["problem"], st["options"], *st["out"])
    elif kind == "poly":
        lgw.lgw_sigma_c_poly(h, st["sys"].s, st["problem"], st["options"], st["case"]["g"],
                             *st["interval"], *st["out"])
    elif kind == "band":
        lgw.lgw_sigma_band(h, st["sys"].s, st["problem"], st["options"], st["out"])
        return {"sigma": st["out"]}
    elif kind == "batched":
        o = st["out"]
        lgw.lgw_sigma_c_batched(h, [s.s for s in st["systems"]], st["problems"], st["options"],
                                [x[0] for x in o], [x[1] for x in o], [x[2] for x in o])
        return [dict(zip(("sigma", "e", "z"), x)) for x in o]
    elif kind == "grad":
        c = st["case"]
        e = autograd.qp_energies(st["L"], st["eps"], c["n_v"], c["n_c"], st["problem"],
                                 st["options"], h, CK)
        dL, deps = torch.autograd.grad(e, (st["L"], st["eps"]), st["dE"])
        return {"e": e.detach(), "dL": dL, "deps": deps}
    elif kind == "coeffs":
        lgw.lgw_sigma_from_coeffs(h, st["sys"].s, st["problem"], st["options"], *st["coeffs"],
                                  *st["out"])
    else:
        lgw.lgw_fit_factors(h, st["C"], st["metric"], st["out"])
        return {"B": st["out"]}
    return dict(zip(("sigma", "e", "z"), st["out"]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c, kind = case, case["kind"]
    if kind == "batched":
        w = [work(dict(p, kind="sigma")) for p in _parts(c)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    if kind == "fit":
        n, A = c["n_pairs"], c["n_aux"]
        return {"bytes": 8.0 * (2 * n * A + A * A), "flops": 1.0 * n * A * A + A ** 3 / 3.0}
    B, k, F = c["n_t"] * c["n_m"], c["k"], c["n_freq"]
    # each fraction level: one complex subtraction and division; grid and about six QP points
    tail = dict(bytes=16.0 * B * k + 16.0 * c["n_t"] * F, flops=10.0 * B * k * (F + 6.0))
    if kind == "coeffs":
        return {"bytes": tail["bytes"], "flops": tail["flops"] + 30.0 * B * k * k}
    N, A = c["n_v"] * c["n_c"], c["n_aux"]
    per = {"fp64": 8.0, "bf16": 2.0, "fp8": 1.0, "fp8_deq": 1.0}[c["precision"]]
    read = per * N * A + 8.0 * B * A + 8.0 * (c["n_v"] + c["n_c"])
    matvec = 4.0 * N * A * B
    gs = 4.0 * N * B * k * (k + 1) / 2.0      # one projection and one update per stored vector
    # a basis larger than the caches is read once per step
    basis = 8.0 * N * B * k * (k - 1) / 2.0 if 8.0 * N * B * k > 128e6 else 0.0
    start = 2.0 * N * A * B
    if kind == "sigma":
        full = c["reorth"] != "none"
        return {"bytes": read + tail["bytes"] + (basis if full else 0.0),
                "flops": start + matvec * k + (gs if full else 6.0 * N * B * k) + tail["flops"]}
    if kind == "poly":
        return {"bytes": read + tail["bytes"],
                "flops": start + matvec * k * c["g"] + 6.0 * N * B * k * c["g"] + tail["flops"]}
    if kind == "band":
        G = c["n_m"]
        return {"bytes": read + 16.0 * c["n_t"] ** 2 * F + 8.0 * N * G * k * (k - 1) / 2.0,
                "flops": (start + matvec * k + gs) * G / B
                + 10.0 * G * c["n_t"] ** 2 * k * (F + k)}
    # forward, and the gradient from the stored basis (two products per step) or by taking the
    # recurrence back (a recomputed and a transposed matvec and two outer products per step)
    if c["reorth"] == "none":
        flops = start + matvec * k * (1.0 + 2.0 + 1.0)
        return {"bytes": 8.0 * N * A * 2 + 8.0 * B * A, "flops": flops + tail["flops"]}
    return {"bytes": 8.0 * N * A * 2 + 8.0 * B * A + basis,
            "flops": start + matvec * k * 2.0 + gs * 2.0 + tail["flops"]}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by torch alone
# ---------------------------------------------------------------------------
def _casida(c, eps, L):
    Delta = (eps[None, c["n_v"]:] - eps[:c["n_v"], None]).reshape(-1)
    d = Delta.sqrt()
    return Delta, d, lambda X: X * Delta ** 2 + CK * d * (((X * d) @ L) @ L.T)


def _lanczos(apply, b, k, full):
    """k steps from the rows of b: alpha, beta [B, k], beta0, and the basis as a list."""
    beta0 = b.norm(dim=1)
    q, qp, bj = b / beta0[:, None], None, None
    Q, al, be = [q], [], []
    for j in range(k):
        w = apply(q)
        if qp is not None:
            w = w - bj[:, None] * qp
        a = (w * q).sum(1)
        w = w - a[:, None] * q
        if full:
            for _ in range(2):
                S = torch.stack(Q, 1)
                w = w - torch.einsum("bj,bjn->bn", torch.einsum("bjn,bn->bj", S, w), S)
                del S
        bj = w.norm(dim=1)
        al.append(a)
        be.append(bj)
        qp, q = q, w / bj[:, None]
        if j + 1 < k:
            Q.append(q)
    return torch.stack(al, 1), torch.stack(be, 1), beta0, Q


def _gauss(alpha, beta):
    T = torch.diag_embed(alpha) + torch.diag_embed(beta[:, :-1], 1) + torch.diag_embed(beta[:, :-1], -1)
    return torch.linalg.eigh(T)


def _sum_poles(c, eps, Om, W, x):
    """Sigma and its derivative at x [n_t, n_x] from poles Om and weights W [n_t * n_m, k]."""
    t, m = _orbitals(c)
    m = torch.tensor(m, device=_dev())
    eta = torch.where(m < c["n_v"], 1.0, -1.0).double()
    S = torch.zeros(x.shape, dtype=torch.complex128, device=_dev())
    dS = torch.zeros_like(S)
    Om, W = Om.reshape(len(t), len(m), -1), W.reshape(len(t), len(m), -1)
    for i in range(len(t)):
        for j in range(0, len(m), 16):
            e = eta[j:j + 16, None, None]
            z = torch.complex(x[i][None] - eps[m[j:j + 16]][:, None],
                              (-DELTA * eta[j:j + 16, None]).expand(-1, x.shape[1]))
            den = z[:, :, None] + e * Om[i, j:j + 16][:, None, :]
            S[i] += (W[i, j:j + 16][:, None, :] / den).sum((0, 2))
            dS[i] -= (W[i, j:j + 16][:, None, :] / den ** 2).sum((0, 2))
    return S, dS


def _sigma_qp(c, eps, Om, W):
    """Sigma on the grid, and the root of E = eps_t + Re Sigma(E) by Newton's method; where it
    does not settle, the root nearest eps_t between grid points."""
    t, _ = _orbitals(c)
    grid = torch.linspace(-30.0, 30.0, c["n_freq"], dtype=F64, device=_dev()).expand(len(t), -1)
    sig, _ = _sum_poles(c, eps, Om, W, grid)
    e0 = eps[torch.tensor(t, device=_dev())][:, None]
    E, done = e0.clone(), torch.zeros_like(e0, dtype=torch.bool)
    for _ in range(50):
        S, dS = _sum_poles(c, eps, Om, W, E)
        dE = (E - e0 - S.real) / (1.0 - dS.real)
        E = torch.where(done, E, E - dE)
        done = done | (dE.abs() <= 1e-10 * E.abs().clamp(min=1.0))
        if bool(done.all()):
            break
    for i in range(len(t)):
        if bool(done[i]):
            continue
        f = grid[i] - e0[i] - sig[i].real
        at = torch.nonzero((f[:-1] * f[1:] < 0) | (f[:-1] == 0))[:, 0]
        lo, hi, flo = grid[i][at].clone(), grid[i][at + 1].clone(), f[at]
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            S, _ = _sum_poles(c, eps, Om, W, mid.expand(len(t), -1))
            left = ((mid - e0[i] - S[i].real) < 0) == (flo < 0)
            lo, hi = torch.where(left, mid, lo), torch.where(left, hi, mid)
        root = 0.5 * (lo + hi)
        E[i] = root[(root - e0[i]).abs().argmin()]
    _, dS = _sum_poles(c, eps, Om, W, E)
    return dict(sigma=torch.view_as_real(sig), e=E[:, 0], z=(1.0 / (1.0 - dS.real))[:, 0])


def _starts(c, seed, L, d):
    return d * (_couplings(c, seed).reshape(-1, c["n_aux"]) @ L.T)


def _poly_apply(apply, g, lo, hi):
    """p_g(C) for the Chebyshev interpolant of sqrt on [lo, hi], by Clenshaw's recurrence."""
    j = (torch.arange(g + 1, dtype=F64) + 0.5) / (g + 1)
    f = torch.sqrt(0.5 * (hi + lo) + 0.5 * (hi - lo) * torch.cos(math.pi * j))
    co = [float(2.0 / (g + 1) * (f * torch.cos(i * math.pi * j)).sum()) for i in range(g + 1)]
    co[0] *= 0.5

    def S(X):
        return (2.0 * apply(X) - (hi + lo) * X) / (hi - lo)

    def D(X):
        b1, b2 = torch.zeros_like(X), torch.zeros_like(X)
        for i in range(g, 0, -1):
            b1, b2 = co[i] * X + (2.0 * S(b1) if i < g else 0.0) - b2, b1
        return co[0] * X + S(b1) - b2

    return D


def _exact_sigma(c, seed):
    eps, L = _eps(c, seed), _factor(c, seed)
    Delta, d, apply = _casida(c, eps, L)
    al, be, b0, _ = _lanczos(apply, _starts(c, seed, L, d), c["k"], c["reorth"] != "none")
    th, U = _gauss(al, be)
    Om = th.sqrt()
    return _sigma_qp(c, eps, Om, b0[:, None] ** 2 * U[:, 0] ** 2 / Om)


def _exact_poly(c, seed):
    eps, L = _eps(c, seed), _factor(c, seed)
    Delta, d, apply = _casida(c, eps, L)
    D = _poly_apply(apply, c["g"], *_interval(c, eps))
    al, be, b0, _ = _lanczos(D, _starts(c, seed, L, d), c["k"], False)
    Om, U = _gauss(al, be)
    return _sigma_qp(c, eps, Om, b0[:, None] ** 2 * U[:, 0] ** 2 / Om)


def _exact_band(c, seed):
    """Block Krylov basis of each summed orbital, k vectors in the band method's order, and
    f(T) of T = Q C Q^T."""
    eps, L = _eps(c, seed), _factor(c, seed)
    Delta, d, apply = _casida(c, eps, L)
    p, G, k = c["n_t"], c["n_m"], c["k"]
    b = _starts(c, seed, L, d).reshape(p, G, -1)
    Q = torch.zeros(k, G, b.shape[2], dtype=F64, device=_dev())

    def append(n, w):
        for _ in range(2):
            w = w - torch.einsum("jg,jgn->gn", torch.einsum("jgn,gn->jg", Q[:n], w), Q[:n])
        Q[n] = w / w.norm(dim=1, keepdim=True)

    for a in range(p):
        append(a, b[a])
    CQ = torch.zeros_like(Q)
    for j in range(k):
        CQ[j] = apply(Q[j])
        if j + p < k:
            append(j + p, CQ[j].clone())
    T = torch.einsum("ign,jgn->gij", Q, CQ)
    R = torch.einsum("jgn,agn->gja", Q[:p], b)
    th, U = torch.linalg.eigh(0.5 * (T + T.transpose(1, 2)))
    V = torch.einsum("gjs,gja->gas", U[:, :p], R)
    Om = th.sqrt()
    x = torch.linspace(-30.0, 30.0, c["n_freq"], dtype=F64, device=_dev())[None]
    out = torch.zeros(p, p, c["n_freq"], 2, dtype=F64, device=_dev())
    _, m = _orbitals(c)
    for i in range(p):
        for j in range(p):
            S = torch.zeros(1, c["n_freq"], dtype=torch.complex128, device=_dev())
            W = V[:, i] * V[:, j] / Om
            for g in range(0, G, 16):
                mm = torch.tensor(m[g:g + 16], device=_dev())
                eta = torch.where(mm < c["n_v"], 1.0, -1.0).double()
                z = torch.complex(x - eps[mm][:, None],
                                  (-DELTA * eta[:, None]).expand(-1, x.shape[1]))
                den = z[:, :, None] + eta[:, None, None] * Om[g:g + 16][:, None, :]
                S[0] += (W[g:g + 16][:, None, :] / den).sum((0, 2))
            out[i, j] = torch.view_as_real(S[0])
    return {"sigma": out}


def _terms(c, Om, U, b0, z, eta):
    """Gauss-rule value of b^T f(C) b, f = 1 / (sqrt(C) (z + eta sqrt(C)))."""
    den = torch.complex(z.real[:, None] + eta[:, None] * Om, z.imag[:, None].expand_as(Om))
    return (b0 ** 2) * (U[:, 0] ** 2 / (Om * den)).sum(1).real


def _exact_grad(c, seed):
    t, m = _orbitals(c)
    eps0, L0 = _eps(c, seed), _factor(c, seed)
    full = c["reorth"] != "none"
    Delta, d, apply = _casida(c, eps0, L0)
    M = _couplings(c, seed).reshape(-1, c["n_aux"])
    al, be, b0, Q = _lanczos(apply, d * (M @ L0.T), c["k"], full)
    th, U = _gauss(al, be)
    Om = th.sqrt()
    r = _sigma_qp(c, eps0, Om, b0[:, None] ** 2 * U[:, 0] ** 2 / Om)
    w = _weights(c, seed) * r["z"]
    ti = torch.tensor(t, device=_dev())
    vm = torch.tensor(m, device=_dev()).repeat(len(t))
    eta = torch.where(vm < c["n_v"], 1.0, -1.0).double()
    cw = w.repeat_interleave(len(m))
    E = r["e"].repeat_interleave(len(m))
    L, eps = L0.clone().requires_grad_(), eps0.clone().requires_grad_()
    Delta, d, apply = _casida(c, eps, L)
    z = torch.complex(E - eps[vm], -DELTA * eta)
    if not full:
        # the derivative of the k-step energies themselves
        al, be, b0, _ = _lanczos(apply, d * (M @ L.T), c["k"], False)
        th, U = _gauss(al, be)
        F = _terms(c, th.sqrt(), U, b0, z, eta)
        total = (cw * F).sum() + (w * eps[ti]).sum()
    else:
        # in the Krylov basis: dF = 2 (f(C) b).db + tr(Q Gamma Q^T dC) + (dF/dz) dz
        zc = z.detach()
        f = 1.0 / (Om * (zc[:, None] + eta[:, None] * Om))
        u1 = U[:, 0]
        ay = 2.0 * b0[:, None] * torch.einsum("bij,bj->bi", U, (f * u1).real)
        s, q = Om[:, :, None], Om[:, None, :]
        zz, ee = zc[:, None, None], eta[:, None, None]
        Fd = -(zz + ee * (s + q)) / (s * q * (zz + ee * s) * (zz + ee * q)) / (s + q)
        Gm = (b0 ** 2)[:, None, None] * torch.einsum(
            "bis,bst,bjt->bij", U, Fd.real * u1[:, :, None] * u1[:, None, :], U)
        S = torch.stack(Q, 1)
        y = torch.einsum("bi,bin->bn", ay * cw[:, None], S)
        R = torch.einsum("bij,bjn->bin", Gm * cw[:, None, None], S)
        diag = (R * S).sum((0, 1))
        b = d * (M @ L.T)
        total = (w * eps[ti]).sum() + (y * b).sum() + (diag * Delta ** 2).sum()
        dfdz = -(b0 ** 2) * (u1 ** 2 / (Om * (zc[:, None] + eta[:, None] * Om) ** 2)).sum(1).real
        total = total - (cw * dfdz * eps[vm]).sum()
        P = (S.reshape(-1, S.shape[2]) * d.detach()) @ L0            # Q^T D L
        X = torch.zeros_like(L0)
        X.addmm_(R.reshape(-1, R.shape[2]).T, P)                     # G D L
        total = total + 2.0 * CK * (d.detach()[:, None] * X * L).sum() + \
            2.0 * CK * (d * (X * L0).sum(1)).sum()
    dL, deps = torch.autograd.grad(total, (L, eps))
    return {"e": r["e"], "dL": dL, "deps": deps}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "fit":
        C, metric = _fit_inputs(c, seed)
        return {"B": C @ torch.linalg.cholesky(metric)}
    if kind == "coeffs":
        al, be, b0, _ = _tridiagonals(c, seed)
        th, U = _gauss(al, be)
        Om = th.sqrt()
        return _sigma_qp(c, _eps(c, seed), Om, b0[:, None] ** 2 * U[:, 0] ** 2 / Om)
    if kind == "batched":
        parts = _parts(c)
        if sum(work(dict(p, kind="sigma"))["flops"] for p in parts) > 4e12:
            return None
        return [_exact_sigma(p, 100 * seed + i) for i, p in enumerate(parts)]
    if work(c)["flops"] > 8e12:        # about 20 seconds in 64 bits
        return None
    return {"sigma": _exact_sigma, "poly": _exact_poly, "band": _exact_band,
            "grad": _exact_grad}[kind](c, seed)
