// Continued fractions on the frequency grid (Eq. 14, 10) and the
// quasiparticle equation, FP64.
//
// For a target t and summed orbital m with Jacobi matrix (a, b^2) and total
// weight W of the Omega-space measure (built by the spectral map):
//   Sigma_tm(omega) = -eta_m G(zeta),  zeta = -eta_m (omega - eps_m) + i delta,
//   G(zeta) = W / (zeta - a_0 - b_1^2 / (zeta - a_1 - b_2^2 / (...)))
// which is Eq. 11 (z_m = omega - eps_m - i eta_m delta, zeta = -eta_m z_m).
// The spectral map's measure comes as its poles and weights, and G as their
// sum sum_j wt_j / (zeta - Omega_j); the fraction is evaluated for the forms
// whose own tridiagonal it is (polynomial, Tamm-Dancoff).
// Sigma_t = sum over the summed set of Sigma_tm (Eq. 10).
#include <cooperative_groups.h>

#include <algorithm>

#include "fp_iter.cuh"
#include "lgw_internal.cuh"

namespace lgw {

struct cplx {
  double re, im;
};

// G(zeta) by bottom-up evaluation of the continued fraction; optionally the
// derivative dG/dzeta by differentiating the recurrence.
template <bool DERIV>
__device__ __forceinline__ void cf_eval(const double *__restrict__ a, const double *__restrict__ b2,
                                        int n, double W, double zr, double zi, cplx &G, cplx &dG) {
  double tr = zr - a[n - 1], ti = zi;
  double dr = 1.0, di = 0.0;   // dT/dzeta
  for (int i = n - 2; i >= 0; --i) {
    const double inv = 1.0 / fma(tr, tr, ti * ti);
    const double q = b2[i] * inv;          // b^2 / T = q * conj(T)
    const double fr = q * tr, fi = -q * ti;
    if (DERIV) {
      // d(b^2/T) = -b^2 dT / T^2 ; T^-2 = conj(T)^2 inv^2
      const double ir = (tr * tr - ti * ti) * inv * inv, ii = -2.0 * tr * ti * inv * inv;
      const double pr = dr * ir - di * ii, pi = dr * ii + di * ir;
      dr = 1.0 + b2[i] * pr;
      di = b2[i] * pi;
    }
    tr = zr - a[i] - fr;
    ti = zi - fi;
  }
  const double inv = 1.0 / fma(tr, tr, ti * ti);
  G.re = W * tr * inv;
  G.im = -W * ti * inv;
  if (DERIV) {
    const double ir = (tr * tr - ti * ti) * inv * inv, ii = -2.0 * tr * ti * inv * inv;
    const double pr = dr * ir - di * ii, pi = dr * ii + di * ir;
    dG.re = -W * pr;
    dG.im = -W * pi;
  }
}

// One thread per (target, frequency, slice of the summed set): loops over its
// slice of m and the poles.  Threads of a warp share t and m and read the same
// poles (broadcast loads).  Slices as in k_cf_grid below.  Bound by the FP64
// pipe: 8 operations per pole, against about 18 per level of the fraction
// (2 targets x 1000 frequencies x 256 orbitals x 200: 2.13 -> 1.57 ms).
__global__ void k_cf_poles(CfProblem p, JacobiBufs jb, double *__restrict__ out, int mchunk) {
  pdl_wait();
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  const int ti = blockIdx.y, sl = blockIdx.z;
  if (f >= p.n_freq) return;
  const double om = p.omega[f], d2 = p.delta * p.delta;
  const int mi0 = sl * mchunk, mi1 = min(p.n_m, mi0 + mchunk);
  double sr = 0.0, si = 0.0;
  for (int mi = mi0; mi < mi1; ++mi) {
    const int v = ti * p.n_m + mi;
    const int n = jb.n[v];
    const int m = p.m_idx[mi];
    const double eta = (m < p.n_v) ? 1.0 : -1.0;
    const double zr = -eta * (om - p.eps[m]);
    const double *x0 = jb.a + (size_t)v * p.k, *w0 = jb.b2 + (size_t)v * p.k;
    double gr = 0.0, gi = 0.0;   // sum wt x / (x^2 + delta^2) and sum wt / (x^2 + delta^2)
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const double x = zr - x0[j];
      const double r = w0[j] * pole_rcp(fma(x, x, d2));
      gr = fma(r, x, gr);
      gi += r;
    }
    sr -= eta * gr;
    si = fma(eta * p.delta, gi, si);
  }
  const size_t o = (((size_t)sl * p.n_t + ti) * p.n_freq + f) * 2;
  out[o] = sr;
  out[o + 1] = si;
}

// One thread per (target, frequency, slice of the summed set): loops over its
// slice of m and the continued-fraction depth.  Threads of a warp share t and
// m and read the same coefficients (broadcast loads).  With one slice the
// thread writes Sigma_t(omega_f) itself; otherwise its partial sum goes to
// part[slice] and k_cf_reduce adds the slices in a fixed order.
__global__ void k_cf_grid(CfProblem p, JacobiBufs jb, double *__restrict__ out, int mchunk) {
  pdl_wait();
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  const int ti = blockIdx.y, sl = blockIdx.z;
  if (f >= p.n_freq) return;
  const double om = p.omega[f];
  const int mi0 = sl * mchunk, mi1 = min(p.n_m, mi0 + mchunk);
  double sr = 0.0, si = 0.0;
  for (int mi = mi0; mi < mi1; ++mi) {
    const int v = ti * p.n_m + mi;
    const int n = jb.n[v];
    if (n <= 0) continue;
    const int m = p.m_idx[mi];
    const double eta = (m < p.n_v) ? 1.0 : -1.0;
    const double zr = -eta * (om - p.eps[m]);
    cplx G, dG;
    cf_eval<false>(jb.a + (size_t)v * p.k, jb.b2 + (size_t)v * p.k, n, jb.w0[v], zr, p.delta, G,
                   dG);
    if (jb.g0 == nullptr) {
      sr -= eta * G.re;
      si -= eta * G.im;
    } else {
      // (G(zeta) - G(0)) / z,  z = omega - eps_m - i eta delta
      const double xr = om - p.eps[m], xi = -eta * p.delta;
      const double inv = 1.0 / fma(xr, xr, xi * xi);
      const double nr = G.re - jb.g0[v], ni = G.im;
      sr += (nr * xr + ni * xi) * inv;
      si += (ni * xr - nr * xi) * inv;
    }
  }
  const size_t o = (((size_t)sl * p.n_t + ti) * p.n_freq + f) * 2;
  out[o] = sr;
  out[o + 1] = si;
}

__global__ void k_cf_reduce(const double *__restrict__ part, int S, size_t n,
                            double *__restrict__ sigma) {
  pdl_wait();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int sl = 0; sl < S; ++sl) s += part[(size_t)sl * n + i];
  sigma[i] = s;
}

// A target's QP equation runs on one cluster of QP_CTAS blocks: its few
// evaluations of Sigma_t, one after the other, are FP64-bound, and one warp
// keeps only one of the 608 FP64 units busy (2 targets, 256 summed orbitals,
// 200 levels: 3.85 ms for the solve; the clusters take 0.078 ms).
constexpr int QP_CTAS = 8, QP_THREADS = 256, QP_WARPS = QP_THREADS / 32;

struct QpShared {
  double warp[QP_WARPS][2];
  double part[2][2];    // this block's sums, by the parity of the evaluation
  double tot[2];
};

// Re Sigma_t(E) and Re dSigma_t/domega at one real E, on every thread of the
// cluster.  Pole sums: warps split the summed set, lanes the poles; fractions:
// threads split the summed set.  Partial sums meet in a fixed order.  The
// parity buffers are reused two evaluations later, after every block has
// passed the barrier in between and so has read them.
__device__ void sigma_at(const CfProblem &p, const JacobiBufs &jb, int ti, double E,
                         QpShared &sh, int &par, double &S, double &dS) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int rank = (int)cl.block_rank();
  double sr = 0.0, dr = 0.0;
  if (jb.poles) {
    const double d2 = p.delta * p.delta;
    for (int mi = rank * QP_WARPS + wid; mi < p.n_m; mi += QP_CTAS * QP_WARPS) {
      const int v = ti * p.n_m + mi;
      const int n = jb.n[v];
      const int m = p.m_idx[mi];
      const double eta = (m < p.n_v) ? 1.0 : -1.0;
      const double zr = -eta * (E - p.eps[m]);
      const double *x0 = jb.a + (size_t)v * p.k, *w0 = jb.b2 + (size_t)v * p.k;
      double gr = 0.0;
      for (int j = lane; j < n; j += 32) {
        // G = sum wt / zeta_j, dG/dzeta = -sum wt / zeta_j^2, zeta_j = x + i delta
        const double x = zr - x0[j];
        const double inv = pole_rcp(fma(x, x, d2));
        const double r = w0[j] * inv;
        gr = fma(r, x, gr);
        dr = fma(-(r * inv), fma(x, x, -d2), dr);
      }
      sr -= eta * gr;
    }
  } else {
    for (int mi = rank * QP_THREADS + (int)threadIdx.x; mi < p.n_m;
         mi += QP_CTAS * QP_THREADS) {
      const int v = ti * p.n_m + mi;
      const int n = jb.n[v];
      if (n <= 0) continue;
      const int m = p.m_idx[mi];
      const double eta = (m < p.n_v) ? 1.0 : -1.0;
      cplx G, dG;
      cf_eval<true>(jb.a + (size_t)v * p.k, jb.b2 + (size_t)v * p.k, n, jb.w0[v],
                    -eta * (E - p.eps[m]), p.delta, G, dG);
      if (jb.g0 == nullptr) {
        sr -= eta * G.re;
        dr += dG.re;
      } else {
        // S = (G(zeta) - G(0)) / z, zeta = -eta z:
        // dS/dz = -eta G'(zeta) / z - S / z
        const double xr = E - p.eps[m], xi = -eta * p.delta;
        const double inv = 1.0 / fma(xr, xr, xi * xi);
        const double nr = G.re - jb.g0[v], ni = G.im;
        const double qr = (nr * xr + ni * xi) * inv, qi = (ni * xr - nr * xi) * inv;
        sr += qr;
        const double gr = -eta * dG.re - qr, gi = -eta * dG.im - qi;
        dr += (gr * xr + gi * xi) * inv;
      }
    }
  }
  sr = warp_sum(sr);
  dr = warp_sum(dr);
  if (lane == 0) {
    sh.warp[wid][0] = sr;
    sh.warp[wid][1] = dr;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int w = 0; w < QP_WARPS; ++w) s += sh.warp[w][threadIdx.x];
    sh.part[par][threadIdx.x] = s;
  }
  cl.sync();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int r = 0; r < QP_CTAS; ++r) s += cl.map_shared_rank(sh.part[par], r)[threadIdx.x];
    sh.tot[threadIdx.x] = s;
  }
  __syncthreads();
  S = sh.tot[0];
  dS = sh.tot[1];
  par ^= 1;
}

// QP equation E = e0 + Re Sigma_t(E), e0 = eps_t + s_t: Newton from e0; if it
// fails, bracket sign changes of f on the grid (from the grid values of
// Sigma), bisect each and keep the root nearest e0 (ties: larger Z).
// One cluster per target; every thread follows the same iterates.
__global__ void __cluster_dims__(QP_CTAS, 1, 1) __launch_bounds__(QP_THREADS)
    k_qp(CfProblem p, JacobiBufs jb, const double *__restrict__ sigma, int max_iter, double tol,
         double *e_qp, double *z_qp, unsigned *status) {
  pdl_wait();
  namespace cg = cooperative_groups;
  __shared__ QpShared sh;
  const int ti = blockIdx.x / QP_CTAS;
  const bool lead = blockIdx.x % QP_CTAS == 0 && threadIdx.x == 0;
  const int t = p.targets[ti];
  const double e0 = p.eps[t] + (p.shift ? p.shift[ti] : 0.0);
  double E = e0, Z = 0.0, S, dS;
  int par = 0;
  bool ok = false;
  if (p.qp_mode == 1) {
    // linearised: E = e0 + Z Re Sigma(e0), Z = 1 / (1 - Re Sigma'(e0))
    sigma_at(p, jb, ti, e0, sh, par, S, dS);
    Z = 1.0 / (1.0 - dS);
    E = e0 + Z * S;
  } else {
    for (int it = 0; it < max_iter; ++it) {
      sigma_at(p, jb, ti, E, sh, par, S, dS);
      const double f = E - e0 - S;
      const double fp = 1.0 - dS;
      const double dE = f / fp;
      if (fp == 0.0 || !isfinite(dE)) break;
      E -= dE;
      if (fabs(dE) <= tol * fmax(1.0, fabs(E))) {
        ok = true;
        break;
      }
    }
    if (ok) {
      sigma_at(p, jb, ti, E, sh, par, S, dS);
      Z = 1.0 / (1.0 - dS);
    } else {
      bool found = false;
      double best_r = 0.0, best_z = 0.0, best_d = 0.0;
      const double *sg = sigma + (size_t)ti * p.n_freq * 2;
      for (int g = 0; g + 1 < p.n_freq; ++g) {
        const double f0 = p.omega[g] - e0 - sg[2 * g];
        const double f1 = p.omega[g + 1] - e0 - sg[2 * g + 2];
        if (!(f0 == 0.0 || f0 * f1 < 0.0)) continue;
        double lo = p.omega[g], hi = p.omega[g + 1], flo = f0;
        double mid = 0.5 * (lo + hi);
        for (int it = 0; it < 200; ++it) {
          mid = 0.5 * (lo + hi);
          sigma_at(p, jb, ti, mid, sh, par, S, dS);
          const double fm = mid - e0 - S;
          if ((fm < 0.0) == (flo < 0.0)) {
            lo = mid;
            flo = fm;
          } else {
            hi = mid;
          }
          if (hi - lo <= tol * fmax(1.0, fabs(mid))) break;
        }
        const double r = 0.5 * (lo + hi);
        sigma_at(p, jb, ti, r, sh, par, S, dS);
        const double zr = 1.0 / (1.0 - dS);
        const double dist = fabs(r - e0);
        if (!found || dist < best_d || (dist == best_d && zr > best_z)) {
          found = true;
          best_r = r;
          best_z = zr;
          best_d = dist;
        }
      }
      if (found) {
        E = best_r;
        Z = best_z;
      } else {
        if (lead) atomicOr(status, ST_NO_CONV);
        E = NAN;
        Z = NAN;
      }
    }
  }
  if (lead) {
    e_qp[ti] = E;
    if (z_qp) z_qp[ti] = Z;
  }
  cg::this_cluster().sync();   // no block leaves while another may read its sums
}

int cf_slices(const CfProblem &p) {
  // enough (target, frequency, slice) threads to hide the FP64 latency of
  // the continued-fraction chains: about 128k, at most 64 slices
  if (p.n_t <= 0 || p.n_freq <= 0 || p.n_m <= 0) return 1;
  const long long tf = (long long)p.n_t * p.n_freq;
  long long S = (131072 + tf - 1) / tf;
  S = std::min<long long>(S, std::min(p.n_m, 64));
  return (int)std::max<long long>(S, 1);
}

int launch_cf_grid(const CfProblem &p, JacobiBufs jb, double *sigma, double *part, int S,
                   cudaStream_t st) {
  if (p.n_freq <= 0 || p.n_t <= 0) return 0;
  if (part == nullptr) S = 1;
  const int mchunk = (p.n_m + S - 1) / S;
  S = std::max(1, (p.n_m + mchunk - 1) / std::max(1, mchunk));
  dim3 grid((p.n_freq + 127) / 128, p.n_t, S);
  double *out = S == 1 ? sigma : part;
  if (jb.poles)
    launch_pdl(k_cf_poles, grid, dim3(128), 0, st, p, jb, out, std::max(1, mchunk));
  else
    launch_pdl(k_cf_grid, grid, dim3(128), 0, st, p, jb, out, std::max(1, mchunk));
  if (S > 1) {
    const size_t n = (size_t)p.n_t * p.n_freq * 2;
    launch_pdl(k_cf_reduce, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, part, S, n,
               sigma);
    return 2;
  }
  return 1;
}

void launch_qp(const CfProblem &p, JacobiBufs jb, const double *sigma, int max_iter, double tol,
               double *e_qp, double *z_qp, unsigned *status, cudaStream_t st) {
  if (p.n_t <= 0) return;
  launch_pdl(k_qp, dim3(p.n_t * QP_CTAS), dim3(QP_THREADS), 0, st, p, jb, sigma, max_iter, tol,
             e_qp, z_qp, status);
}

}  // namespace lgw
