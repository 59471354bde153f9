// Adjoint of the QP energies: d(sum_t dE_t E_t)/dL and /d(eps).
//
// E_t = eps_t + s_t + Re Sigma_t(E_t), so dE_t = Z_t (d eps_t + Re dSigma_t)
// at fixed omega = E_t (implicit function).  Each term of Sigma_t is
// F = b^T f(C) b with f(theta) = 1 / (sqrt(theta) (z_m + eta_m sqrt(theta)))
// (Eq. 7-12).  In the k-step Krylov basis Q of (C, b) with
// T_k = U diag(theta) U^T and u1 = U^T e1:
//   dF/db = y = 2 f(C) b      ~ Q a_y,   a_y = 2 beta0 Re U (f(theta) o u1)
//   dF/dC = G                 ~ Q Gam Q^T,  Gam = beta0^2 Re U (F o u1 u1^T) U^T
//   dF/dz = -beta0^2 sum_s u1s^2 / (Omega_s (z + eta Omega_s)^2)
// with F_st the divided differences of f (Daleckii-Krein); exact when the
// Krylov space is the whole space.  With C = Delta^2 + c_K D L L^T D,
// D = diag(Delta^1/2) and b = D L M:
//   dL     = 2 c_K D (G D L) + D (y M^T)
//   dDelta = 2 Delta diag(G) + c_K diag(L (G D L)^T) / d + y b / (2 Delta)
// All per-vector weights c_v = dE_t Z_t are folded into a_y, Gam and dz.
// The eigen-decompositions, coefficients and Gam P are FP64.  The large
// contractions P = Q^T D L and SC = Q R run on the FP64 pipe in the FP64
// mode and as three split-BF16 tensor-core products (hi hi + hi lo + lo hi,
// FP64 sums of FP32 chunks) in the BF16 mode, where y and diag(Q Gam Q^T)
// also move to the FP32 pipe.
#include "lgw_internal.cuh"

namespace lgw {

// --------------------------------------------------------------------------
// Full eigen-decomposition of each T_k: implicit symmetric QR with Wilkinson
// shifts, chasing downwards.  One block per vector: warp 0 runs the scalar
// chain of a sweep and leaves its rotations in shared memory; the other warps
// apply the previous sweep's to the rows of V = U^T (row s = eigenvector s,
// coalesced) meanwhile.
//
// What bounds it: the scalar chain, about 1.7 n sweeps of rotations in
// sequence, each FP64 instruction of which holds its unit for 64 clocks
// however few lanes it has.  So even lanes carry what belongs to c and odd
// lanes what belongs to s: one division, one square and one diagonal update
// per rotation serve both.  The operations and their order stay those of one
// thread's chain (the split of Gamma P that follows rounds to 16 bits, where a
// last-place difference now and then moves a digit).  128 vectors, k 120: 45.3
// ms with the row updates in the chain, 25 ms now (13.9 with reciprocal square
// roots in place of hypot and the divisions, which moved dL by 1e-9).
// --------------------------------------------------------------------------
constexpr int EIG_THREADS = 128;

__global__ void __launch_bounds__(EIG_THREADS) k_eig_full(AdjCtx a) {
  pdl_wait();
  extern __shared__ double sm[];
  __shared__ int ctl[2][3];   // by sweep parity: first row, rotations, 1 = no convergence
  const int tid = threadIdx.x;
  const int b = blockIdx.x, k = a.k;
  double *d = sm, *e = d + k;
  double2 *rot = reinterpret_cast<double2 *>(e + k);   // [2][k]
  double *V = a.V + (size_t)b * k * k;
  const int v = a.vec0 + b;
  const int n = (b < a.nvec) ? a.k_eff[v] : 0;
  for (int i = tid; i < k * k; i += EIG_THREADS)
    V[i] = ((i / k) == (i % k) && (i / k) < n) ? 1.0 : 0.0;
  for (int i = tid; i < k; i += EIG_THREADS) {
    d[i] = (i < n) ? a.alpha[(size_t)v * k + i] : 0.0;
    e[i] = (i + 1 < n) ? a.beta[(size_t)v * k + i] : 0.0;
  }
  if (tid < 2) ctl[tid][0] = -1, ctl[tid][1] = ctl[tid][2] = 0;
  __syncthreads();
  const double eps = 2.220446049250313e-16;
  int hi = n - 1, iter = 0;   // warp 0, alike in every lane
  const int max_iter = 60 * n + 60;
  const bool odd = (tid & 1) != 0;
  for (int sweep = 0;; ++sweep) {
    const int cur = sweep & 1, prev = cur ^ 1;
    if (tid < 32) {
      int lo = -1, nr = 0;
      while (hi > 0 && fabs(e[hi - 1]) <= eps * (fabs(d[hi - 1]) + fabs(d[hi]))) {
        __syncwarp();
        if (tid == 0) e[hi - 1] = 0.0;
        __syncwarp();
        --hi;
      }
      if (hi > 0 && ++iter <= max_iter) {
        lo = hi - 1;
        while (lo > 0 && fabs(e[lo - 1]) > eps * (fabs(d[lo - 1]) + fabs(d[lo]))) --lo;
        __syncwarp();
        if (tid == 0 && lo > 0) e[lo - 1] = 0.0;
        // Wilkinson shift from the trailing 2 x 2 block
        const double dl = 0.5 * (d[hi - 1] - d[hi]);
        const double bb = e[hi - 1];
        const double den = dl + copysign(sqrt(fma(dl, dl, bb * bb)), dl != 0.0 ? dl : 1.0);
        const double mu = d[hi] - bb * bb / den;
        double a0 = d[lo], b0 = e[lo];
        double x = a0 - mu, z = b0;
        __syncwarp();   // every lane has read what lane 0 writes below
        for (int i = lo; i < hi; ++i) {
          // R = [[c, s], [-s, c]] maps (x, z) to (r, 0); T <- R T R^T on rows i, i + 1
          const double c0 = d[i + 1], en = e[i + 1];   // e has k entries, k > hi
          const double r = hypot(x, z);
          const double q = r > 0.0 ? (odd ? z : x) / r : (odd ? 0.0 : 1.0);   // s or c
          const double q2 = q * q;
          const double o = __shfl_xor_sync(0xffffffffu, q, 1);
          const double o2 = __shfl_xor_sync(0xffffffffu, q2, 1);
          const double m = q * en;                      // c e_{i+1}, or the bulge
          const double csn = q * o;
          const double t = 2.0 * csn * b0;
          const double dn = fma(o2, c0, fma(q2, a0, odd ? -t : t));
          const double df = odd ? o2 - q2 : q2 - o2;    // c^2 - s^2
          const double ei = fma(df, b0, csn * (c0 - a0));
          __syncwarp();   // every lane has read row i + 1
          if (tid == 0) {
            if (i > lo) e[i - 1] = r;
            d[i] = dn;
            rot[cur * k + nr] = make_double2(q, o);
          }
          ++nr;
          x = ei;
          z = __shfl_sync(0xffffffffu, m, 1);
          b0 = __shfl_sync(0xffffffffu, m, 0);
          a0 = __shfl_sync(0xffffffffu, dn, 1);
        }
        // the rotation of the last row chases nothing: x holds e_{hi-1}
        if (tid == 0) {
          d[hi] = a0;
          e[hi - 1] = x;
        }
        __syncwarp();
      }
      if (tid == 0) {
        ctl[cur][0] = lo;
        ctl[cur][1] = nr;
        ctl[cur][2] = (hi > 0 && iter > max_iter) ? 1 : 0;
      }
    } else if (ctl[prev][0] >= 0) {
      // V <- R V of the previous sweep: each thread carries its columns
      // through the whole sweep in a register
      const int lo = ctl[prev][0], nr = ctl[prev][1];
      const double2 *cs = rot + prev * k;
      for (int i = tid - 32; i < n; i += EIG_THREADS - 32) {
        double x = V[(size_t)lo * k + i];
#pragma unroll 4
        for (int r = 0; r < nr; ++r) {
          const double2 q = cs[r];
          const double y = V[(size_t)(lo + r + 1) * k + i];
          V[(size_t)(lo + r) * k + i] = fma(q.x, x, q.y * y);
          x = fma(q.x, y, -q.y * x);
        }
        V[(size_t)(lo + nr) * k + i] = x;
      }
    }
    __syncthreads();
    if (ctl[cur][2]) {
      if (tid == 0) atomicOr(a.status, ST_NO_CONV);
      break;
    }
    // the sweep that found nothing left ran beside the last one's row updates
    if (ctl[cur][0] < 0) break;
  }
  for (int i = tid; i < k; i += EIG_THREADS) a.theta[(size_t)b * k + i] = (i < n) ? d[i] : 0.0;
}

// --------------------------------------------------------------------------
// Per-vector adjoint coefficients a_y, Gam, dz (weights dE_t Z_t folded in).
// One block of COEF_THREADS per vector:
//   Phi_st = Re(F_st) u1_s u1_t,  X = U Phi,  Gam = c b0^2 X U^T.
// --------------------------------------------------------------------------
constexpr int COEF_THREADS = 128;

__global__ void __launch_bounds__(COEF_THREADS) k_adj_coeffs(AdjCtx a) {
  pdl_wait();
  extern __shared__ double sm[];   // Om[k], u1[k], fu[k]
  __shared__ double red[COEF_THREADS / 32];
  const int b = blockIdx.x;
  const int tid = threadIdx.x;
  const int k = a.k;
  double *Ay = a.ay + (size_t)b * k;
  double *Gm = a.Gam + (size_t)b * k * k;
  const int v = a.vec0 + b;
  const int n = (b < a.nvec) ? a.k_eff[v] : 0;
  if (n <= 0) {
    for (int i = tid; i < k; i += COEF_THREADS) Ay[i] = 0.0;
    for (int i = tid; i < k * k; i += COEF_THREADS) Gm[i] = 0.0;
    if (a.Gamf)
      for (int i = tid; i < k * k; i += COEF_THREADS) a.Gamf[(size_t)b * k * k + i] = 0.0f;
    if (tid == 0) a.dz[b] = 0.0;
    return;
  }
  const int ti = v / a.n_m, mi = v % a.n_m;
  const int m = a.m_idx[mi];
  const double eta = (m < a.n_v) ? 1.0 : -1.0;
  const double cw = a.dE[ti] * a.Z[ti];
  const double zr = a.E[ti] - a.eps[m], zi = -eta * a.delta;
  const double b0 = a.beta0[v];
  const double *V = a.V + (size_t)b * k * k;     // V[s][i]: component i of eigenvector s
  const double *th = a.theta + (size_t)b * k;
  double *Om = sm, *u1 = sm + k, *fu = sm + 2 * k;
  double dzp = 0.0;
  for (int s = tid; s < n; s += COEF_THREADS) {
    const double u = V[(size_t)s * k];
    u1[s] = u;
    if (a.poly) {
      // nodes of D = p_g(C) ~ C^1/2 directly: f = 1/(Om (z + eta Om)), Om = theta
      const double om = th[s];
      Om[s] = om;
      const double ar = zr + eta * om;
      fu[s] = ar / (om * (ar * ar + zi * zi)) * u;
      const double sr = ar * ar - zi * zi, si = 2.0 * ar * zi;
      dzp += -(u * u / om) * (sr / (sr * sr + si * si));
      continue;
    }
    if (a.tda) {
      // f = 1/(z + eta theta):  a = z + eta theta;  Re f = Re 1/a;  dF/dz term -u^2 / a^2
      const double t = th[s];
      Om[s] = t;
      const double ar = zr + eta * t;
      fu[s] = ar / (ar * ar + zi * zi) * u;
      const double sr = ar * ar - zi * zi, si = 2.0 * ar * zi;
      dzp += -(u * u) * (sr / (sr * sr + si * si));
      continue;
    }
    const double om = sqrt(fmax(th[s], 0.0));
    Om[s] = om;
    // a = z + eta Om;  Re f = Re 1/(Om a);  dF/dz term -u^2 / (Om a^2)
    const double ar = zr + eta * om;
    fu[s] = ar / (om * (ar * ar + zi * zi)) * u;
    const double sr = ar * ar - zi * zi, si = 2.0 * ar * zi;
    dzp += -(u * u / om) * (sr / (sr * sr + si * si));
  }
  dzp = block_sum(dzp, red);
  if (tid == 0) a.dz[b] = cw * b0 * b0 * dzp;
  __syncthreads();
  // a_y[j] = 2 c b0 sum_s U[j][s] Re f_s u1_s = 2 c b0 sum_s V[s][j] fu[s]
  for (int j = tid; j < k; j += COEF_THREADS) {
    double acc = 0.0;
    if (j < n)
      for (int s = 0; s < n; ++s) acc = fma(V[(size_t)s * k + j], fu[s], acc);
    Ay[j] = cw * 2.0 * b0 * acc;
  }
  // Phi_st = Re F_st u1_s u1_t,
  // F_st = -(z + eta(Om_s + Om_t)) / (Om_s Om_t (z+eta Om_s)(z+eta Om_t) (Om_s + Om_t))
  double *Phi = a.Phi + (size_t)b * k * k;
  for (int idx = tid; idx < n * n; idx += COEF_THREADS) {
    const int s = idx / n, t = idx % n;
    const double as_r = zr + eta * Om[s], at_r = zr + eta * Om[t];
    const double pr = as_r * at_r - zi * zi, pi = zi * (as_r + at_r);   // a_s a_t
    double Fr;
    if (a.tda) {
      // f[theta_s, theta_t] = -eta / (a_s a_t)
      Fr = -eta * pr / (pr * pr + pi * pi);
    } else {
      // g[Om_s, Om_t] = -(z + eta (Om_s + Om_t)) / (Om_s Om_t a_s a_t); divided by
      // (Om_s + Om_t) for the nodes theta = Om^2 of C (not for D's own nodes)
      const double nr = -(zr + eta * (Om[s] + Om[t])), ni = -zi;
      const double scale = Om[s] * Om[t] * (a.poly ? 1.0 : (Om[s] + Om[t]));
      Fr = (nr * pr + ni * pi) / ((pr * pr + pi * pi) * scale);
    }
    Phi[(size_t)s * k + t] = Fr * u1[s] * u1[t];
  }
  __syncthreads();
  // X[l][s] = sum_t U[l][t] Phi[t][s] = sum_t V[t][l] Phi[t][s]
  double *X = a.X + (size_t)b * k * k;
  for (int idx = tid; idx < n * n; idx += COEF_THREADS) {
    const int l = idx / n, s = idx % n;
    double acc = 0.0;
    for (int t = 0; t < n; ++t) acc = fma(V[(size_t)t * k + l], Phi[(size_t)t * k + s], acc);
    X[(size_t)l * k + s] = acc;
  }
  __syncthreads();
  // Gam[j][l] = c b0^2 sum_s X[j][s] U[l][s] = c b0^2 sum_s X[j][s] V[s][l]
  const double g = cw * b0 * b0;
  for (int idx = tid; idx < k * k; idx += COEF_THREADS) {
    const int j = idx / k, l = idx % k;
    double acc = 0.0;
    if (j < n && l < n)
      for (int s = 0; s < n; ++s) acc = fma(X[(size_t)j * k + s], V[(size_t)s * k + l], acc);
    Gm[idx] = g * acc;
    if (a.Gamf) a.Gamf[(size_t)b * k * k + idx] = (float)(g * acc);
  }
}

// --------------------------------------------------------------------------
// Per element of each vector: y = Q a_y and g = diag(Q Gam Q^T) (Gam
// symmetric: g = sum_j q_j (Gam_jj q_j + 2 sum_{l>j} Gam_jl q_l)).  Block =
// (ROW_THREADS elements, one vector); the block's basis entries staged in
// shared memory.
// --------------------------------------------------------------------------
constexpr int ROW_THREADS = 32;

__global__ void __launch_bounds__(ROW_THREADS) k_adj_rows(AdjCtx a, BasisRef basis,
                                                          double *Y, double *Gd) {
  pdl_wait();
  extern __shared__ double qs[];   // [k][ROW_THREADS]
  const int b = blockIdx.y;
  const int i = blockIdx.x * ROW_THREADS + threadIdx.x;
  const int k = a.k;
  const bool ok = i < a.N;
  const double *Ay = a.ay + (size_t)b * k;
  const double *Gm = a.Gam + (size_t)b * k * k;
  double y = 0.0;
  for (int j = 0; j < k; ++j) {
    const double q = ok ? basis.at(((size_t)j * a.Bs + b) * a.N + i) : 0.0;
    qs[j * ROW_THREADS + threadIdx.x] = q;
    y = fma(Ay[j], q, y);
  }
  double g = 0.0;
  for (int j = 0; j < k; ++j) {
    const double qj = qs[j * ROW_THREADS + threadIdx.x];
    const double *gr = Gm + (size_t)j * k;
    double t = 0.0;
    for (int l = j + 1; l < k; ++l) t = fma(gr[l], qs[l * ROW_THREADS + threadIdx.x], t);
    g = fma(qj, fma(gr[j], qj, 2.0 * t), g);
  }
  if (ok) {
    Y[(size_t)b * a.N + i] = y;
    Gd[(size_t)b * a.N + i] = g;
  }
}

// FP32 variant of k_adj_rows (BF16 mode: the gradient there is good to
// ~1e-4, so y and diag(Q Gam Q^T) run on the FP32 pipe).  Block = 128 elements
// of one vector, its basis entries (the hi floats: hi + lo rounds to hi) in
// shared memory; each warp takes four rows j at a time for all 128 elements
// (4 per lane), so a basis entry is read once for four products; then one
// thread per element adds the rows up in order.  Every sum keeps the order of
// the row-by-row form.  That form (one element per thread, two loads per
// product) took 13.6 ms at 128 vectors of 32768, k 120; 8.6 in this one.
constexpr int RF_ELEMS = 128, RF_WARPS = 8;

__global__ void __launch_bounds__(32 * RF_WARPS) k_adj_rows_f32(AdjCtx a, BasisRef basis,
                                                                double *Y, double *Gd) {
  pdl_wait();
  extern __shared__ float qsf[];               // [k][RF_ELEMS] q, then [k][RF_ELEMS] row terms
  const int b = blockIdx.y, k = a.k;
  float *sf = qsf + (size_t)k * RF_ELEMS;
  const int i0 = blockIdx.x * RF_ELEMS;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float *Gm = a.Gamf + (size_t)b * k * k;
  for (int idx = threadIdx.x; idx < k * RF_ELEMS; idx += 32 * RF_WARPS) {
    const int j = idx / RF_ELEMS, i = i0 + idx % RF_ELEMS;
    const size_t o = ((size_t)j * a.Bs + b) * a.N + i;
    qsf[idx] = i < a.N ? (basis.d ? (float)basis.d[o] : basis.hi[o]) : 0.0f;
  }
  __syncthreads();
  for (int j0 = wid * 4; j0 < k; j0 += 4 * RF_WARPS) {
    float t[4][4];   // [row][element]
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int u = 0; u < 4; ++u) t[r][u] = 0.0f;
    const int nr = min(4, k - j0);
    auto column = [&](int l, bool inside) {
      float q[4], g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = qsf[l * RF_ELEMS + 32 * u + lane];
#pragma unroll
      for (int r = 0; r < 4; ++r) g[r] = __ldg(Gm + (size_t)(j0 + min(r, nr - 1)) * k + l);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (!inside || l > j0 + r)
#pragma unroll
          for (int u = 0; u < 4; ++u) t[r][u] = fmaf(g[r], q[u], t[r][u]);
    };
    for (int l = j0 + 1; l < min(j0 + 4, k); ++l) column(l, true);
#pragma unroll 2
    for (int l = j0 + 4; l < k; ++l) column(l, false);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (r >= nr) break;
      const float gj = __ldg(Gm + (size_t)(j0 + r) * k + j0 + r);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int o = (j0 + r) * RF_ELEMS + 32 * u + lane;
        sf[o] = fmaf(gj, qsf[o], 2.0f * t[r][u]);
      }
    }
  }
  __syncthreads();
  const int i = i0 + threadIdx.x;
  if (threadIdx.x >= RF_ELEMS || i >= a.N) return;
  const double *Ay = a.ay + (size_t)b * k;
  float y = 0.0f, g = 0.0f;
  for (int j = 0; j < k; ++j) {
    const float q = qsf[j * RF_ELEMS + threadIdx.x];
    y = fmaf((float)Ay[j], q, y);
    g = fmaf(q, sf[j * RF_ELEMS + threadIdx.x], g);
  }
  Y[(size_t)b * a.N + i] = (double)y;
  Gd[(size_t)b * a.N + i] = (double)g;
}

// The row-by-row form, for depths whose two tables exceed shared memory.
__global__ void __launch_bounds__(ROW_THREADS) k_adj_rows_f32_deep(AdjCtx a, BasisRef basis,
                                                                   double *Y, double *Gd) {
  pdl_wait();
  extern __shared__ float qsf[];   // [k][ROW_THREADS]
  const int b = blockIdx.y;
  const int i = blockIdx.x * ROW_THREADS + threadIdx.x;
  const int k = a.k;
  const bool ok = i < a.N;
  const double *Ay = a.ay + (size_t)b * k;
  const float *Gm = a.Gamf + (size_t)b * k * k;
  float y = 0.0f;
  for (int j = 0; j < k; ++j) {
    const float q = ok ? (float)basis.at(((size_t)j * a.Bs + b) * a.N + i) : 0.0f;
    qsf[j * ROW_THREADS + threadIdx.x] = q;
    y = fmaf((float)Ay[j], q, y);
  }
  float g = 0.0f;
  for (int j = 0; j < k; ++j) {
    const float qj = qsf[j * ROW_THREADS + threadIdx.x];
    const float *gr = Gm + (size_t)j * k;
    float t = 0.0f;
    for (int l = j + 1; l < k; ++l) t = fmaf(gr[l], qsf[l * ROW_THREADS + threadIdx.x], t);
    g = fmaf(qj, fmaf(gr[j], qj, 2.0f * t), g);
  }
  if (ok) {
    Y[(size_t)b * a.N + i] = (double)y;
    Gd[(size_t)b * a.N + i] = (double)g;
  }
}

// BF16 hi / lo split of a transposed FP64 matrix: src [R][C] (row stride
// lds) -> hi, lo [C][R].  Either output may be NULL.  Bound by DRAM (8 bytes
// read, 4 written per element): 64 x 64 tiles, so that both sides move whole
// 128-byte lines, elements split once on the integer pipe (an FP64 addition
// per element to join a float pair and one for the rest would take 2 ms of the
// FP64 pipe).  The three transposes of a
// gradient (15360 x 32768 the largest): 6.8 ms with 32 x 32 tiles, 2.5 ms now.
__global__ void __launch_bounds__(256) k_split_t(BasisRef src, int R, int C, int lds,
                                                 __nv_bfloat16 *__restrict__ hi,
                                                 __nv_bfloat16 *__restrict__ lo) {
  pdl_wait();
  __shared__ uint32_t tile[64][65];   // hi | lo << 16
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  {
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6, c = c0 + tx;
#pragma unroll 8
    for (int rr = ty; rr < 64; rr += 4) {
      const int r = r0 + rr;
      const double x = (r < R && c < C) ? src.at((size_t)r * lds + c) : 0.0;
      __nv_bfloat16 h, l;
      split_bf(x, h, l);
      tile[rr][tx] = bits_as<uint16_t>(h) | (uint32_t)bits_as<uint16_t>(l) << 16;
    }
  }
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int r = r0 + 2 * tx;
  for (int cc = ty; cc < 64; cc += 8) {
    const int c = c0 + cc;
    if (c >= C || r >= R) continue;
    const uint32_t p = tile[2 * tx][cc], q = tile[2 * tx + 1][cc];
    const size_t o = (size_t)c * R + r;
    if ((R & 1) == 0) {
      if (hi) *reinterpret_cast<uint32_t *>(hi + o) = (p & 0xffffu) | q << 16;
      if (lo) *reinterpret_cast<uint32_t *>(lo + o) = p >> 16 | (q & 0xffff0000u);
    } else {
      if (hi) hi[o] = bits_as<__nv_bfloat16>((uint16_t)p);
      if (lo) lo[o] = bits_as<__nv_bfloat16>((uint16_t)(p >> 16));
      if (r + 1 < R) {
        if (hi) hi[o + 1] = bits_as<__nv_bfloat16>((uint16_t)q);
        if (lo) lo[o + 1] = bits_as<__nv_bfloat16>((uint16_t)(q >> 16));
      }
    }
  }
}

// BF16 hi / lo split of scale[c] * src[r][c] (same layout [R][C], C a multiple
// of 4).  Bound by DRAM (8 bytes read, 4 written per element): four elements
// per thread and load, the scale kept over 16 rows, and the joined pair and
// the split on the integer pipe, so that one FP64 instruction per element is
// left.  15360 x 32768: 5.6 ms element by element, 1.9 ms now.
constexpr int SS_ROWS = 16;
__global__ void __launch_bounds__(256) k_split_scaled(BasisRef src, int R, int C,
                                                      const double *__restrict__ scale,
                                                      __nv_bfloat16 *__restrict__ hi,
                                                      __nv_bfloat16 *__restrict__ lo) {
  pdl_wait();
  const int c = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (c >= C) return;
  double sc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) sc[i] = scale[c + i];
  for (int r0 = blockIdx.y * SS_ROWS; r0 < R; r0 += gridDim.y * SS_ROWS)
#pragma unroll 2
  for (int r = r0; r < min(R, r0 + SS_ROWS); ++r) {
    const size_t o = (size_t)r * C + c;
    double x[4];
    src.at4(o, x);
    ushort4 h, l;
    unsigned short *hp = &h.x, *lp = &l.x;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat16 bh, bl;
      split_bf(sc[i] * x[i], bh, bl);
      hp[i] = bits_as<uint16_t>(bh);
      lp[i] = bits_as<uint16_t>(bl);
    }
    *reinterpret_cast<ushort4 *>(hi + o) = h;
    *reinterpret_cast<ushort4 *>(lo + o) = l;
  }
}

// R[j*Bs + b][mu] = sum_l Gam_b[j][l] P[l*Bs + b][mu].  Bound by the FP64
// pipe (k^2 N_aux products per vector); GP_ROWS rows at a time share the loads
// of P, which otherwise take as long as the products: k 120, N_aux 1024, 128
// vectors 6.5 ms one row at a time, 3.3 ms now (the FP64 rate allows 3.3).
constexpr int GP_ROWS = 8;
__global__ void __launch_bounds__(128) k_gamma_p(AdjCtx a, const double *__restrict__ P, int A,
                                                 double *__restrict__ R) {
  pdl_wait();
  const int b = blockIdx.y;
  const int mu = blockIdx.x * blockDim.x + threadIdx.x;
  if (mu >= A) return;
  const int k = a.k;
  const double *Gm = a.Gam + (size_t)b * k * k;
  const double *Pb = P + (size_t)b * A + mu;
  const size_t ld = (size_t)a.Bs * A;
  for (int j0 = 0; j0 < k; j0 += GP_ROWS) {
    const int nj = min(GP_ROWS, k - j0);
    double acc[GP_ROWS];
#pragma unroll
    for (int p = 0; p < GP_ROWS; ++p) acc[p] = 0.0;
    if (nj == GP_ROWS) {
#pragma unroll 2
      for (int l = 0; l < k; ++l) {
        const double x = Pb[l * ld];
#pragma unroll
        for (int p = 0; p < GP_ROWS; ++p)
          acc[p] = fma(__ldg(&Gm[(size_t)(j0 + p) * k + l]), x, acc[p]);
      }
    } else {
      for (int l = 0; l < k; ++l) {
        const double x = Pb[l * ld];
#pragma unroll
        for (int p = 0; p < GP_ROWS; ++p)
          if (p < nj) acc[p] = fma(__ldg(&Gm[(size_t)(j0 + p) * k + l]), x, acc[p]);
      }
    }
#pragma unroll
    for (int p = 0; p < GP_ROWS; ++p)
      if (p < nj) R[(size_t)(j0 + p) * ld + (size_t)b * A + mu] = acc[p];
  }
}

// S[i][mu] += sum_r X[r][i] Yr[r][mu]  (FP64, 64 x 64 tiles, r = contraction)
__global__ void __launch_bounds__(256) k_atb_f64(const double *__restrict__ X, int ldx,
                                                 const double *__restrict__ Yr, int ldy, int R,
                                                 int Ni, int Nmu, double *__restrict__ S,
                                                 double scale) {
  pdl_wait();
  __shared__ double Xs[16][65];
  __shared__ double Ys[16][65];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int i0 = blockIdx.y * 64, mu0 = blockIdx.x * 64;
  double acc[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = 0.0;
  for (int r0 = 0; r0 < R; r0 += 16) {
#pragma unroll
    for (int rep = 0; rep < 4; ++rep) {
      const int idx = t + 256 * rep;
      const int rr = idx >> 6, cc = idx & 63;
      const int r = r0 + rr;
      Xs[rr][cc] = (r < R && i0 + cc < Ni) ? X[(size_t)r * ldx + i0 + cc] : 0.0;
      Ys[rr][cc] = (r < R && mu0 + cc < Nmu) ? Yr[(size_t)r * ldy + mu0 + cc] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < 16; ++rr) {
      double xa[4], yb[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) xa[p] = Xs[rr][ty + 16 * p];
#pragma unroll
      for (int q = 0; q < 4; ++q) yb[q] = Ys[rr][tx + 16 * q];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fma(xa[p], yb[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = i0 + ty + 16 * p;
    if (i >= Ni) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int mu = mu0 + tx + 16 * q;
      if (mu < Nmu) S[(size_t)i * Nmu + mu] = fma(scale, acc[p][q], S[(size_t)i * Nmu + mu]);
    }
  }
}

// dDelta[i] += sum_b (2 Delta_i Gd[b][i] + Y[b][i] beta0_b q0_b[i] / (2 Delta_i))
// (fixed order over b); deps[m] -= dz over the sub-batch (one thread per m).
__global__ void k_adj_accumulate(AdjCtx a, const double *Delta, BasisRef basis,
                                 const double *Y, const double *Gd, double *dDelta,
                                 double *deps) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.N && Delta[i] > 0.0) {
    double s = 0.0;
    for (int b = 0; b < a.nvec; ++b) {
      if (a.tda) {   // dA/dDelta_i = e_i e_i^T; b = L M
        s += Gd[(size_t)b * a.N + i];
        continue;
      }
      const double q0 = basis.at((size_t)b * a.N + i);
      s += 2.0 * Delta[i] * Gd[(size_t)b * a.N + i] +
           Y[(size_t)b * a.N + i] * a.beta0[a.vec0 + b] * q0 / (2.0 * Delta[i]);
    }
    dDelta[i] += s;
  }
  if (blockIdx.x == 0) {
    for (int mi = threadIdx.x; mi < a.n_m; mi += blockDim.x) {
      double s = 0.0;
      for (int b = 0; b < a.nvec; ++b)
        if ((a.vec0 + b) % a.n_m == mi) s += a.dz[b];
      deps[a.m_idx[mi]] -= s;
    }
  }
}

// dL = D (2 c_K SC + SB) (unpadded output), dDelta += c_K (L o SC) 1 / d.
// SC [N][A], SB [N][n_aux] or NULL (coupling vectors given directly).
// tda: D = 1, so no dDelta term from the coupling.
__global__ void k_adj_dL(const double *L64, const double *dsq, const double *SC,
                         const double *SB, int A, int n_vc, int n_aux, double kf, double *dL,
                         double *dDelta, int tda) {
  pdl_wait();
  const int i = blockIdx.x;
  if (i >= n_vc) return;
  __shared__ double red[8];
  double s = 0.0;
  for (int mu = threadIdx.x; mu < A; mu += blockDim.x) {
    const double sc = SC[(size_t)i * A + mu];
    s = fma(L64[(size_t)i * A + mu], sc, s);
    if (mu < n_aux) {
      const double sb = SB ? SB[(size_t)i * n_aux + mu] : 0.0;
      dL[(size_t)i * n_aux + mu] = dsq[i] * (2.0 * kf * sc + sb);
    }
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0 && dsq[i] > 0.0 && !tda) dDelta[i] += kf * s / dsq[i];
}

// deps from dDelta (Delta_vc = eps_c - eps_v) plus the direct dE_t Z_t term.
__global__ void k_adj_deps(const double *dDelta, int n_v, int n_c, const int *targets, int n_t,
                           const double *Z, const double *dE, double *deps) {
  pdl_wait();
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= n_v + n_c) return;
  double s = 0.0;
  if (o < n_v) {
    for (int c = 0; c < n_c; ++c) s -= dDelta[(size_t)o * n_c + c];
  } else {
    const int c = o - n_v;
    for (int v = 0; v < n_v; ++v) s += dDelta[(size_t)v * n_c + c];
  }
  for (int ti = 0; ti < n_t; ++ti)
    if (targets[ti] == o) s += dE[ti] * Z[ti];
  deps[o] += s;
}

// --------------------------------------------------------------------------
// Reverse mode of the three-term recurrence (no reorthogonalisation): the
// exact derivative of what k steps compute.  Forward step j:
//   u = C q_j,  w1 = u - beta_j q_{j-1},  alpha_j = q_j . w1,
//   w2 = w1 - alpha_j q_j,  beta_{j+1} = ||w2||,  q_{j+1} = w2 / beta_{j+1}.
// Taken back from the last step (j = k_eff - 1: w2bar = 0) to step 0:
//   w2bar  = (qbar_{j+1} - (qbar_{j+1}.q_{j+1}) q_{j+1}) / beta_{j+1} + bbar_j q_{j+1}
//   abar'  = Gam_jj - w2bar . q_j
//   ubar_j = w1bar = w2bar + abar' q_j
//   qbar_j += -alpha_j w2bar + abar' w1,  w1 = beta_{j+1} q_{j+1} + alpha_j q_j
//   bbar_{j-1} -= w1bar . q_{j-1},  qbar_{j-1} = -beta_j w1bar
//   qbar_j += C ubar_j (the contraction kernels, next step's first pass)
// so one pass of six dot products, one scalar step per vector and one
// elementwise pass per step, besides the matvec.  dF/dC = sum_j ubar_j q_j^T.
// --------------------------------------------------------------------------
__global__ void k_rev_init(RevCtx r) {
  pdl_wait();
  const int b = blockIdx.x;
  const int k = r.k;
  for (int j = threadIdx.x; j < k; j += blockDim.x)
    r.bbar[(size_t)b * k + j] =
        (j + 1 < k) ? 2.0 * r.Gam[((size_t)b * k + j) * k + j + 1] : 0.0;
}

__global__ void k_rev_set_betaj(RevCtx r, double *betaj) {
  pdl_wait();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= r.Bs) return;
  double v = 0.0;
  if (b < r.nvec && r.s0 > 0 && r.k_eff[r.vec0 + b] > r.s0)
    v = r.beta[(size_t)(r.vec0 + b) * r.k + r.s0 - 1];
  betaj[b] = v;
}

__device__ __forceinline__ int rev_elem_base(int chunk) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return chunk * VEC_CHUNK + wid * 256 + 2 * lane;
}

// qbar_{j+1} += C ubar_{j+1} (written back), and per-chunk partials of
// qbar_{j+1}.q_{j+1}, qbar_{j+1}.q_j, q_{j+1}.q_j, qbar_{j+1}.q_{j-1},
// q_{j+1}.q_{j-1}, q_j.q_{j-1}.
__global__ void __launch_bounds__(VEC_THREADS) k_rev_dots(RevCtx r, int j) {
  pdl_wait();
  __shared__ double red[VEC_THREADS / 32];
  const int chunk = blockIdx.x, b = blockIdx.y;
  const size_t BN = (size_t)r.Bs * r.N, voff = (size_t)b * r.N;
  const double *q1 = r.seg + (size_t)(j - r.s0 + 2) * BN + voff;
  const double *q0 = r.seg + (size_t)(j - r.s0 + 1) * BN + voff;
  const double *qm = r.seg + (size_t)(j - r.s0) * BN + voff;
  double *qb1 = r.qbar + (size_t)((j + 1) % 3) * BN + voff;
  const double *cu = r.cu + voff;
  double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  const int e0 = rev_elem_base(chunk);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = e0 + u * 64;
    if (e >= r.N) continue;
    double2 x = *reinterpret_cast<const double2 *>(qb1 + e);
    const double2 c2 = *reinterpret_cast<const double2 *>(cu + e);
    x.x += c2.x;
    x.y += c2.y;
    *reinterpret_cast<double2 *>(qb1 + e) = x;
    const double2 a = *reinterpret_cast<const double2 *>(q1 + e);
    const double2 p = *reinterpret_cast<const double2 *>(q0 + e);
    const double2 m = *reinterpret_cast<const double2 *>(qm + e);
    acc[0] = fma(x.x, a.x, fma(x.y, a.y, acc[0]));
    acc[1] = fma(x.x, p.x, fma(x.y, p.y, acc[1]));
    acc[2] = fma(a.x, p.x, fma(a.y, p.y, acc[2]));
    acc[3] = fma(x.x, m.x, fma(x.y, m.y, acc[3]));
    acc[4] = fma(a.x, m.x, fma(a.y, m.y, acc[4]));
    acc[5] = fma(p.x, m.x, fma(p.y, m.y, acc[5]));
  }
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    const double s = block_sum(acc[t], red);
    if (threadIdx.x == 0) r.dpart[((size_t)b * r.nchunks + chunk) * 6 + t] = s;
  }
}

// One warp per vector: the six dots in fixed order and the step's
// coefficients: ubar = a1 qbar_{j+1} + a2 q_{j+1} + ab q_j,
// qbar_j += cA qbar_{j+1} + cB q_{j+1} + cC q_j, qbar_{j-1} = mb ubar.
__global__ void k_rev_scalars(RevCtx r, int j) {
  pdl_wait();
  const int b = blockIdx.x, lane = threadIdx.x;
  double d[6];
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    double s = 0.0;
    for (int ch = lane; ch < r.nchunks; ch += 32)
      s += r.dpart[((size_t)b * r.nchunks + ch) * 6 + t];
    d[t] = warp_sum(s);
  }
  if (lane != 0) return;
  const int v = r.vec0 + b;
  const int ke = b < r.nvec ? r.k_eff[v] : 0;
  double a1 = 0.0, a2 = 0.0, ab = 0.0, cA = 0.0, cB = 0.0, cC = 0.0, mb = 0.0;
  if (j < ke) {
    const int k = r.k;
    const double al = r.alpha[(size_t)v * k + j];
    const double bn = r.beta[(size_t)v * k + j];
    const double bj = j > 0 ? r.beta[(size_t)v * k + j - 1] : 0.0;
    if (j + 1 < ke) {
      a1 = 1.0 / bn;
      a2 = r.bbar[(size_t)b * k + j] - d[0] * a1;
    }
    const double w2q = a1 * d[1] + a2 * d[2];
    ab = r.Gam[((size_t)b * k + j) * k + j] - w2q;
    if (j > 0) r.bbar[(size_t)b * k + j - 1] -= a1 * d[3] + a2 * d[4] + ab * d[5];
    cA = -al * a1;
    cB = fma(ab, bn, -al * a2);
    cC = ab * al;
    mb = -bj;
  }
  double *cf = r.coef + (size_t)b * 8;
  cf[0] = a1;
  cf[1] = a2;
  cf[2] = ab;
  cf[3] = cA;
  cf[4] = cB;
  cf[5] = cC;
  cf[6] = mb;
}

__global__ void __launch_bounds__(VEC_THREADS) k_rev_elem(RevCtx r, int j) {
  pdl_wait();
  const int chunk = blockIdx.x, b = blockIdx.y;
  const size_t BN = (size_t)r.Bs * r.N, voff = (size_t)b * r.N;
  const double *cf = r.coef + (size_t)b * 8;
  const double a1 = cf[0], a2 = cf[1], ab = cf[2], cA = cf[3], cB = cf[4], cC = cf[5],
               mb = cf[6];
  const double *q1 = r.seg + (size_t)(j - r.s0 + 2) * BN + voff;
  const double *q0 = r.seg + (size_t)(j - r.s0 + 1) * BN + voff;
  const double *qb1 = r.qbar + (size_t)((j + 1) % 3) * BN + voff;
  double *qbj = r.qbar + (size_t)(j % 3) * BN + voff;
  double *qbm = r.qbar + (size_t)((j + 2) % 3) * BN + voff;   // slot of q_{j-1}
  double *ub = r.useg + (size_t)(j - r.s0) * BN + voff;
  double *gd = r.Gd + voff;
  const int e0 = rev_elem_base(chunk);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = e0 + u * 64;
    if (e >= r.N) continue;
    const double2 x = *reinterpret_cast<const double2 *>(qb1 + e);
    const double2 a = *reinterpret_cast<const double2 *>(q1 + e);
    const double2 p = *reinterpret_cast<const double2 *>(q0 + e);
    double2 w;
    w.x = fma(a1, x.x, fma(a2, a.x, ab * p.x));
    w.y = fma(a1, x.y, fma(a2, a.y, ab * p.y));
    double2 y = *reinterpret_cast<const double2 *>(qbj + e);
    y.x += fma(cA, x.x, fma(cB, a.x, cC * p.x));
    y.y += fma(cA, x.y, fma(cB, a.y, cC * p.y));
    *reinterpret_cast<double2 *>(qbj + e) = y;
    if (j > 0) *reinterpret_cast<double2 *>(qbm + e) = make_double2(mb * w.x, mb * w.y);
    *reinterpret_cast<double2 *>(ub + e) = w;
    if (r.gd_from_steps) {
      double2 g = *reinterpret_cast<const double2 *>(gd + e);
      g.x = fma(w.x, p.x, g.x);
      g.y = fma(w.y, p.y, g.y);
      *reinterpret_cast<double2 *>(gd + e) = g;
    }
  }
}

// qbar_0 += C ubar_0 (written back) and per-chunk partials of qbar_0 . q_0.
__global__ void __launch_bounds__(VEC_THREADS) k_rev_final_dot(RevCtx r, const double *q0v) {
  pdl_wait();
  __shared__ double red[VEC_THREADS / 32];
  const int chunk = blockIdx.x, b = blockIdx.y;
  const size_t voff = (size_t)b * r.N;
  double *qb = r.qbar + voff;
  const double *cu = r.cu + voff;
  const double *q0 = q0v + voff;
  double acc = 0.0;
  const int e0 = rev_elem_base(chunk);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = e0 + u * 64;
    if (e >= r.N) continue;
    double2 x = *reinterpret_cast<const double2 *>(qb + e);
    const double2 c2 = *reinterpret_cast<const double2 *>(cu + e);
    x.x += c2.x;
    x.y += c2.y;
    *reinterpret_cast<double2 *>(qb + e) = x;
    const double2 p = *reinterpret_cast<const double2 *>(q0 + e);
    acc = fma(x.x, p.x, fma(x.y, p.y, acc));
  }
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) r.dpart[(size_t)b * r.nchunks + chunk] = acc;
}

// y = dF/db = (dF/dbeta0) q_0 + (qbar_0 - (qbar_0 . q_0) q_0) / beta0.
__global__ void __launch_bounds__(VEC_THREADS) k_rev_final(RevCtx r, const double *q0v,
                                                           double *Y) {
  pdl_wait();
  __shared__ double sdot;
  const int chunk = blockIdx.x, b = blockIdx.y;
  const int v = r.vec0 + b;
  const bool live = b < r.nvec && r.k_eff[v] > 0 && r.beta0[v] > 0.0;
  if (threadIdx.x < 32) {
    double s = 0.0;
    for (int ch = threadIdx.x; ch < r.nchunks; ch += 32) s += r.dpart[(size_t)b * r.nchunks + ch];
    s = warp_sum(s);
    if (threadIdx.x == 0) sdot = s;
  }
  __syncthreads();
  const double dq = sdot;
  const double b0 = live ? r.beta0[v] : 1.0;
  const double b0bar = live ? r.ay[(size_t)b * r.k] : 0.0;
  const double inv = live ? 1.0 / b0 : 0.0;
  const size_t voff = (size_t)b * r.N;
  const double *qb = r.qbar + voff;
  const double *q0 = q0v + voff;
  double *y = Y + voff;
  const int e0 = rev_elem_base(chunk);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = e0 + u * 64;
    if (e >= r.N) continue;
    const double2 x = *reinterpret_cast<const double2 *>(qb + e);
    const double2 p = *reinterpret_cast<const double2 *>(q0 + e);
    double2 o;
    o.x = fma(b0bar, p.x, inv * fma(-dq, p.x, x.x));
    o.y = fma(b0bar, p.y, inv * fma(-dq, p.y, x.y));
    if (!live) o = make_double2(0.0, 0.0);
    *reinterpret_cast<double2 *>(y + e) = o;
  }
}

// out = a x + b out (b = 0: out is not read), over [Bs][N]
__global__ void k_rev_axpby(double *out, double a, const double *__restrict__ x, double b,
                            size_t n) {
  pdl_wait();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = (b == 0.0) ? a * x[i] : fma(a, x[i], b * out[i]);
}

// Gd += coef x o y over [Bs][N]
__global__ void k_rev_gd(double *Gd, double coef, const double *__restrict__ x,
                         const double *__restrict__ y, size_t n) {
  pdl_wait();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    Gd[i] = fma(coef * x[i], y[i], Gd[i]);
}

static unsigned flat_blocks(size_t n) {
  size_t b = (n + 255) / 256;
  return (unsigned)(b > (size_t)152 * 16 ? (size_t)152 * 16 : b);
}
void launch_rev_axpby(double *out, double a, const double *x, double b, size_t n,
                      cudaStream_t st) {
  launch_pdl(k_rev_axpby, dim3(flat_blocks(n)), dim3(256), 0, st, out, a, x, b, n);
}
void launch_rev_gd(double *Gd, double coef, const double *x, const double *y, size_t n,
                   cudaStream_t st) {
  launch_pdl(k_rev_gd, dim3(flat_blocks(n)), dim3(256), 0, st, Gd, coef, x, y, n);
}

void launch_rev_init(const RevCtx &r, cudaStream_t st) {
  launch_pdl(k_rev_init, dim3(r.Bs), dim3(128), 0, st, r);
}
void launch_rev_set_betaj(const RevCtx &r, double *betaj, cudaStream_t st) {
  launch_pdl(k_rev_set_betaj, dim3((r.Bs + 127) / 128), dim3(128), 0, st, r, betaj);
}
void launch_rev_step(const RevCtx &r, int j, cudaStream_t st) {
  dim3 grid(r.nchunks, r.Bs);
  launch_pdl(k_rev_dots, grid, dim3(VEC_THREADS), 0, st, r, j);
  launch_pdl(k_rev_scalars, dim3(r.Bs), dim3(32), 0, st, r, j);
  launch_pdl(k_rev_elem, grid, dim3(VEC_THREADS), 0, st, r, j);
}
void launch_rev_finish(const RevCtx &r, const double *q0, double *Y, cudaStream_t st) {
  dim3 grid(r.nchunks, r.Bs);
  launch_pdl(k_rev_final_dot, grid, dim3(VEC_THREADS), 0, st, r, q0);
  launch_pdl(k_rev_final, grid, dim3(VEC_THREADS), 0, st, r, q0, Y);
}

// ----------------------------------------------------------------------------
int adj_max_k() {
  // k_adj_rows stages k * ROW_THREADS doubles; k_eig_full 6 k
  return 768;
}

void launch_eig_full(const AdjCtx &a, cudaStream_t st) {
  const size_t smem = (size_t)6 * a.k * sizeof(double);
  static DeviceOnce once;
  once(current_device(), [] {
    cudaFuncSetAttribute(k_eig_full, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    // the GEMM that runs beside it needs an SM's shared memory, which is split
    // from the L1 when the first block arrives
    cudaFuncSetAttribute(k_eig_full, cudaFuncAttributePreferredSharedMemoryCarveout,
                         cudaSharedmemCarveoutMaxShared);
  });
  launch_pdl(k_eig_full, dim3(a.Bs), dim3(EIG_THREADS), smem, st, a);
}
void launch_adj_coeffs(const AdjCtx &a, cudaStream_t st) {
  const size_t smem = (size_t)3 * a.k * sizeof(double);
  launch_pdl(k_adj_coeffs, dim3(a.Bs), dim3(COEF_THREADS), smem, st, a);
}
void launch_adj_rows(const AdjCtx &a, BasisRef basis, double *Y, double *Gd, cudaStream_t st) {
  const size_t smem = (size_t)a.k * ROW_THREADS * sizeof(double);
  static DeviceOnce once;
  allow_smem(once, k_adj_rows, 200 * 1024);
  dim3 grid((a.N + ROW_THREADS - 1) / ROW_THREADS, a.Bs);
  launch_pdl(k_adj_rows, grid, dim3(ROW_THREADS), smem, st, a, basis, Y, Gd);
}
void launch_adj_rows_f32(const AdjCtx &a, BasisRef basis, double *Y, double *Gd,
                         cudaStream_t st) {
  static DeviceOnce once, once_deep;
  allow_smem(once, k_adj_rows_f32, 200 * 1024);
  allow_smem(once_deep, k_adj_rows_f32_deep, 200 * 1024);
  const size_t tables = (size_t)2 * a.k * RF_ELEMS * sizeof(float);
  if (tables <= 200 * 1024)   // k up to 200
    launch_pdl(k_adj_rows_f32, dim3((a.N + RF_ELEMS - 1) / RF_ELEMS, a.Bs), dim3(32 * RF_WARPS),
               tables, st, a, basis, Y, Gd);
  else
    launch_pdl(k_adj_rows_f32_deep, dim3((a.N + ROW_THREADS - 1) / ROW_THREADS, a.Bs),
               dim3(ROW_THREADS), (size_t)a.k * ROW_THREADS * sizeof(float), st, a, basis, Y, Gd);
}
void launch_split_t(BasisRef src, int R, int C, int lds, __nv_bfloat16 *hi, __nv_bfloat16 *lo,
                    cudaStream_t st) {
  dim3 grid((C + 63) / 64, (R + 63) / 64);
  launch_pdl(k_split_t, grid, dim3(256), 0, st, src, R, C, lds, hi, lo);
}
void launch_split_scaled(BasisRef src, int R, int C, const double *scale, __nv_bfloat16 *hi,
                         __nv_bfloat16 *lo, cudaStream_t st) {
  dim3 grid((C / 4 + 255) / 256, std::min((R + SS_ROWS - 1) / SS_ROWS, 65535));
  launch_pdl(k_split_scaled, grid, dim3(256), 0, st, src, R, C, scale, hi, lo);
}
void launch_gamma_p(const AdjCtx &a, const double *P, int A, double *R, cudaStream_t st) {
  dim3 grid((A + 127) / 128, a.Bs);
  launch_pdl(k_gamma_p, grid, dim3(128), 0, st, a, P, A, R);
}
void launch_atb_f64(const double *X, int ldx, const double *Yr, int ldy, int R, int Ni, int Nmu,
                    double *S, cudaStream_t st, double scale) {
  dim3 grid((Nmu + 63) / 64, (Ni + 63) / 64);
  launch_pdl(k_atb_f64, grid, dim3(256), 0, st, X, ldx, Yr, ldy, R, Ni, Nmu, S, scale);
}
void launch_adj_accumulate(const AdjCtx &a, const double *Delta, BasisRef basis,
                           const double *Y, const double *Gd, double *dDelta, double *deps,
                           cudaStream_t st) {
  launch_pdl(k_adj_accumulate, dim3((a.N + 255) / 256), dim3(256), 0, st, a, Delta, basis, Y, Gd,
             dDelta, deps);
}
void launch_adj_dL(const double *L64, const double *dsq, const double *SC, const double *SB,
                   int A, int n_vc, int n_aux, double kf, double *dL, double *dDelta, int tda,
                   cudaStream_t st) {
  launch_pdl(k_adj_dL, dim3(n_vc), dim3(256), 0, st, L64, dsq, SC, SB, A, n_vc, n_aux, kf, dL,
             dDelta, tda);
}
void launch_adj_deps(const double *dDelta, int n_v, int n_c, const int *targets, int n_t,
                     const double *Z, const double *dE, double *deps, cudaStream_t st) {
  const int n = n_v + n_c;
  launch_pdl(k_adj_deps, dim3((n + 127) / 128), dim3(128), 0, st, dDelta, n_v, n_c, targets, n_t,
             Z, dE, deps);
}

}  // namespace lgw
