// Spectral map of each Lanczos tridiagonal (Eq. 12-14), FP64.
//
// A k-step Lanczos on C from b gives T_k whose Gauss rule (nodes theta_j,
// weights ||b||^2 u_1j^2, u_1j the first components of T_k's eigenvectors)
// reproduces b^T f(C) b for polynomials f of degree < 2k.  Eq. 12 needs
// f(C) = C^-1/2 (z + eta C^1/2)^-1, i.e. the resolvent of D = C^1/2 with the
// weights divided by Omega:  Sigma_tm(omega) = -eta G(-eta z),
//   G(zeta) = sum_j wt_j / (zeta - Omega_j),  Omega_j = sqrt(theta_j),
//   wt_j = ||b||^2 u_1j^2 / Omega_j,
// the sum over poles of Eq. 11.  The fraction kernels evaluate that sum: it
// equals the continued fraction of the measure's Jacobi matrix (Eq. 14), has
// no serial chain over the depth, and needs no rebuild of that matrix.
//
// One block per start vector, one eigenvalue per thread.
#include <algorithm>

#include "lgw_internal.cuh"

namespace lgw {

// --------------------------------------------------------------------------
// Gauss rule of T_k.  theta_j is the (j+1)-th smallest eigenvalue.
//   1. FP32 bisection on the number of negative pivots of T - x (22 halvings
//      of the Gershgorin interval).  The computed count is the exact count of
//      a matrix within a few FP32 roundings of T, so theta_j lies within
//      2^-18 of the interval's width of the result.
//   2. FP64 Sturm counts at both ends of that bracket: they show that it
//      holds theta_j alone, or move and widen it.
//   3. Newton's method on p(x) = det(T - x) inside the bracket, p and p' from
//      the three-term recurrence of the trailing minors r_i (bottom row
//      first); its sign changes are the Sturm count, which narrows the
//      bracket at every evaluation.  While the bracket holds more than one
//      eigenvalue (clusters, ghosts of a recurrence without
//      reorthogonalisation), or where Newton's step leaves it, it is halved.
//   u_1j^2 = |r_1 / p'|, the product formula prod_i (theta_j - mu_i) /
//   prod_{i != j} (theta_j - theta_i) (mu: eigenvalues of T without its first
//   row and column), from the same last evaluation.
//
// What bounds it: GB300's FP64 pipe (2 lanes per SM clock).  Pure FP64
// bisection needs 60 counts of 3 operations per level and eigenvalue, and the
// separate weight recurrences 10 more; this needs 2 counts and about 3
// evaluations of 5 (21).  One warp per vector also left most of the chip
// idle at a few hundred vectors.  512 vectors, k = 200: 2.4 ms, against 22.6
// ms for one warp per vector, pure bisection and the Jacobi rebuild.
// --------------------------------------------------------------------------
constexpr int SPEC_THREADS = 256;
constexpr int SPEC_FP32_ITS = 22;
constexpr int SPEC_MAX_ITS = 160;

__device__ __forceinline__ bool finite_bits(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ int hi_abs(double p) { return __double2hiint(p) & 0x7fffffff; }

// The trailing minors r_i = det(T_{i:n} - x) from the last row up: p = r_0,
// r1 = r_1, dp = dp/dx (DERIV), all on one common scale, and the number of
// eigenvalues below x.  ab[i] = (a_i, b_i^2), b_i coupling rows i and i + 1.
// A zero minor takes the opposite sign of its predecessor at a magnitude that
// later minors cannot see.  Signs and magnitudes are tested on the integer
// pipe; the common power-of-two rescaling every eight levels is exact (a
// level grows the minors by less than 2^4 on a T of width below 2).
template <bool DERIV>
__device__ __forceinline__ void sturm_eval(const double2 *ab, int n, double x, double &p,
                                           double &dp, double &r1, int &count) {
  constexpr int kBig = (1023 + 400) << 20, kSmall = (1023 - 400) << 20;
  double p0 = 1.0, p1 = ab[n - 1].x - x, d0 = 0.0, d1 = -1.0;
  if (p1 == 0.0) p1 = -0x1p-900;
  int neg = __double2hiint(p1) < 0 ? 1 : 0, cnt = neg;
  int i = n - 2;
  while (i >= 0) {
    const int stop = max(-1, i - 8);
    for (; i > stop; --i) {
      const double2 v = ab[i];
      const double c = v.x - x;
      double p2 = fma(c, p1, -v.y * p0);
      if (DERIV) {
        const double d2 = fma(c, d1, fma(-v.y, d0, -p1));
        d0 = d1;
        d1 = d2;
      }
      if (((__double2hiint(p2) << 1) | __double2loint(p2)) == 0)
        p2 = neg ? 0x1p-900 : -0x1p-900;
      const int ng = __double2hiint(p2) < 0 ? 1 : 0;
      cnt += ng ^ neg;
      neg = ng;
      p0 = p1;
      p1 = p2;
    }
    const int m = max(hi_abs(p0), hi_abs(p1));
    if (max(m, DERIV ? hi_abs(d1) : 0) > kBig) {
      p0 *= 0x1p-400;
      p1 *= 0x1p-400;
      if (DERIV) {
        d0 *= 0x1p-400;
        d1 *= 0x1p-400;
      }
    } else if (m < kSmall) {
      p0 *= 0x1p+400;
      p1 *= 0x1p+400;
      if (DERIV) {
        d0 *= 0x1p+400;
        d1 *= 0x1p+400;
      }
    }
  }
  p = p1;
  r1 = p0;
  dp = d1;
  count = cnt;
}

// theta_j of the n x n scaled matrix ab (abf: the same about mid, in FP32), all
// of whose eigenvalues lie in [glo, ghi], w < ghi - glo < 1.1 w; wt = u_1j^2.
// The 32 lanes of a warp call it together; a lane without an eigenvalue
// (real == false) takes part in the loops only.
__device__ __noinline__ double eigenvalue(const double2 *ab, const float2 *abf, int n, int j,
                                          bool real, double glo, double ghi, double mid,
                                          double w, double &wt_out) {
  const double tol = 0x1p-50;
  // 1. FP32 bracket
  float flo = -0.51f * (float)w, fhi = 0.51f * (float)w;
  for (int it = 0; it < SPEC_FP32_ITS; ++it) {
    const float x = 0.5f * (flo + fhi);
    float q = 1.0f, bb = 0.0f;
    int cnt = 0;
    for (int i = 0; i < n; ++i) {
      const float2 t = abf[i];
      q = (t.x - x) - __fdividef(bb, q);
      if (fabsf(q) < 1e-9f) q = -1e-9f;
      cnt += q < 0.0f ? 1 : 0;
      bb = t.y;
    }
    if (cnt <= j)
      flo = x;
    else
      fhi = x;
  }
  double x = mid + 0.5 * ((double)flo + (double)fhi);
  double lo = fmax(x - 0x1p-18 * w, glo), hi = fmin(x + 0x1p-18 * w, ghi);
  // 2. FP64 counts at its ends
  int cl, ch;
  double p, dp, r1;
  sturm_eval<false>(ab, n, lo, p, dp, r1, cl);
  sturm_eval<false>(ab, n, hi, p, dp, r1, ch);
  if (cl > j) {
    hi = lo;
    ch = cl;
    lo = glo;
    cl = 0;
    x = 0.5 * (lo + hi);
  } else if (ch <= j) {
    lo = hi;
    cl = ch;
    hi = ghi;
    ch = n;
    x = 0.5 * (lo + hi);
  }
  // 3. Newton inside the bracket
  bool act = real;
  double th = x, wt = 0.0, dx_prev = 1e300;
  for (int it = 0; it < SPEC_MAX_ITS && __any_sync(0xffffffffu, act); ++it) {
    int cnt;
    sturm_eval<true>(ab, n, x, p, dp, r1, cnt);
    if (!act) continue;
    if (cnt <= j) {
      lo = x;
      cl = cnt;
    } else {
      hi = x;
      ch = cnt;
    }
    const bool alone = cl == j && ch == j + 1;
    const double dx = p / dp, adx = fabs(dx), xn = x - dx;
    wt = fabs(r1 / dp);
    // converged, or at the rounding level of p / p'
    if (alone && (adx <= tol || (adx <= 0x1p-44 && adx >= 0.25 * dx_prev))) {
      th = xn >= lo && xn <= hi ? xn : x;
      act = false;
    } else if (hi - lo <= tol) {
      th = 0.5 * (lo + hi);
      act = false;
    } else {
      // every other pass halves the bracket once Newton drags
      const bool newton = alone && xn > lo && xn < hi && !(it > 8 && (it & 1));
      dx_prev = newton ? adx : 1e300;
      x = newton ? xn : 0.5 * (lo + hi);
      th = x;
    }
  }
  wt_out = wt;
  return th;
}

__global__ void __launch_bounds__(SPEC_THREADS) k_spectral(
    const double *__restrict__ alpha, const double *__restrict__ beta,
    const double *__restrict__ beta0, const int *__restrict__ k_eff, int k, JacobiBufs jb,
    unsigned long long *min_theta_bits, unsigned *status) {
  pdl_wait();
  extern __shared__ double2 ab[];                       // [k] scaled (a, b^2)
  float2 *abf = reinterpret_cast<float2 *>(ab + k);     // [k] the same about the middle, FP32
  double *ths = reinterpret_cast<double *>(abf + k);    // [k] scaled nodes
  double *mus = ths + k;                                // [k] eigenvalues without row 0
  __shared__ double slo[SPEC_THREADS / 32], shi[SPEC_THREADS / 32];
  const int v = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nw = blockDim.x >> 5;
  // A depth outside [0, k] (possible only for caller-supplied tridiagonals)
  // is flagged and the vector skipped: its rows hold at most k entries.
  int n = k_eff[v];
  if (n < 0 || n > k) {
    if (tid == 0) atomicOr(status, ST_BAD_INPUT);
    n = 0;
  }
  if (tid == 0) jb.n[v] = n;
  if (n <= 0) return;
  const double *al = alpha + (size_t)v * k, *be = beta + (size_t)v * k;
  // Gershgorin interval
  double glo = 1e300, ghi = -1e300;
  bool nan = !finite_bits(beta0[v]);
  for (int i = tid; i < n; i += blockDim.x) {
    const double a = al[i];
    nan |= !finite_bits(a) || (i + 1 < n && !finite_bits(be[i]));
    const double r = (i > 0 ? fabs(be[i - 1]) : 0.0) + (i + 1 < n ? fabs(be[i]) : 0.0);
    glo = fmin(glo, a - r);
    ghi = fmax(ghi, a + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  if (lane == 0) {
    slo[wid] = glo;
    shi[wid] = ghi;
  }
  // A coefficient that is not a number: the counts below would still close in
  // on some node, and weights formed from the nodes alone would be finite.  The
  // vector's weights are NaN instead, and with them all that is summed from it.
  if (__syncthreads_or(nan)) {
    for (int j = tid; j < n; j += blockDim.x) {
      jb.a[(size_t)v * k + j] = 1.0;
      jb.b2[(size_t)v * k + j] = __longlong_as_double(0x7ff8000000000000LL);
    }
    return;
  }
  glo = slo[0];
  ghi = shi[0];
  for (int w = 1; w < nw; ++w) {
    glo = fmin(glo, slo[w]);
    ghi = fmax(ghi, shi[w]);
  }
  // T on a power-of-two scale (exact) that brings the width into [1, 2)
  const double width = fmax(fmax(ghi - glo, 1e-14 * fmax(fabs(glo), fabs(ghi))), 1e-290);
  const int ex = ilogb(width);
  const double sc = ldexp(1.0, -ex);
  const double w = width * sc, pad = 1e-12 * w;
  glo = glo * sc - pad;
  ghi = ghi * sc + pad;
  const double mid = 0.5 * (glo + ghi);
  for (int i = tid; i < n; i += blockDim.x) {
    const double a = al[i] * sc;
    const double b = i + 1 < n ? be[i] * sc : 0.0;
    ab[i] = make_double2(a, b * b);
    abf[i] = make_float2((float)(a - mid), (float)(b * b));
  }
  __syncthreads();

  double *node = jb.a + (size_t)v * k, *weight = jb.b2 + (size_t)v * k;
  for (int j0 = 0; j0 < n; j0 += blockDim.x) {
    const int j = j0 + tid;
    if (j - lane >= n) break;   // this warp's eigenvalues are done
    double wt;
    const double th = eigenvalue(ab, abf, n, j, j < n, glo, ghi, mid, w, wt);
    if (j < n) {
      ths[j] = n == 1 ? ab[0].x : th;
      weight[j] = n == 1 ? 1.0 : wt;
    }
  }
  __syncthreads();
  // A close pair's weights are ill-conditioned one by one: r_1 / p' of the two
  // nodes errs by eps ||T|| / gap, and their sum with it.  The product formula
  // over the computed nodes and the computed eigenvalues without row 0 gives
  // the weights of a nearby tridiagonal, whose sums over a cluster are right.
  // Nodes that coincide to the last bit have the eigenvalues between them there
  // too; their factors are 0 / 0, and the group's weight, which the other
  // factors give, is shared equally.
  bool close = false;
  for (int j = tid; j + 1 < n; j += blockDim.x) close |= ths[j + 1] - ths[j] < 0x1p-16 * w;
  if (__syncthreads_or(close)) {
    for (int j0 = 0; j0 < n - 1; j0 += blockDim.x) {
      const int j = j0 + tid;
      if (j - lane >= n - 1) break;
      double wt;
      const double mu = eigenvalue(ab + 1, abf + 1, n - 1, j, j < n - 1, glo, ghi, mid, w, wt);
      // interlacing, also where rounding has broken it
      if (j < n - 1)
        mus[j] = fmin(fmax(mu, fmin(ths[j], ths[j + 1])), fmax(ths[j], ths[j + 1]));
    }
    __syncthreads();
    for (int j = tid; j < n; j += blockDim.x) {
      const double th = ths[j];
      double wt = 1.0;
      int same = 1;   // nodes that coincide with this one, itself included
      for (int i = 0; i < n; ++i) {
        if (i == j) continue;
        // mu between theta_i and theta_j: a factor within [0, 1]
        const double den = th - ths[i];
        if (den != 0.0)
          wt *= (th - mus[i < j ? i : i - 1]) / den;
        else
          ++same;
      }
      if (same > 1) wt /= same;
      weight[j] = wt;
    }
  }
  // Gauss nodes -> (Omega_j, wt_j); the smallest node for the report
  const double b0 = beta0[v];
  double tmin = 1e300;
  bool bad = false;
  for (int j = tid; j < n; j += blockDim.x) {
    const double t = ldexp(ths[j], ex);
    tmin = fmin(tmin, t);
    bad |= !(t > 0.0);
    const double Om = t > 0.0 ? sqrt(t) : 0.0;
    node[j] = Om;
    weight[j] = Om > 0.0 ? b0 * b0 * weight[j] / Om : 0.0;
  }
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tmin = fmin(tmin, __shfl_xor_sync(0xffffffffu, tmin, o));
  if (lane == 0) slo[wid] = tmin;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < nw; ++i) tmin = fmin(tmin, slo[i]);
    if (bad)
      atomicOr(status, ST_NOT_SPD);
    else
      atomicMin(min_theta_bits, (unsigned long long)__double_as_longlong(tmin));
  }
}

void launch_spectral_impl(const double *alpha, const double *beta, const double *beta0,
                          const int *k_eff, int B, int k, JacobiBufs jb,
                          unsigned long long *min_theta_bits, unsigned *status, cudaStream_t st) {
  // 40 k bytes of shared memory per block: 164 KB at the largest depth
  static DeviceOnce once;
  allow_smem(once, k_spectral, 164 * 1024);
  const int threads = std::min(SPEC_THREADS, (k + 31) / 32 * 32);
  const size_t sh = (size_t)k * (sizeof(double2) + sizeof(float2) + 2 * sizeof(double));
  launch_pdl(k_spectral, dim3(B), dim3(threads), sh, st, alpha, beta, beta0, k_eff, k, jb,
             min_theta_bits, status);
}

// ---------------------------------------------------------------------------
// Spectral interval of C for the polynomial form (text after Eq. 12: p_g is
// fitted on the range of C's eigenvalues).
// ---------------------------------------------------------------------------
// Start vector with entries uniform in [-1, 1) from a counter-based hash
// (splitmix64 of seed + index), zero in the padding.
__global__ void k_hash_vector(double *v, int n_vc, int N, unsigned long long seed) {
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N) return;
  if (e >= n_vc) {
    v[e] = 0.0;
    return;
  }
  unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(e + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  v[e] = (double)(z >> 11) * 0x1p-52 - 1.0;
}

// Number of eigenvalues of the tridiagonal (a, b) below x (Sturm count by
// the LDL^T pivots, zero pivots nudged off zero).
__device__ int sturm_below(const double *a, const double *b, int n, double x, double pivmin) {
  int cnt = 0;
  double d = 1.0;
  for (int i = 0; i < n; ++i) {
    const double bb = i > 0 ? b[i - 1] * b[i - 1] : 0.0;
    d = a[i] - x - (i > 0 ? bb / d : 0.0);
    if (fabs(d) < pivmin) d = -pivmin;
    if (d < 0.0) ++cnt;
  }
  return cnt;
}

// One block: out[0] = min over the pairs of Delta^2 (C = Delta^2 + a positive
// semidefinite term, so no eigenvalue lies below it); out[1] = the largest
// Ritz value of the k-step tridiagonal (a, b) plus the last off-diagonal
// b_k = ||C q_k - ...||, the residual norm that bounds how far the Ritz value
// can lie from an eigenvalue.
__global__ void k_interval(const double *__restrict__ Delta2, int n_vc, const double *a,
                           const double *b, const int *k_eff, double *out) {
  pdl_wait();
  __shared__ double red[256];
  double m = 1e300;
  for (int e = threadIdx.x; e < n_vc; e += blockDim.x) m = fmin(m, Delta2[e]);
  red[threadIdx.x] = m;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  const int n = *k_eff;
  double hi = 0.0;
  if (n > 0) {
    double glo = 1e300, ghi = -1e300, scale = 0.0;
    for (int i = 0; i < n; ++i) {
      const double r = (i > 0 ? fabs(b[i - 1]) : 0.0) + (i + 1 < n ? fabs(b[i]) : 0.0);
      glo = fmin(glo, a[i] - r);
      ghi = fmax(ghi, a[i] + r);
      scale = fmax(scale, fabs(a[i]) + r);
    }
    const double pivmin = 1e-300 + 1e-15 * scale * 1e-15;
    double lo = glo, up = ghi;   // the largest eigenvalue lies in (lo, up]
    for (int it = 0; it < 200 && up - lo > 1e-14 * scale; ++it) {
      const double mid = 0.5 * (lo + up);
      if (sturm_below(a, b, n, mid, pivmin) >= n) up = mid; else lo = mid;
    }
    hi = up + (n - 1 < 0 ? 0.0 : fabs(b[n - 1]));
  }
  out[0] = red[0];
  out[1] = hi;
}

void launch_interval(const double *Delta2, int n_vc, int N, const double *a, const double *b,
                     const int *k_eff, double *out, double *vec, unsigned long long seed,
                     bool make_vector, cudaStream_t st) {
  if (make_vector)
    launch_pdl(k_hash_vector, dim3((N + 255) / 256), dim3(256), 0, st, vec, n_vc, N, seed);
  else
    launch_pdl(k_interval, dim3(1), dim3(256), 0, st, Delta2, n_vc, a, b, k_eff, out);
}
}  // namespace lgw
