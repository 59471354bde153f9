// The static part of the self-energy and the density-fitting front end.
//
// Exchange (text after Eq. 5): Sigma^ex_t = -sum_v (vt|vt).  The pair factors
// share L's metric-folded form, (pq|rs) = sum_mu B_pq,mu B_rs,mu, so with the
// factors M[t][m][:] of the request (vt|vt) = sum_mu M[t][v][mu]^2 for the
// occupied orbitals v of the summed set.
//
// Density fitting: with fitting coefficients C_ab,mu and the Coulomb metric
// V_mu,nu = (mu|nu), (ab|cd) = sum C_ab,mu V_mu,nu C_cd,nu; V = R R^T
// (Cholesky, R lower) gives the factors B = C R.  FP64 throughout.
#include <algorithm>

#include "fp_iter.cuh"
#include "lgw_internal.cuh"

namespace lgw {

__global__ void k_sigma_x(const double *__restrict__ M, int n_m, int n_aux,
                          const int *__restrict__ m_idx, int n_v, double *__restrict__ out) {
  pdl_wait();
  __shared__ double red[8];
  const int t = blockIdx.x;
  double s = 0.0;
  for (int mi = 0; mi < n_m; ++mi) {
    if (m_idx[mi] >= n_v) continue;
    const double *row = M + ((size_t)t * n_m + mi) * n_aux;
    for (int mu = threadIdx.x; mu < n_aux; mu += blockDim.x) s = fma(row[mu], row[mu], s);
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) out[t] = -s;
}

// --------------------------------------------------------------------------
// Blocked right-looking Cholesky, NB x NB blocks, in place on the lower
// triangle of a [n][n] row-major matrix.
// --------------------------------------------------------------------------
constexpr int NB = 64;

// Factor the diagonal block at (j0, j0): one CTA, columns in panels of eight.
// A warp's FP64 instruction holds its scheduler's pipe for 76 clocks whatever
// the lanes do, so the count of instructions per warp is what bounds the serial
// chain of 64 columns.  Every warp factors the panel's eight diagonal rows
// (lanes 0..7) along with a quarter of the rows below (lanes 8..), by shuffles
// and without barriers; then the panel updates the rest of the block, row i and
// row 63 - i dealt together to the same threads.  216 us per block with one
// thread per row and square root, division and row sums in sequence, 109 us
// column by column with three barriers each, 75 us now.
constexpr int POTRF_THREADS = 128, PW = 8;
constexpr int CM_ROWS = 256;   // rows of a column-maximum tile of 64 columns

// Largest finite exponent field of 64 columns of a tile of C, into col.
__device__ void col_max_tile(const ColMax &cm, int n, int tile) {
  const int strips = (n + 63) / 64, c = (tile % strips) * 64 + (threadIdx.x & 63);
  const int r0 = (tile / strips) * CM_ROWS, r1 = min(cm.n_pairs, r0 + CM_ROWS);
  if (c >= n) return;
  int m = 0;
#pragma unroll 8
  for (int r = r0 + (threadIdx.x >> 6); r < r1; r += POTRF_THREADS / 64) {
    const double x = cm.C[(size_t)r * n + c];
    const int f = (__double2hiint(x) >> 20) & 0x7ff;
    if (nonzero_bits(x) && f < 2047) m = max(m, max(f, 1));
  }
  if (m > 0) atomicMax(&cm.col[c], m);
}

__global__ void __launch_bounds__(POTRF_THREADS) k_potrf_diag(double *A, int n, int j0,
                                                              unsigned *status, ColMax cm) {
  pdl_wait();
  if (blockIdx.x > 0) {   // beside the first diagonal block
    col_max_tile(cm, n, blockIdx.x - 1);
    return;
  }
  __shared__ double blk[NB][NB + 1];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int nb = min(NB, n - j0);
  for (int idx = t; idx < NB * NB; idx += POTRF_THREADS) {
    const int r = idx / NB, c = idx % NB;
    // past the matrix: the identity, which leaves the rest as it is
    blk[r][c] = r < nb ? (c <= r ? A[(size_t)(j0 + r) * n + j0 + c] : 0.0) : (r == c ? 1.0 : 0.0);
  }
  __syncthreads();
#pragma unroll 1
  for (int p0 = 0; p0 < nb; p0 += PW) {
    const int below = NB - p0 - PW, quarter = (below + 3) / 4;   // rows under the panel, per warp
    const int row = lane < PW ? p0 + lane : p0 + PW + w * quarter + lane - PW;
    const bool mine = lane < PW || (lane - PW < quarter && row < NB);
    double v[PW];
#pragma unroll
    for (int c = 0; c < PW; ++c) v[c] = mine ? blk[row][p0 + c] : 0.0;
#pragma unroll
    for (int j = 0; j < PW; ++j) {
      double d = __shfl_sync(0xffffffffu, v[j], j);
      if (!(d > 0.0)) {
        if (t == 0) atomicOr(status, ST_NOT_SPD);
        d = 1.0;
      }
      double x, s;
      if (d > 1e-280 && d < 1e280) {
        const double r = rsqrt_iter(d);
        s = sqrt_from(d, r);
        x = div_from(v[j], s, r);
      } else {   // infinities too
        s = sqrt(d);
        x = v[j] / s;
      }
      v[j] = lane == j ? s : x;
#pragma unroll
      for (int c = j + 1; c < PW; ++c) {
        const double l = __shfl_sync(0xffffffffu, v[j], c);
        v[c] = fma(-v[j], l, v[c]);
      }
    }
    __syncthreads();   // every warp has read the diagonal rows
    if (mine && (w == 0 || lane >= PW)) {
#pragma unroll
      for (int c = 0; c < PW; ++c)
        if (p0 + c <= row) blk[row][p0 + c] = v[c];
    }
    __syncthreads();
    if (below > 0) {
      // rows p0 + 8 + m and 63 - m, each up to its diagonal: together below + 1
      // elements, dealt to `per` threads
      int per = 4;
      while (2 * per * (below / 2) <= POTRF_THREADS) per *= 2;
      const int m = t / per, l = t % per;
      if (m < below / 2) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int i = hf ? NB - 1 - m : p0 + PW + m;
          double li[PW];
#pragma unroll
          for (int p = 0; p < PW; ++p) li[p] = blk[i][p0 + p];
#pragma unroll 1
          for (int c = p0 + PW + l; c <= i; c += per) {
            double x = blk[i][c];
#pragma unroll
            for (int p = 0; p < PW; ++p) x = fma(-li[p], blk[c][p0 + p], x);
            blk[i][c] = x;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int idx = t; idx < NB * NB; idx += POTRF_THREADS) {
    const int r = idx / NB, c = idx % NB;
    if (r < nb && c <= r) A[(size_t)(j0 + r) * n + j0 + c] = blk[r][c];
  }
}

// rows below the diagonal block: L_i = A_i L_jj^{-T} by forward substitution,
// eight threads per row (thread l holds columns l, l + 8, ...), the row in
// registers.  212 us per panel with a row per thread in global memory; 34 us now.
constexpr int TRSM_ROWS = 16;

__global__ void __launch_bounds__(8 * TRSM_ROWS) k_trsm_panel(double *A, int n, int j0) {
  pdl_wait();
  __shared__ double Ljj[NB][NB + 1];
  __shared__ double rd[NB];
  const int t = threadIdx.x, l = t & 7;
  const int nb = min(NB, n - j0);   // a panel exists only below a full block
  for (int idx = t; idx < NB * NB; idx += 8 * TRSM_ROWS) {
    const int r = idx / NB, c = idx % NB;
    Ljj[r][c] = (r < nb && c <= r) ? A[(size_t)(j0 + r) * n + j0 + c] : (r == c ? 1.0 : 0.0);
  }
  __syncthreads();
  if (t < NB) rd[t] = 1.0 / Ljj[t][t];
  __syncthreads();
  const int i = j0 + nb + blockIdx.x * TRSM_ROWS + (t >> 3);
  const bool ok = i < n;
  double *row = A + (size_t)(ok ? i : 0) * n + j0;
  double x[NB / 8];
#pragma unroll
  for (int k = 0; k < NB / 8; ++k) x[k] = ok && 8 * k + l < nb ? row[8 * k + l] : 0.0;
#pragma unroll
  for (int kb = 0; kb < NB / 8; ++kb) {
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      const int c = 8 * kb + cc;
      // a reciprocal outside the normal range (or of an infinity): divide
      const bool plain = !(fabs(rd[c]) > 1e-150 && fabs(rd[c]) < 1e150);
      const double q = plain ? x[kb] / Ljj[c][c] : div_from(x[kb], Ljj[c][c], rd[c]);
      const double v = __shfl_sync(0xffffffffu, q, cc, 8);
      if (l == cc) x[kb] = v;
      if (l > cc) x[kb] = fma(-v, Ljj[8 * kb + l][c], x[kb]);
#pragma unroll
      for (int k = kb + 1; k < NB / 8; ++k) x[k] = fma(-v, Ljj[8 * k + l][c], x[k]);
    }
  }
  if (!ok) return;
#pragma unroll
  for (int k = 0; k < NB / 8; ++k)
    if (8 * k + l < nb) row[8 * k + l] = x[k];
}

// trailing update A[i][j] -= sum_p L[i][j0+p] L[j][j0+p] for i, j >= j0+nb,
// lower triangle.  32 x 32 output tiles, 2 x 2 per thread: FP64-bound, and
// 64 x 64 tiles left most of the chip without one (86 us per update on average
// at n 1024; 46 us now).
__global__ void __launch_bounds__(256) k_syrk_update(double *A, int n, int j0, int nb) {
  pdl_wait();
  const int t0 = j0 + nb;
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj > bi) return;
  __shared__ double Xs[NB][33];
  __shared__ double Ys[NB][33];
  const int i0 = t0 + bi * 32, jj0 = t0 + bj * 32;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  for (int idx = t; idx < 32 * NB; idx += 256) {
    const int p = idx & (NB - 1), r = idx / NB;
    Xs[p][r] = (i0 + r < n && p < nb) ? A[(size_t)(i0 + r) * n + j0 + p] : 0.0;
    Ys[p][r] = (jj0 + r < n && p < nb) ? A[(size_t)(jj0 + r) * n + j0 + p] : 0.0;
  }
  __syncthreads();
  double acc[2][2] = {};
#pragma unroll 8
  for (int p = 0; p < NB; ++p) {
    const double x0 = Xs[p][ty], x1 = Xs[p][ty + 16], y0 = Ys[p][tx], y1 = Ys[p][tx + 16];
    acc[0][0] = fma(x0, y0, acc[0][0]);
    acc[0][1] = fma(x0, y1, acc[0][1]);
    acc[1][0] = fma(x1, y0, acc[1][0]);
    acc[1][1] = fma(x1, y1, acc[1][1]);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = i0 + ty + 16 * q;
    if (i >= n) continue;
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int j = jj0 + tx + 16 * w;
      if (j < n && j <= i) A[(size_t)i * n + j] -= acc[q][w];
    }
  }
}

__global__ void k_zero_upper(double *A, int n) {
  pdl_wait();
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * n) return;
  const int i = (int)(idx / n), j = (int)(idx % n);
  if (j > i) A[idx] = 0.0;
}

// Cm[M][N] = Am[M][K] Bm[K][N], row-major, FP64 (64 x 64 tiles)
__global__ void __launch_bounds__(256) k_gemm_nn_f64(const double *__restrict__ Am,
                                                     const double *__restrict__ Bm, int M, int N,
                                                     int K, double *__restrict__ Cm) {
  pdl_wait();
  __shared__ double As[16][65];
  __shared__ double Bs[16][65];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  double acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
    for (int rep = 0; rep < 4; ++rep) {
      const int idx = t + 256 * rep;
      const int kk = idx & 15, m = idx >> 4;          // A tile: 64 rows x 16
      As[kk][m] = (m0 + m < M && k0 + kk < K) ? Am[(size_t)(m0 + m) * K + k0 + kk] : 0.0;
      const int nn = idx & 63, k2 = idx >> 6;         // B tile: 16 x 64 cols
      Bs[k2][nn] = (k0 + k2 < K && n0 + nn < N) ? Bm[(size_t)(k0 + k2) * N + n0 + nn] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty + 16 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int nn = n0 + tx + 16 * j;
      if (nn < N) Cm[(size_t)m * N + nn] = acc[i][j];
    }
  }
}

// ----------------------------------------------------------------------------
void launch_sigma_x(const double *M, int n_t, int n_m, int n_aux, const int *m_idx, int n_v,
                    double *out, cudaStream_t st) {
  if (n_t > 0) launch_pdl(k_sigma_x, dim3(n_t), dim3(256), 0, st, M, n_m, n_aux, m_idx, n_v, out);
}

// R = the metric, and the column maxima start at zero.
__global__ void __launch_bounds__(256) k_fit_init(const double *__restrict__ metric, size_t n2,
                                                  double *__restrict__ R, int *__restrict__ col,
                                                  int nc) {
  pdl_wait();
  const size_t step = (size_t)gridDim.x * 256, i0 = (size_t)blockIdx.x * 256 + threadIdx.x;
  for (size_t i = i0; i < n2; i += step) R[i] = metric[i];
  for (size_t i = i0; i < (size_t)nc; i += step) col[i] = 0;
}
void launch_fit_init(const double *metric, int n, double *R, int *col, int nc, cudaStream_t st) {
  const size_t n2 = (size_t)n * n;
  launch_pdl(k_fit_init, dim3((unsigned)std::min<size_t>((n2 + 255) / 256, 152 * 8)), dim3(256), 0,
             st, metric, n2, R, col, col ? nc : 0);
}

int launch_cholesky(double *A, int n, unsigned *status, cudaStream_t st, const ColMax &cm) {
  int launches = 0;
  const int tiles = cm.col ? (n + 63) / 64 * ((cm.n_pairs + CM_ROWS - 1) / CM_ROWS) : 0;
  for (int j0 = 0; j0 < n; j0 += NB) {
    const int nb = std::min(NB, n - j0);
    launch_pdl(k_potrf_diag, dim3(j0 == 0 ? 1 + tiles : 1), dim3(POTRF_THREADS), 0, st, A, n, j0,
               status, cm);
    ++launches;
    const int rest = n - j0 - nb;
    if (rest > 0) {
      launch_pdl(k_trsm_panel, dim3((rest + TRSM_ROWS - 1) / TRSM_ROWS), dim3(8 * TRSM_ROWS), 0,
                 st, A, n, j0);
      const int tiles = (rest + 31) / 32;
      launch_pdl(k_syrk_update, dim3(tiles, tiles), dim3(256), 0, st, A, n, j0, nb);
      launches += 2;
    }
  }
  launch_pdl(k_zero_upper, dim3((unsigned)(((size_t)n * n + 255) / 256)), dim3(256), 0, st, A, n);
  return launches + 1;
}

void launch_gemm_nn_f64(const double *A, const double *B, int M, int N, int K, double *C,
                        cudaStream_t st) {
  dim3 grid((N + 63) / 64, (M + 63) / 64);
  launch_pdl(k_gemm_nn_f64, grid, dim3(256), 0, st, A, B, M, N, K, C);
}

}  // namespace lgw
