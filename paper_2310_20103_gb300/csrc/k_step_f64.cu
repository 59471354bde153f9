// The vector part of one FP64 Lanczos step in one kernel (Eq. 13):
//   alpha_j = q_j . w,  w <- w - alpha_j q_j,  full Gram-Schmidt against the
//   stored q_0..q_j (two passes, the second always or by the norm criterion),
//   beta_{j+1} = ||w||, breakdown test, q_{j+1} = w / beta_{j+1},
// and, for the tensor-core FP64 products, the digits of Delta^1/2 q_{j+1} (on L's
// row scales, xd.scale).
//
// One cluster of nchunks blocks per vector, a block per chunk of VEC_CHUNK
// elements, w in registers throughout; sums over the vector meet in the
// blocks' shared memory (read by every block in the same order, so results do
// not depend on scheduling).
//
// Why: as ten kernels of this step, w went through memory at each, a vector
// of one or two chunks kept one warp of a block busy (elements were dealt out
// 256 to a warp), and launches cost as much as the work.  Elements are dealt out 512 to
// the block, so a short vector spreads over all four FP64 units of an SM.
// What bounds it now: the FP64 pipe (2 operations per element, row and pass).
#include <cooperative_groups.h>

#include "lgw_internal.cuh"
#include "oz_digits.cuh"

namespace lgw {
namespace {
namespace cg = cooperative_groups;

constexpr int SE = 4;   // element pairs per thread

__device__ __forceinline__ int pair_elem(int chunk, int u) {
  return chunk * VEC_CHUNK + u * (2 * VEC_THREADS) + 2 * (int)threadIdx.x;
}
// How many of a warp's SE pairs per thread lie inside the vector.  Operations
// on the zeros past its end would take their share of the FP64 pipe: N_vc 256
// leaves four of a block's eight warps empty (160 vectors, k 64, CGS2: 65 us
// per step with them at work, 42 us without).
__device__ __forceinline__ int warp_pairs(int N, int chunk, int warp) {
  const int left = N - chunk * VEC_CHUNK - 64 * warp;
  return max(0, min(SE, (left + 2 * VEC_THREADS - 1) / (2 * VEC_THREADS)));
}

// RB rows from row r0 on (the last one again past the end), NU pairs per
// thread, loaded before any of them is used: the loads of a batch overlap
// (one row at a time a row costs an L2 round trip).
template <int NU, int RB>
__device__ __forceinline__ void load_rows(const VecCtx &c, int r0, int nrows, size_t voff,
                                          int chunk, int nu, double2 (&q)[RB][NU]) {
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    const double *row = slot_ptr(c, min(r0 + r, nrows - 1)) + voff;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      if (u >= nu) break;
      const int e = pair_elem(chunk, u);
      q[r][u] = e < c.N ? *reinterpret_cast<const double2 *>(row + e) : make_double2(0.0, 0.0);
    }
  }
}

// Dots of the block's chunk of w with rows 0..nrows-1 into part[0..nrows),
// 16 rows per reduction.
template <int NU>
__device__ void step_dots(const VecCtx &c, int nrows, int b, int chunk, int nu,
                          const double2 (&w)[SE], double (*sred)[16], double *part) {
  constexpr int RB = NU == 1 ? 8 : 4;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // the warps of the chunk that hold elements
  const int nw = min(VEC_THREADS / 32, (c.N - chunk * VEC_CHUNK + 63) / 64);
  const size_t voff = (size_t)b * c.N;
  for (int r0 = 0; r0 < nrows; r0 += 16) {
    if (nu > 0) {
      double acc[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) acc[r] = 0.0;
#pragma unroll
      for (int rb = 0; rb < 16; rb += RB) {
        if (r0 + rb < nrows) {
          double2 q[RB][NU];
          load_rows<NU, RB>(c, r0 + rb, nrows, voff, chunk, nu, q);
#pragma unroll
          for (int u = 0; u < NU; ++u) {
            if (u >= nu) break;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
              acc[rb + r] = fma(q[r][u].x, w[u].x, acc[rb + r]);
              acc[rb + r] = fma(q[r][u].y, w[u].y, acc[rb + r]);
            }
          }
        }
      }
      // transposed butterfly: lane l ends with row l % 16, then the two halves
#pragma unroll
      for (int off = 8; off >= 1; off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < off; ++i) {
          const double send = up ? acc[i] : acc[i + off];
          const double keep = up ? acc[i + off] : acc[i];
          acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      }
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
      if (lane < 16) sred[wid][lane] = acc[0];
    }
    __syncthreads();
    if (threadIdx.x < 16 && r0 + (int)threadIdx.x < nrows) {
      double s = 0.0;
      for (int w8 = 0; w8 < nw; ++w8) s += sred[w8][threadIdx.x];
      part[r0 + threadIdx.x] = s;
    }
    __syncthreads();
  }
}

// w <- w - sum_i h_i q_i; returns this thread's share of ||w||^2.
template <int NU>
__device__ double step_update(const VecCtx &c, int nrows, int b, int chunk, int nu,
                              double2 (&w)[SE], const double *h) {
  constexpr int RB = NU == 1 ? 8 : 4;
  const size_t voff = (size_t)b * c.N;
  if (nu == 0) return 0.0;
  for (int i = 0; i < nrows; i += RB) {
    double2 q[RB][NU];
    load_rows<NU, RB>(c, i, nrows, voff, chunk, nu, q);
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      if (u >= nu) break;
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        if (i + r >= nrows) break;
        const double hi = h[i + r];
        w[u].x = fma(-hi, q[r][u].x, w[u].x);
        w[u].y = fma(-hi, q[r][u].y, w[u].y);
      }
    }
  }
  double nrm = 0.0;
#pragma unroll
  for (int u = 0; u < NU; ++u)
    if (u < nu) nrm = fma(w[u].x, w[u].x, fma(w[u].y, w[u].y, nrm));
  return nrm;
}

template <bool GS>
__global__ void __launch_bounds__(VEC_THREADS, GS ? 2 : 4)
    k_step_f64(VecCtx c, int j, OzOperand xd) {
  extern __shared__ double dyn[];   // GS: coefficients of both passes' partials, and their sums
  __shared__ double red[VEC_THREADS / 32];
  __shared__ double sred[GS ? VEC_THREADS / 32 : 1][16];
  __shared__ double part[3];        // the block's ||w||^2 before, between and after the passes
  __shared__ int xmax;
  pdl_wait();
  cg::cluster_group cl = cg::this_cluster();
  const int nb = gridDim.x, chunk = blockIdx.x, b = blockIdx.y, v = c.vec0 + b;
  const bool lead = chunk == 0 && threadIdx.x == 0;
  const size_t voff = (size_t)b * c.N;
  double *qn = slot_ptr(c, j + 1) + voff;
  // the same verdict in every block of the cluster (k_eff only moves to j + 1)
  if (!(b < c.nvec && c.k_eff[v] > j)) {
#pragma unroll
    for (int u = 0; u < SE; ++u) {
      const int e = pair_elem(chunk, u);
      if (e >= c.N) continue;
      *reinterpret_cast<double2 *>(qn + e) = make_double2(0.0, 0.0);
      if (xd.d) oz::store_digits2(0.0, 0.0, 1, b, e, xd);
    }
    if (lead) {
      c.betaj[b] = 0.0;
      c.sinv[b] = 0.0;
      if (xd.d) xd.e[b] = 1;
    }
    return;
  }
  const int nrows = j + 1;
  const int nu = warp_pairs(c.N, chunk, threadIdx.x >> 5);
  // at most 512 elements: one pair per thread (the others' operations would
  // each take their share of the FP64 pipe)
  const bool one = c.N <= 2 * VEC_THREADS;
  auto dots = [&](const double2 (&x)[SE], double *out) {
    if (one)
      step_dots<1>(c, nrows, b, chunk, nu, x, sred, out);
    else
      step_dots<SE>(c, nrows, b, chunk, nu, x, sred, out);
  };
  auto update = [&](double2 (&x)[SE], const double *co) {
    return one ? step_update<1>(c, nrows, b, chunk, nu, x, co)
               : step_update<SE>(c, nrows, b, chunk, nu, x, co);
  };
  double *h1 = dyn, *h2 = dyn + c.kmax1, *h = dyn + 2 * c.kmax1;
  // ||w||^2 over the cluster from part[i] of every block
  auto total = [&](int i) {
    double s = 0.0;
    for (int r = 0; r < nb; ++r) s += cl.map_shared_rank(part, r)[i];
    return s;
  };
  auto share = [&](int i, double mine) {
    mine = block_sum_to0(mine, red);
    if (threadIdx.x == 0) part[i] = mine;
  };
  // alpha_j from the contraction's partials (every block sums them itself)
  double s = 0.0;
  for (int t = threadIdx.x; t < c.n_mt; t += VEC_THREADS) s += c.alpha_part[(size_t)t * c.Bs + b];
  const double alpha = block_sum(s, red);
  const double amax = fmax(c.amax[b], fabs(alpha));
  const double *qj = slot_ptr(c, j) + voff;
  double2 w[SE];
  double nrm = 0.0;
#pragma unroll
  for (int u = 0; u < SE; ++u) {
    const int e = pair_elem(chunk, u);
    w[u] = make_double2(0.0, 0.0);
    if (u >= nu) continue;
    if (e < c.N) {
      const double2 q2 = *reinterpret_cast<const double2 *>(qj + e);
      w[u] = *reinterpret_cast<const double2 *>(c.w + voff + e);
      w[u].x = fma(-alpha, q2.x, w[u].x);
      w[u].y = fma(-alpha, q2.y, w[u].y);
    }
    nrm = fma(w[u].x, w[u].x, fma(w[u].y, w[u].y, nrm));
  }
  share(0, nrm);
  int norm_at = 0;
  bool second = false;
  if (GS) {
    dots(w, h1);
    cl.sync();
    for (int i = threadIdx.x; i < nrows; i += VEC_THREADS) {
      double t = 0.0;
      for (int r = 0; r < nb; ++r) t += cl.map_shared_rank(h1, r)[i];
      h[i] = t;
    }
    __syncthreads();
    share(1, update(w, h));
    norm_at = 1;
    second = c.reorth == LGW_REORTH_CGS2;
    if (!second) {
      cl.sync();
      second = total(1) < 0.5 * total(0);
    }
    if (second) {
      dots(w, h2);
      cl.sync();
      for (int i = threadIdx.x; i < nrows; i += VEC_THREADS) {
        double t = 0.0;
        for (int r = 0; r < nb; ++r) t += cl.map_shared_rank(h2, r)[i];
        h[i] = t;
      }
      __syncthreads();
      share(2, update(w, h));
      norm_at = 2;
    }
  }
  if (threadIdx.x == 0) xmax = 0;
  cl.sync();
  const double beta = sqrt(total(norm_at));
  const bool stop = !(beta > c.tol * amax);
  const double inv = (stop || !(beta > 0.0)) ? 0.0 : 1.0 / beta;
  if (lead) {
    c.alpha[(size_t)v * c.k + j] = alpha;
    c.amax[b] = amax;
    c.beta[(size_t)v * c.k + j] = beta;
    c.betaj[b] = beta;
    c.sinv[b] = inv;
    if (GS) c.flag2[b] = second ? 1 : 0;
    if (GS && second && c.reorth != LGW_REORTH_CGS2) atomicAdd(c.n_second, 1);
    if (stop) c.k_eff[v] = j + 1;
  }
  int m = 0;
#pragma unroll
  for (int u = 0; u < SE; ++u) {
    const int e = pair_elem(chunk, u);
    if (e >= c.N) continue;
    w[u].x = inv > 0.0 ? w[u].x * inv : 0.0;
    w[u].y = inv > 0.0 ? w[u].y * inv : 0.0;
    *reinterpret_cast<double2 *>(qn + e) = w[u];
    if (xd.d) {
      const double2 d = *reinterpret_cast<const double2 *>(xd.scale + e);
      w[u].x *= d.x;
      w[u].y *= d.y;
      m = max(m, max(oz::exp_field(w[u].x), oz::exp_field(w[u].y)));
    }
  }
  if (xd.d) {
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&xmax, m);
    cl.sync();
    m = 1;
    for (int r = 0; r < nb; ++r) m = max(m, *cl.map_shared_rank(&xmax, r));
    if (lead) xd.e[b] = m;
#pragma unroll
    for (int u = 0; u < SE; ++u) {
      const int e = pair_elem(chunk, u);
      if (e < c.N) oz::store_digits2(w[u].x, w[u].y, m, b, e, xd);
    }
  }
  cl.sync();   // no block leaves while another may read its sums
}

template <bool GS>
void launch_one(const VecCtx &c, int j, const OzOperand &x, cudaStream_t st) {
  static DeviceOnce once;
  once(current_device(), [] {
    cudaFuncSetAttribute(k_step_f64<GS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaFuncSetAttribute(k_step_f64<GS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         STEP_MAX_K1 * 3 * (int)sizeof(double));
  });
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(c.nchunks, c.Bs);
  cfg.blockDim = dim3(VEC_THREADS);
  cfg.dynamicSmemBytes = GS ? (size_t)3 * c.kmax1 * sizeof(double) : 0;
  cfg.stream = st;
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = c.nchunks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  cudaLaunchKernelEx(&cfg, k_step_f64<GS>, c, j, x);
}
}  // namespace

// One cluster per vector where its chunks fit one and the coefficients fit
// shared memory; else false (the passes run as kernels of their own).  With
// Gram-Schmidt up to 8 blocks: whole requests of 24 CGS2 steps take 2.0 ms
// fused against 3.4 ms at N_vc 512, 5.4 against 6.5 at 8192, 9.2 against 10.2
// at 16290 (8 chunks), but 23.0 against 22.1 at 32768, where clusters of 16
// leave blocks of a processing cluster unused.  Without it 16 blocks still
// gain (9.7 against 9.9 ms at 32768).
bool launch_step_f64(const VecCtx &c, int j, const OzOperand &x, cudaStream_t st) {
  const bool gs = c.reorth != LGW_REORTH_NONE;
  if (c.nchunks > (gs ? 8 : 16) || c.xh != nullptr || c.pair) return false;
  if (gs && c.kmax1 > STEP_MAX_K1) return false;
  if (gs)
    launch_one<true>(c, j, x, st);
  else
    launch_one<false>(c, j, x, st);
  return true;
}

}  // namespace lgw
