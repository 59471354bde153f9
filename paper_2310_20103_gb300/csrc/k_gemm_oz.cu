// FP64 matrix products on the tensor cores by error-free slicing (the scheme
// of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012) 95).
//
// GB300 executes FP64 at 2 lanes per SM clock (1.2 TFLOP/s); its BF16 tensor
// cores multiply small integers exactly and add them exactly in FP32 up to
// 2^24.  Each operand row (along the contraction) is scaled by a power of two
// above its largest magnitude, x = 2^e sum_s d_s 2^(-6-7s), into 8 signed
// 7-bit digits d_s in [-64, 64]: a resolution of 2^-56 of the row's largest
// element, where FP64's own rounding of that element is 2^-53.  Then
//   sum_k x_k y_k = 2^(ex+ey-12) sum_t 2^(-7t) S_t,  S_t = sum_{i+j=t} d_i . d_j
// over t = 0..8 (43 digit products; the dropped ones are below 2^-62 of the
// largest product).  Products are at most 2^12, so over 1024 terms S_0..S_3
// are exact multiples of their unit below 2^24 of it; the others carry weights
// of 2^-28 and less and may round.  Every 1024 terms the sums are joined in
// 64-bit integers and rounded once to FP64.
//
// What the digits lose is relative to the two rows' largest elements, max |x_k|
// max |y_k|, where the roundings of an FMA chain are relative to the terms x_k
// y_k.  For rows whose large elements meet (normal matrices, Krylov vectors)
// that is less than FP64's own roundings: against exact sums, B = C R with 1024
// terms errs by 2.6e-16 of its norm, the FMA chain by 1.08e-15
// (tests/test_gpu_f64_products.py).  Rows graded along the contraction, one
// rising where the other falls, would lose digits: what is graded by index is
// balanced first, by exact powers of two, for L and the vectors by L's rows and
// columns (ensure_digits), for density fitting by the auxiliary functions
// (tests/test_gpu_f64_graded.py).
//
// N_vc 32768, N_aux 1024, 64 vectors: 180 us per product on average (C x with
// its digits 474 us), against 3.6 and 4.1 ms on the FP64 pipe (24 TFLOP/s in
// FP64 terms).  Where a tile of L y spends its time: 73 us in the products
// (43 per K block, 19 MMAs of 64 to 256 columns per 16 terms, 63% of the BF16
// rate: an MMA of few columns costs more than its share) and then the joined
// sums with the tensor pipe idle (TMEM holds one tile).  These took 60 us with
// four warps, a memory round trip per column and the conversions on the FP64
// pipe (244 us per product); now eight warps issue all loads of eight columns
// first and convert on the integer pipe.
//
// Layout: digits as BF16, [slice][K block of 64][row][64], so a TMA box (64
// elements by rows) is one contiguous run, as for the other contractions.  A
// CTA owns 128 rows of A by NT rows of B and keeps S_0 .. S_7 as 8 NT TMEM
// columns: digit i of A against the stacked digits 0..7-i of B is one product
// of N = (8-i) NT columns that lands in S_i .. S_7, so an A tile is read once
// however many digits of B it meets.  An MMA whose columns cross a multiple of
// 256 gives wrong sums, so at NT = 64 the product is split there.  Digit s is
// stored with its weight 2^(-7s) (BF16 is a float), so S_8 is simply added to
// S_7's columns.  B's eight tiles of a K block have two buffers, A's go through
// a ring of single tiles.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>

#include "fp_bits.cuh"
#include "oz_digits.cuh"
#include "oz_plan.cuh"
#include "tc_ptx.cuh"

namespace lgw {
namespace oz {

using namespace tc;

constexpr int EPI_WARPS = 8;    // two per TMEM lane quarter, each half of the columns
constexpr int NTHREADS = 64 + 32 * EPI_WARPS;

template <int NT>
struct Cfg {
  static constexpr int A_BYTES = BM * KB * 2;
  static constexpr int B_BYTES = S * NT * KB * 2;
  static constexpr int A_STAGES = NT == 64 ? 6 : 8;
  static constexpr int BOX = NT == 64 ? 4 : 8;   // B's slices per box (32 KB at most)
  static constexpr int BAR_BYTES = 256;
  static constexpr int SMEM = 1024 + 2 * B_BYTES + A_STAGES * A_BYTES + BAR_BYTES;
  static constexpr uint32_t TMEM_COLS = S * NT;
};

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *tm, uint64_t *bar, int x,
                                            int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}
// 8 consecutive FP32 columns of this thread's TMEM lane (no wait)
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]),
        "=f"(r[7])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 2^sh sum_t 2^(40 - 7t) S_t from the weighted sums s[t] = 2^(-7t) S_t: a 64-bit
// integer below 2^62.3 in magnitude, seven more bits of what lies below its
// unit where a double has room for them, one rounding.  On the integer pipe
// throughout (the FP64 pipe's conversions run at 2 lanes per SM clock).
__device__ __forceinline__ double join_sums(const float (&s)[8], int sh) {
  const int h = __float2int_rn(s[0]) * 128 + __float2int_rn(s[1] * 0x1p+7f);
  const int g = __float2int_rn(s[2] * 0x1p+14f) * 128 + __float2int_rn(s[3] * 0x1p+21f);
  const float low = (s[6] + s[7]) * 0x1p+40f;
  const int il = __float2int_rn(low);
  const int f = __float2int_rn(s[5] * 0x1p+35f) * 32 + il;
  long long t = ((long long)h << 33) + (long long)g * (1 << 19) +
                (long long)__float2int_rn(s[4] * 0x1p+28f) * 4096 + f;
  if (t + (1LL << 55) >= 0 && t < (1LL << 55)) {
    t = t * 128 + __float2int_rn((low - (float)il) * 128.0f);
    sh -= 7;
  }
  return ll2d_scaled(t, sh);
}

// out[col * ldo + row] of the tile's products; the epilogues of the FP64
// contractions (k_gemm_f64.cu), and plain or accumulated output.
struct Epi {
  int mode;
  const int *ea, *eb;      // exponent fields of A's and B's rows
  double *out;             // OZ_PART: [split][Ncols][ldo]; else [Ncols][ldo]
  int ldo;
  double scale;            // OZ_ADD: out += scale * product
  int lower;               // A's row i is zero before K index i: skip those K blocks
  const double *Delta2, *dsq, *cd, *q, *qprev, *betaj;
  double *alpha_part;      // [M / 64][Ncols] partials of q . w, or NULL
  unsigned *status;
  // CHECK: the K blocks' exponents of A's and B's rows, and the matrices
  // themselves, A's row i the column i of xa
  const short *ba, *bb;
  const double *xa, *xb;
  int ldxa, ldxb, K;
};

// Whether eight digits are enough for a tile's products.  What they lose is
// relative to max |a_i| max |b_j|, so an output (i, j) is as good as FP64's
// while some K block's largest |a| times its largest |b| comes near that.  False
// where more than an eighth of the tile's outputs miss it by more than 2^6: a
// chance small element in a short last block is not counted, operands graded
// against one another are.  Where in some K block no row falls far below its own
// largest element, as usual, the outputs need not be looked at one by one.  The
// epilogue's warps ask while the products run.
constexpr int LOSS_BITS = 6;
struct LossShared {
  int da[32], db[32];   // by K block: the rows' largest distance from their maxima
  int bad, all;
};
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

template <int NT>
__device__ bool digits_do(const Epi &e, int m0, int n0, int M, int Ncols, int nkb,
                          LossShared &sh) {
  const int t = threadIdx.x - 64, kfirst = e.lower ? m0 / KB : 0;
  if (t == 0) sh.bad = sh.all = 0;
  for (int k0 = kfirst; k0 < nkb; k0 += 32) {
    epi_sync();
    if (t < 32) sh.da[t] = sh.db[t] = k0 + t < nkb ? 0 : 1 << 20;
    epi_sync();
    const int k = t & 31, part = t >> 5;
    if (k0 + k < nkb) {
      int xa = 0, xb = 0;   // rows of zeros have no say
#pragma unroll
      for (int i = 0; i < BM / 8; ++i) {
        const int r = m0 + part * (BM / 8) + i, f = r < M ? e.ea[r] : 0;
        const int d = r < M ? f - e.ba[(size_t)r * nkb + k0 + k] : 0;
        if (f > 0) xa = max(xa, d);
      }
#pragma unroll
      for (int i = 0; i < NT / 8; ++i) {
        const int r = n0 + part * (NT / 8) + i, f = r < Ncols ? e.eb[r] : 0;
        const int d = r < Ncols ? f - e.bb[(size_t)r * nkb + k0 + k] : 0;
        if (f > 0) xb = max(xb, d);
      }
      atomicMax(&sh.da[k], xa);
      atomicMax(&sh.db[k], xb);
    }
    epi_sync();
    for (int i = 0; i < 32; ++i)
      if (sh.da[i] + sh.db[i] <= LOSS_BITS) return true;
  }
  const int row = m0 + (t & 127);
  int bad = 0, all = 0;
  if (row < M)
    for (int j = (t >> 7) * (NT / 2); j < ((t >> 7) + 1) * (NT / 2) && n0 + j < Ncols; ++j) {
      int best = 2 * OZ_ZERO;
      for (int k = kfirst; k < nkb; ++k)
        best = max(best, e.ba[(size_t)row * nkb + k] + e.bb[(size_t)(n0 + j) * nkb + k]);
      if (best <= 0) continue;   // no product at all: exactly zero
      ++all;
      bad += e.ea[row] + e.eb[n0 + j] - best > LOSS_BITS ? 1 : 0;
    }
  atomicAdd(&sh.bad, bad);
  atomicAdd(&sh.all, all);
  epi_sync();
  return 8 * sh.bad <= sh.all;
}

// The tile by FP64 multiplications, one chain over K per output (the order of
// k_gemm_nn_f64).
template <int NT>
__device__ void tile_f64(const Epi &e, int m0, int n0, int M, int Ncols) {
  const int t = threadIdx.x - 64, row = m0 + (t & 127), c0 = n0 + (t >> 7) * (NT / 2);
  if (row >= M) return;
  for (int g = 0; g < NT / 2; g += 8) {
    double acc[8] = {};
    for (int k = 0; k < e.K; ++k) {
      const double x = e.xa[(size_t)k * e.ldxa + row];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        acc[i] = fma(e.xb[(size_t)min(c0 + g + i, Ncols - 1) * e.ldxb + k], x, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (c0 + g + i < Ncols) e.out[(size_t)(c0 + g + i) * e.ldo + row] = acc[i];
  }
}

// CHECK: outputs that the digits are not enough for are formed in FP64 (OZ_PART
// of one split).
template <int NT, bool CHECK>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              int M, int Ncols, int num_kb, int kb_per_split, Epi e) {
  using C = Cfg<NT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t *bbuf = smem, *aring = smem + 2 * C::B_BYTES;
  uint64_t *afull = reinterpret_cast<uint64_t *>(aring + C::A_STAGES * C::A_BYTES);
  uint64_t *aempty = afull + C::A_STAGES;
  uint64_t *bfull = aempty + C::A_STAGES;   // [2]
  uint64_t *bempty = bfull + 2;             // [2]
  uint64_t *tfull = bempty + 2;             // the eight sums of a chunk are complete
  uint64_t *tempty = tfull + 1;             // and have been read
  uint64_t *mdone = tempty + 1;             // every MMA issued by the CTA has completed
  uint32_t *tslot = reinterpret_cast<uint32_t *>(mdone + 1);
  // alpha partials per epilogue warp, over the B buffers once their last
  // MMAs are done
  double(*red)[NT] = reinterpret_cast<double(*)[NT]>(bbuf);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // N tiles fastest: the CTAs that share A's tiles run together
  const int m_tile = blockIdx.y, n_tile = blockIdx.x, split = blockIdx.z;
  const int kb1 = min(num_kb, (split + 1) * kb_per_split);
  const int kb0 = max(split * kb_per_split, e.lower ? m_tile * (BM / KB) : 0);
  const int nk = max(0, kb1 - kb0);
  const int chunks = (nk + CHUNK_KB - 1) / CHUNK_KB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::A_STAGES; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, EPI_WARPS);
    mbar_init(mdone, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tslot, C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      int na = 0, nb = 0;   // tiles issued
      bool ok = true;
      for (int it = 0; it < nk && ok; ++it) {
        const int bs = it & 1;
        if (!mbar_wait(&bempty[bs], ((it >> 1) & 1) ^ 1, e.status)) break;
        mbar_expect_tx(&bfull[bs], C::B_BYTES);
        for (int p = 0; p < S; p += C::BOX)
          tma_load_4d(bbuf + bs * C::B_BYTES + p * (NT * KB * 2), &tmB, &bfull[bs], 0, n_tile * NT,
                      kb0 + it, p);
        nb = it + 1;
        for (int i = 0; i < S; ++i, ++na) {
          const int as = na % C::A_STAGES;
          if (!mbar_wait(&aempty[as], ((na / C::A_STAGES) & 1) ^ 1, e.status)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&afull[as], C::A_BYTES);
          tma_load_4d(aring + as * C::A_BYTES, &tmA, &afull[as], 0, m_tile * BM, kb0 + it, i);
        }
      }
      // every issued copy must have landed before the CTA may exit
      for (int i = max(0, na - C::A_STAGES); i < na; ++i)
        mbar_wait(&afull[i % C::A_STAGES], (i / C::A_STAGES) & 1, e.status);
      for (int i = max(0, nb - 2); i < nb; ++i) mbar_wait(&bfull[i & 1], (i >> 1) & 1, e.status);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int na = 0;
      bool ok = true;
      for (int c = 0; c < chunks && ok; ++c) {
        if (c > 0 && !mbar_wait(tempty, (c - 1) & 1, e.status)) break;
        tc_fence_after();
        const int it1 = min(nk, (c + 1) * CHUNK_KB);
        for (int it = c * CHUNK_KB; it < it1 && ok; ++it) {
          const int bs = it & 1;
          if (!mbar_wait(&bfull[bs], (it >> 1) & 1, e.status)) {
            ok = false;
            break;
          }
          const uint64_t db = make_sdesc(smem_u32(bbuf + bs * C::B_BYTES));
#pragma unroll 1
          for (int i = 0; i < S; ++i, ++na) {
            const int as = na % C::A_STAGES;
            if (!mbar_wait(&afull[as], (na / C::A_STAGES) & 1, e.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t da = make_sdesc(smem_u32(aring + as * C::A_BYTES));
            // columns i NT .. 8 NT, split at 256: lo columns from B's first
            // rows, hi columns from the rows after them
            const int c0 = i * NT, hi0 = max(c0, 256);
            const int lo = max(0, min(256, S * NT) - c0), hi = max(0, S * NT - hi0);
            const uint32_t idlo = make_idesc(BM, lo), idhi = make_idesc(BM, hi);
            const uint64_t dbhi = db + (uint64_t)((hi0 - c0) * 128 >> 4);
            const uint64_t db8 = db + (uint64_t)((S - i) * NT * 128 >> 4);
#pragma unroll
            for (int kk = 0; kk < KB / 16; ++kk) {
              const uint32_t acc = (it > c * CHUNK_KB || i > 0 || kk > 0) ? 1u : 0u;
              if (lo > 0) umma_bf16(tmem + (uint32_t)c0, da + 2 * kk, db + 2 * kk, idlo, acc);
              if (hi > 0) umma_bf16(tmem + (uint32_t)hi0, da + 2 * kk, dbhi + 2 * kk, idhi, acc);
              // t = 8: digit 8 - i of B, into S_7
              if (i > 0)
                umma_bf16(tmem + 7 * NT, da + 2 * kk, db8 + 2 * kk, make_idesc(BM, NT), 1u);
            }
            umma_commit(&aempty[as]);
          }
          if (ok) umma_commit(&bempty[bs]);
        }
        if (ok) umma_commit(tfull);
      }
      // no MMA may still write TMEM when it is freed (also after a timeout)
      umma_commit(mdone);
      mbar_wait(mdone, 0, e.status);
    }
  } else {
    // ------------------------------ epilogue ------------------------------
    // warp & 3 is the TMEM lane quarter a warp can read
    const int qd = warp & 3, half = (warp - 2) >> 2;
    const int row = m_tile * BM + qd * 32 + lane;
    const bool rok = row < M;
    const int fa = rok ? e.ea[row] : 1;
    const bool with_q = e.mode == OZ_LANCZOS || e.mode == OZ_APPLY;
    const bool with_prev = e.mode == OZ_LANCZOS && e.qprev != nullptr;
    double d2 = 0.0, cdr = 0.0;
    if (rok && with_q) {
      d2 = e.Delta2[row];
      cdr = e.cd[row];
    } else if (rok && e.mode == OZ_START) {
      cdr = e.dsq[row];
    }
    double *out = e.out + (e.mode == OZ_PART ? (size_t)split * Ncols * e.ldo : 0);
    __shared__ LossShared loss;
    const bool do_f64 =
        CHECK && !digits_do<NT>(e, m_tile * BM, n_tile * NT, M, Ncols, num_kb, loss);
    for (int c = 0; c < chunks; ++c) {
      if (!mbar_wait(tfull, c & 1, e.status)) break;
      tc_fence_after();
      const bool last = c + 1 == chunks;
      const bool add_old = c > 0 || e.mode == OZ_ADD;
#pragma unroll 1
      for (int c8 = half * (NT / 2); c8 < (half + 1) * (NT / 2); c8 += 8) {
        const int col0 = n_tile * NT + c8;
        if (col0 >= Ncols) break;
        const uint32_t tc0 = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)c8;
        float s[S][8];
#pragma unroll
        for (int t = 0; t < S; ++t)
          tmem_ld8(tc0 + (uint32_t)(t * NT), s[t]);
        // everything the eight columns need from memory, before the first use
        double old[8], qv[8], qp[8];
        int fb[8];
        double *o = out + (size_t)col0 * e.ldo + row;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const bool ok = rok && col0 + i < Ncols;
          const size_t oi = (size_t)(col0 + i) * e.ldo + row;
          fb[i] = ok ? e.eb[col0 + i] : 1;
          old[i] = ok && add_old ? o[(size_t)i * e.ldo] : 0.0;
          qv[i] = ok && last && with_q ? e.q[oi] : 0.0;
          qp[i] = ok && last && with_prev ? e.qprev[oi] : 0.0;
        }
        tmem_ld_wait();
#pragma unroll
        for (int t = 0; t < S; ++t)
#pragma unroll
          for (int i = 0; i < 8; ++i) asm volatile("" : "+f"(s[t][i]));   // no use before the wait
        double v[8], part[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float v8[S];
#pragma unroll
          for (int t = 0; t < S; ++t) v8[t] = s[t][i];
          // row scales 2^(field - 1022); a non-finite row gives NaN
          v[i] = join_sums(v8, max(fa, 1) + max(fb[i], 1) - 2044 - 52);
          if (fa >= 2047 || fb[i] >= 2047) v[i] = __longlong_as_double(0x7ff8000000000000LL);
          part[i] = 0.0;
        }
        if (e.mode == OZ_ADD) {
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = fma(e.scale, v[i], old[i]);
        } else {
          if (c > 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] += old[i];
          }
          if (last && e.mode == OZ_START) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = cdr * v[i];
          } else if (last && with_q) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              v[i] = fma(d2, qv[i], cdr * v[i]);
              if (with_prev) v[i] = fma(-(col0 + i < Ncols ? e.betaj[col0 + i] : 0.0), qp[i], v[i]);
              part[i] = rok ? qv[i] * v[i] : 0.0;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (rok && col0 + i < Ncols) o[(size_t)i * e.ldo] = v[i];
        if (e.alpha_part != nullptr && last) {
          // the eight columns' sums over the warp's rows: a transposed
          // butterfly (lane bits 2..0 pick the column), then bits 3 and 4
#pragma unroll
          for (int off = 4; off >= 1; off >>= 1) {
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < off; ++i) {
              const double send = up ? part[i] : part[i + off];
              const double keep = up ? part[i + off] : part[i];
              part[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
          }
          part[0] += __shfl_xor_sync(0xffffffffu, part[0], 8);
          part[0] += __shfl_xor_sync(0xffffffffu, part[0], 16);
          if (lane < 8) red[qd][c8 + lane] = part[0];
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty);
    }
    if (CHECK && do_f64) {
      epi_sync();   // the tile's stores come first
      tile_f64<NT>(e, m_tile * BM, n_tile * NT, M, Ncols);
    }
    if (e.alpha_part != nullptr && chunks > 0) {
      epi_sync();
      for (int i = threadIdx.x - 64; i < 2 * NT; i += 32 * EPI_WARPS) {
        const int hf = i / NT, col = i % NT, b = n_tile * NT + col;
        if (b < Ncols && m_tile * BM + 64 * hf < M)
          e.alpha_part[(size_t)(2 * m_tile + hf) * Ncols + b] =
              red[2 * hf][col] + red[2 * hf + 1][col];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// Digits of an operand
// ---------------------------------------------------------------------------
// 16 consecutive K elements of one operand row into its eight digit planes
__device__ __forceinline__ void store_digits16(const unsigned long long (&u)[16], uint16_t *dst,
                                               size_t plane) {
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      w[i] = digit_bf16(u[2 * i], s) | (digit_bf16(u[2 * i + 1], s) << 16);
    uint4 *o = reinterpret_cast<uint4 *>(dst + s * plane);
    o[0] = make_uint4(w[0], w[1], w[2], w[3]);
    o[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// Shift that brings a contraction index whose largest exponent field is e to a
// common scale, 0 .. 800: up in one operand, down in the other (exactly; indices
// beyond 2^+-400 come as near as that).
__device__ __forceinline__ int even_shift(int e) {
  return e > 0 ? 1423 - min(max(e, 623), 1423) : 0;
}

// A matrix in memory: element (r, c) = x[r * ld + c], times scale[c] where
// given, inside [nr][nc], zero outside; times 2^lift(r, c), which is added to
// the exponents (a multiplication would take the FP64 pipe).  shift and rshift
// are shifts by column and by row; even: shift holds exponent fields instead,
// for even_shift up; reven: exponent fields by row, for even_shift down.
struct Src {
  const double *x, *scale;
  const int *shift, *rshift, *reven;
  bool even;
  size_t ld;
  int nr, nc;
  __device__ __forceinline__ double at(int r, int c) const {
    if (r >= nr || c >= nc) return 0.0;
    const double v = x[(size_t)r * ld + c];
    return scale ? scale[c] * v : v;
  }
  __device__ __forceinline__ int lift(int r, int c) const {
    int s = rshift && r < nr ? rshift[r] : 0;
    if (reven && r < nr) s -= even_shift(reven[r]);
    if (shift && c < nc) s += even ? even_shift(shift[c]) : shift[c];
    return s;
  }
};

// Exponent field of x 2^sh, 0 for zero; subnormals count as the smallest
// normal numbers.
__device__ __forceinline__ int lifted_field(double x, int sh) {
  return nonzero_bits(x) ? max(exp_field(x), 1) + sh : 0;
}

// Largest exponent field of each operand row: the operand's rows are the
// matrix's rows (COLS = false, contraction along c) or its columns.  finite:
// Inf and NaN do not count.  LIFT: with src's shifts (the vectors of every step
// have none: 12 us for 64 of 32768 elements, 17 with the questions for them).
template <bool COLS, bool LIFT>
__global__ void __launch_bounds__(256) k_oz_max(Src src, int *__restrict__ e, bool finite) {
  pdl_wait();
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  const int r = COLS ? r0 + (threadIdx.x >> 6) : r0 + (threadIdx.x >> 2);
  const int c = COLS ? c0 + (threadIdx.x & 63) : c0 + (threadIdx.x & 3) * 16;
  constexpr int DR = COLS ? 4 : 0, DC = COLS ? 0 : 1;
  double v[16];
  int sh[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = src.at(r + DR * i, c + DC * i);
#pragma unroll
  for (int i = 0; i < 16; ++i) sh[i] = LIFT ? src.lift(r + DR * i, c + DC * i) : 0;
  int m = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int f = LIFT ? lifted_field(v[i], sh[i]) : exp_field(v[i]);
    if (!(finite && exp_field(v[i]) == 2047)) m = max(m, f);
  }
  if (COLS) {
    if (m > 0) atomicMax(&e[c], m);
  } else {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    if ((threadIdx.x & 3) == 0 && m > 0) atomicMax(&e[r], m);
  }
}

// blk[kb] of an operand row from the four threads that hold its 64 elements
// (subnormals count as zeros)
__device__ __forceinline__ void store_block_exp(int m, int part, short *blk) {
  const unsigned quad = 0xfu << (threadIdx.x & 28);
  m = max(m, __shfl_xor_sync(quad, m, 1));
  m = max(m, __shfl_xor_sync(quad, m, 2));
  if (part == 0) *blk = (short)(m > 0 ? m : OZ_ZERO);
}

// Digits of a 64 x 64 tile; the operand has `rows` rows and nkb K blocks.
// LIFT: with src's shifts and, where asked for, block exponents.
template <bool COLS, bool LIFT>
__global__ void __launch_bounds__(256) k_oz_slice(Src src, const int *__restrict__ e,
                                                  uint16_t *__restrict__ out, int rows, int nkb,
                                                  short *__restrict__ blk) {
  pdl_wait();
  __shared__ double tile[COLS ? 64 : 1][65];
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  const int i = threadIdx.x >> 2, k0 = (threadIdx.x & 3) * 16;   // row and K offset in the tile
  if (COLS) {
    for (int r = threadIdx.x >> 6; r < 64; r += 4)
      tile[r][threadIdx.x & 63] = src.at(r0 + r, c0 + (threadIdx.x & 63));
    __syncthreads();
  }
  const int row = (COLS ? c0 : r0) + i, kb = COLS ? blockIdx.y : blockIdx.x;
  if (row >= rows || kb >= nkb) return;
  const int f = max(e[row], 1);
  unsigned long long u[16];
  int m = 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const double x = COLS ? tile[k0 + k][i] : src.at(row, c0 + k0 + k);
    const int sh = !LIFT ? 0 : COLS ? src.lift(r0 + k0 + k, row) : src.lift(row, c0 + k0 + k);
    u[k] = fixed56(x, f - sh);
    if (LIFT) m = max(m, lifted_field(x, sh));
  }
  if (LIFT && blk) store_block_exp(m, threadIdx.x & 3, blk + (size_t)row * nkb + kb);
  store_digits16(u, out + ((size_t)kb * rows + row) * 64 + k0, (size_t)nkb * rows * 64);
}

// One operand row per block, up to OZ_ROW_MAX elements: the sum of `splits`
// partials (fixed order, optionally stored to y), its exponent and its digits.
// Sixteen elements lie 17 doubles apart in shared memory: their readers meet
// different banks (8192 rows of 1024 with shifts and block exponents: 93 us,
// 101 without the gap).  LIFT: on src's even shifts, with block exponents to blk.
template <bool LIFT>
__global__ void __launch_bounds__(256) k_oz_rows(const double *__restrict__ x, int splits,
                                                 size_t part, Src src, double *__restrict__ y,
                                                 int *__restrict__ e, uint16_t *__restrict__ out,
                                                 int rows, int nkb, short *__restrict__ blk) {
  extern __shared__ double v[];
  __shared__ int wmax[8];
  pdl_wait();
  const int r = blockIdx.x;
  int m = 0;
  for (int i = threadIdx.x; i < nkb * 64; i += 256) {
    double s = 0.0;
    if (r < src.nr && i < src.nc) {
      const size_t o = (size_t)r * src.ld + i;
      for (int p = 0; p < splits; ++p) s += x[(size_t)p * part + o];
      if (y) y[o] = s;
      if (src.scale) s *= src.scale[i];
    }
    v[i + (i >> 4)] = s;
    if (LIFT)
      m = max(m, lifted_field(s, even_shift(src.shift[i])));
    else
      m = max(m, exp_field(s));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int w = 0; w < 8; ++w) m = max(m, wmax[w]);
  if (threadIdx.x == 0) e[r] = m;
  m = max(m, 1);
  for (int g = threadIdx.x; g < nkb * 4; g += 256) {
    unsigned long long u[16];
    int mb = 0, ev[16];   // shift covers whole K blocks
    if (LIFT) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<int4 *>(ev + 4 * q) =
            *reinterpret_cast<const int4 *>(src.shift + g * 16 + 4 * q);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const double s = v[g * 17 + k];
      const int sh = LIFT ? even_shift(ev[k]) : 0;
      u[k] = fixed56(s, m - sh);
      if (LIFT) mb = max(mb, lifted_field(s, sh));
    }
    if (LIFT) store_block_exp(mb, g & 3, blk + (size_t)r * nkb + (g >> 2));
    store_digits16(u, out + ((size_t)(g >> 2) * rows + r) * 64 + (g & 3) * 16,
                   (size_t)nkb * rows * 64);
  }
}

// Largest exponent fields of the rows and of the columns of x [nr][nc] in one
// pass, with the rows' and columns' own shifts: row[r] of x 2^shift[c], col[c]
// of x 2^rshift[r].  nc a multiple of 64; a block takes 256 rows by 64 columns.
__global__ void __launch_bounds__(256) k_oz_max_both(const double *__restrict__ x, int nr, int nc,
                                                     const int *__restrict__ shift,
                                                     const int *__restrict__ rshift,
                                                     int *__restrict__ row, int *__restrict__ col) {
  pdl_wait();
  const int c = blockIdx.x * 64 + (threadIdx.x & 63), r0 = blockIdx.y * 256;
  const int sc = shift ? shift[c] : 0;
  int m = 0;
#pragma unroll 4
  for (int r = r0 + (threadIdx.x >> 6); r < min(nr, r0 + 256); r += 4) {   // alike in a warp
    const double v = x[(size_t)r * nc + c];
    m = max(m, lifted_field(v, rshift ? rshift[r] : 0));
    const int mr = __reduce_max_sync(0xffffffffu, lifted_field(v, sc));
    if ((threadIdx.x & 31) == 0 && mr > 0) atomicMax(&row[r], mr);
  }
  if (m > 0) atomicMax(&col[c], m);
}

// Balance of a factor along its rows (block 0) and its columns (block 1), from
// their largest exponent fields e_k: shifts s_k = max e - e_k that even the
// factor out, and the vectors' factors 2^-s_k (0 where the factor is zero) and
// base_k 2^-s_k.  Shifts end at 400.  The fields are left at zero for the next
// pass; *bad != 0 if one says Inf or NaN.
__global__ void __launch_bounds__(1024) k_oz_factors(OzBalance rows, OzBalance cols,
                                                     unsigned *bad) {
  pdl_wait();
  const OzBalance o = blockIdx.x == 0 ? rows : cols;
  __shared__ int top;
  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  int m = 0;
  for (int k = threadIdx.x; k < o.n; k += 1024) m = max(m, o.e[k]);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(&top, m);
  __syncthreads();
  if (threadIdx.x == 0 && top >= 2047) atomicOr(bad, 1u);
  for (int k = threadIdx.x; k < o.n; k += 1024) {
    const int e = o.e[k], s = e > 0 ? min(top - e, 400) : 0;
    const double f = e > 0 ? __hiloint2double((1023 - s) << 20, 0) : 0.0;
    o.e[k] = 0;
    o.shift[k] = s;
    o.down[k] = f;
    if (o.base) o.based[k] = o.base[k] * f;
  }
}

static PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 f = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return f;
}

// Map of an operand's digits: (64 elements, rows, K blocks, slices)
static bool encode(CUtensorMap *tm, const OzOperand &o, int box_rows, int box_slices) {
  auto enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[4] = {64, (cuuint64_t)o.rows, (cuuint64_t)o.nkb, (cuuint64_t)S};
  cuuint64_t strides[3] = {128, (cuuint64_t)o.rows * 128, (cuuint64_t)o.nkb * o.rows * 128};
  cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, (cuuint32_t)box_slices};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t *>(o.d), dims, strides,
             box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int NT, bool CHECK>
static void launch(const CUtensorMap &A, const CUtensorMap &B, int M, int Ncols, int nkb, int per,
                   int splits, const Epi &e, cudaStream_t st) {
  static DeviceOnce once;
  allow_smem(once, k_oz_gemm<NT, CHECK>, Cfg<NT>::SMEM);
  const dim3 grid((Ncols + NT - 1) / NT, (M + BM - 1) / BM, splits);
  launch_pdl(k_oz_gemm<NT, CHECK>, grid, dim3(NTHREADS), Cfg<NT>::SMEM, st, A, B, M, Ncols, nkb,
             per, e);
}

template <int NT>
static void launch_any(const CUtensorMap &A, const CUtensorMap &B, int M, int Ncols, int nkb,
                       int per, int splits, const Epi &e, cudaStream_t st) {
  if (e.ba)
    launch<NT, true>(A, B, M, Ncols, nkb, per, splits, e, st);
  else
    launch<NT, false>(A, B, M, Ncols, nkb, per, splits, e, st);
}

template <bool LIFT>
static void launch_rows(const double *x, int splits, size_t part, const Src &src, double *y,
                        const OzOperand &o, cudaStream_t st) {
  static DeviceOnce once;
  allow_smem(once, k_oz_rows<LIFT>, OZ_ROW_MAX / 16 * 17 * sizeof(double));
  launch_pdl(k_oz_rows<LIFT>, dim3(o.rows), dim3(256), (size_t)o.nkb * 68 * sizeof(double), st, x,
             splits, part, src, y, o.e, o.d, o.rows, o.nkb, o.blk);
}

// Exponents (into zeros), then digits, by tiles of 64 x 64.
template <bool COLS, bool LIFT>
static void launch_tiles(const Src &src, const OzOperand &o, cudaStream_t st) {
  const int kr = COLS ? o.nkb : (o.rows + 63) / 64, kc = COLS ? (o.rows + 63) / 64 : o.nkb;
  launch_pdl(k_oz_max<COLS, LIFT>, dim3((src.nc + 63) / 64, (src.nr + 63) / 64), dim3(256), 0, st,
             src, o.e, false);
  launch_pdl(k_oz_slice<COLS, LIFT>, dim3(kc, kr), dim3(256), 0, st, src, o.e, o.d, o.rows, o.nkb,
             o.blk);
}

}  // namespace oz

int oz_splits(int M, int ncols, int nkb) { return oz::k_splits(M, ncols, nkb, device_sms()); }

size_t oz_part_rows(int M, int rows, int slice, int nkb) {
  return oz::part_rows(M, rows, slice, nkb, device_sms());
}

bool launch_oz_gemm(const OzOperand &A, const OzOperand &B, int M, int Ncols, int splits,
                    const OzOut &o, unsigned *status, cudaStream_t st) {
  oz::Epi e{};
  e.mode = o.mode;
  e.ea = A.e;
  e.eb = B.e;
  e.out = o.out;
  e.ldo = o.ldo;
  e.scale = o.scale;
  e.lower = o.lower ? 1 : 0;
  e.Delta2 = o.Delta2;
  e.dsq = o.dsq;
  e.cd = o.cd;
  e.q = o.q;
  e.qprev = o.qprev;
  e.betaj = o.betaj;
  e.alpha_part = o.alpha_part;
  e.status = status;
  if (o.xa) {
    if (o.mode != OZ_PART || splits != 1 || !A.blk || !B.blk) return false;
    e.ba = A.blk;
    e.bb = B.blk;
    e.xa = o.xa;
    e.xb = o.xb;
    e.ldxa = o.ldxa;
    e.ldxb = o.ldxb;
    e.K = o.K;
  }
  const int nkb = A.nkb, per = (nkb + splits - 1) / splits;
  const int m_tiles = (M + oz::BM - 1) / oz::BM;
  const int nt =
      oz::tile_cols(m_tiles, Ncols, o.mode == OZ_PART ? std::min(64, nkb) : 1, device_sms());
  CUtensorMap ta, tb;
  if (A.rows < oz::BM || B.rows < nt || A.nkb != B.nkb || !oz::encode(&ta, A, oz::BM, 1) ||
      !oz::encode(&tb, B, nt, nt == 64 ? oz::Cfg<64>::BOX : OZ_SLICES))
    return false;
  if (nt == 64)
    oz::launch_any<64>(ta, tb, M, Ncols, nkb, per, splits, e, st);
  else if (nt == 32)
    oz::launch_any<32>(ta, tb, M, Ncols, nkb, per, splits, e, st);
  else
    oz::launch_any<16>(ta, tb, M, Ncols, nkb, per, splits, e, st);
  return true;
}

// Digits of x [nr][nc] (row stride ld, optional column scale): operand rows
// are x's rows, or its columns.  up: exponent fields of x's columns (nc rounded
// up to 64 of them) to shift up by, down: of its rows to shift down by.  o.rows covers them (more rows become zeros).
void launch_oz_slice(const double *x, size_t ld, int nr, int nc, const double *scale, bool cols,
                     const OzOperand &o, cudaStream_t st, const int *up, const int *down) {
  const oz::Src src{x, scale, up, nullptr, down, true, ld, nr, nc};
  // short rows: one kernel, a block per row (4.7 us at 160 rows of 256); longer
  // ones spread each row over many blocks (64 rows of 32768: 12 + 20 us)
  if (!cols && !down && o.nkb * 64 <= 4096) {
    if (up)
      oz::launch_rows<true>(x, 1, 0, src, nullptr, o, st);
    else
      oz::launch_rows<false>(x, 1, 0, src, nullptr, o, st);
    return;
  }
  cudaMemsetAsync(o.e, 0, sizeof(int) * o.rows, st);
  if (cols && (up || down))
    oz::launch_tiles<true, true>(src, o, st);
  else if (cols)
    oz::launch_tiles<true, false>(src, o, st);
  else if (up || down)
    oz::launch_tiles<false, true>(src, o, st);
  else
    oz::launch_tiles<false, false>(src, o, st);
}

// y [rows][len] = sum of the split partials, and the digits of o.scale y (len
// <= OZ_ROW_MAX)
void launch_oz_reduce(const double *part, int splits, int nr, int len, double *y,
                      const OzOperand &o, cudaStream_t st) {
  const oz::Src src{part, o.scale, nullptr, nullptr, nullptr, false, (size_t)len, nr, len};
  oz::launch_rows<false>(part, splits, (size_t)nr * len, src, y, o, st);
}

void launch_oz_max_both(const double *x, int nr, int nc, const int *shift, const int *rshift,
                        int *row, int *col, cudaStream_t st) {
  launch_pdl(oz::k_oz_max_both, dim3(nc / 64, (nr + 255) / 256), dim3(256), 0, st, x, nr, nc,
             shift, rshift, row, col);
}

void launch_oz_factors(const OzBalance &rows, const OzBalance &cols, unsigned *bad,
                       cudaStream_t st) {
  launch_pdl(oz::k_oz_factors, dim3(2), dim3(1024), 0, st, rows, cols, bad);
}

// Digits of x [nr][nc] whose rows' (columns') exponents are in o.e already.
void launch_oz_digits(const double *x, int nr, int nc, bool cols, const int *shift,
                      const OzOperand &o, cudaStream_t st) {
  const oz::Src src{x, nullptr, cols ? nullptr : shift, cols ? shift : nullptr, nullptr, false,
                    (size_t)nc, nr, nc};
  const dim3 grid(cols ? (o.rows + 63) / 64 : o.nkb, cols ? o.nkb : (o.rows + 63) / 64);
  if (cols)
    launch_pdl(oz::k_oz_slice<true, true>, grid, dim3(256), 0, st, src, o.e, o.d, o.rows, o.nkb, o.blk);
  else
    launch_pdl(oz::k_oz_slice<false, true>, grid, dim3(256), 0, st, src, o.e, o.d, o.rows, o.nkb, o.blk);
}

void launch_oz_col_max(const double *x, size_t ld, int nr, int nc, int *e, cudaStream_t st) {
  cudaMemsetAsync(e, 0, sizeof(int) * round_up(nc, 64), st);
  constexpr int ROWS = 1 << 21;   // a grid's second dimension ends at 65535 tiles
  for (int r0 = 0; r0 < nr; r0 += ROWS) {
    const int n = std::min(ROWS, nr - r0);
    const oz::Src src{x + (size_t)r0 * ld, nullptr, nullptr, nullptr, nullptr, false, ld, n, nc};
    launch_pdl(oz::k_oz_max<true, false>, dim3((nc + 63) / 64, (n + 63) / 64), dim3(256), 0, st, src, e,
               true);
  }
}

}  // namespace lgw
