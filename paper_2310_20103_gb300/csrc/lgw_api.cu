// C ABI of the lgw library: argument checks, host/device staging, workspace
// management and the per-sub-batch schedule of the hot path.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "lgw_internal.cuh"

using namespace lgw;

struct lgw_handle {
  int device = 0;
  cudaStream_t stream = nullptr;
  lgw_status last = LGW_OK;
  std::string msg;
  unsigned *d_status = nullptr;
  struct Buf {
    void *p = nullptr;
    size_t n = 0;
  };
  std::map<std::string, Buf> bufs;
  size_t ws_limit = 0;   // bytes the workspace may hold (0: no limit)
  size_t ws_bytes = 0;   // bytes it holds
  int launches = 0;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used = 0;
  bool timing = false;
  // captured sub-batch graphs; ws_gen changes whenever a workspace buffer is
  // (re)allocated, which also drops every cached graph
  struct Graph {
    cudaGraphExec_t exec = nullptr;
    int launches = 0;
  };
  std::map<std::string, Graph> graphs;
  unsigned long long ws_gen = 0;
  cudaStream_t cap_stream = nullptr;   // private non-blocking stream for captures
  // lgw_sigma_c_batched runs systems concurrently on these streams, each
  // with its own workspace namespace (ws_prefix)
  std::vector<cudaStream_t> lanes;
  std::string ws_prefix;
  std::vector<lgw_system *> sliced;   // systems that hold digits of L (k_gemm_oz.cu)
  // device memory of systems: the size of every block, and the blocks of
  // released systems that the next one may take (SPARE_MAX bytes at most)
  std::mutex mem_mu;
  std::map<void *, size_t> sys_mem;
  std::multimap<size_t, void *> spare;
  size_t spare_bytes = 0;
  void drop_graphs() {
    for (auto &kv : graphs)
      if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
    graphs.clear();
  }
};

struct lgw_system {
  lgw_handle *h = nullptr;
  SysDev s{};
  // spectral interval of C for the polynomial form, estimated on first use
  bool ivl_ok = false;
  double ivl_lo = 0.0, ivl_hi = 0.0;
  __nv_bfloat16 *Ltb_lo = nullptr;   // bf16(L - bf16(L))^T [A][N], made on first use
  // Tamm-Dancoff view (A = Delta + (c_K/2) L L^T in place of C), made on first use
  SysDev tda{};
  void *tda_buf = nullptr;
  // digits of L for the FP64 products: 1 made, 0 not (not asked for yet, or no
  // memory when last asked), -1 never (L holds Inf or NaN)
  int oz_state = 0;
  void *oz_buf = nullptr;
  const double *ozx_tda = nullptr;   // SysDev::ozx of the Tamm-Dancoff view
};

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------
namespace {

struct Fail {
  lgw_status st;
};

lgw_status set_err(lgw_handle *h, lgw_status st, const char *fmt, ...) {
  if (h) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    h->last = st;
    h->msg = buf;
  }
  return st;
}

#define LGW_TRY_CUDA(h, call)                                                             \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) {                                                              \
      set_err((h), e_ == cudaErrorMemoryAllocation ? LGW_ERR_OOM : LGW_ERR_CUDA,          \
              "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
      throw Fail{(h)->last};                                                              \
    }                                                                                     \
  } while (0)

void check_launch(lgw_handle *h, const char *what) {
  h->launches++;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_err(h, LGW_ERR_CUDA, "launch of %s failed: %s", what, cudaGetErrorString(e));
    throw Fail{h->last};
  }
}

// Memory of systems.  A gradient prepares and releases a system in each of its
// two passes, and the driver maps and unmaps its memory every time: 3.1 ms of
// cudaMalloc and cudaFree in the 19.2 ms of an exact gradient at N_vc 32768,
// N_aux 1024 (1.5 GB).  A handle therefore keeps up to 2 GiB of released
// blocks for its next system (all handles of the process together: less than
// 1% of the device); they go back with lgw_release_workspace, lgw_destroy, when
// a byte limit is set, and before any allocation of the handle is refused.
constexpr size_t SPARE_MAX = (size_t)2 << 30;
std::atomic<size_t> spare_total{0};

void spare_free(lgw_handle *h) {
  std::lock_guard<std::mutex> lock(h->mem_mu);
  for (auto &kv : h->spare) {
    cudaFree(kv.second);
    h->sys_mem.erase(kv.second);
  }
  h->spare.clear();
  spare_total -= h->spare_bytes;
  h->spare_bytes = 0;
}

// NULL (and no sticky error) where the device has no room.
void *sys_alloc(lgw_handle *h, size_t bytes) {
  {
    // the smallest spare block that fits and wastes at most a quarter
    std::lock_guard<std::mutex> lock(h->mem_mu);
    auto it = h->spare.lower_bound(bytes);
    if (it != h->spare.end() && it->first <= bytes + bytes / 4) {
      void *p = it->second;
      h->spare_bytes -= it->first;
      spare_total -= it->first;
      h->spare.erase(it);
      return p;
    }
  }
  void *p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    spare_free(h);
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
  }
  std::lock_guard<std::mutex> lock(h->mem_mu);
  h->sys_mem[p] = bytes;
  return p;
}

// The caller has waited for the work that uses the block.
void sys_free(lgw_handle *h, void *p) {
  if (!p) return;
  std::lock_guard<std::mutex> lock(h->mem_mu);
  const auto it = h->sys_mem.find(p);
  const size_t n = it->second;
  if (h->ws_limit == 0) {
    if (spare_total.fetch_add(n) + n <= SPARE_MAX) {
      h->spare.emplace(n, p);
      h->spare_bytes += n;
      return;
    }
    spare_total -= n;
  }
  h->sys_mem.erase(it);
  cudaFree(p);
}

void free_digits(lgw_system *sys) {
  sys_free(sys->h, sys->oz_buf);
  sys->oz_buf = nullptr;
  sys->s.ozA = sys->s.ozT = sys->tda.ozA = sys->tda.ozT = OzOperand{};
  sys->s.ozx = sys->s.ozy = sys->tda.ozx = sys->tda.ozy = sys->ozx_tda = nullptr;
  sys->oz_state = 0;
}

// Gives back every system's digits of L, the workspace of the digits (oz_*
// buffers) and the spare blocks; the FP64 products then run on the CUDA cores.  False if
// there was nothing to give back.
bool drop_digits(lgw_handle *h) {
  bool any = !h->sliced.empty() || h->spare_bytes != 0;
  for (auto &kv : h->bufs) any = any || (kv.first.find("oz_") != std::string::npos && kv.second.p);
  if (!any) return false;
  cudaDeviceSynchronize();
  for (lgw_system *sys : h->sliced) free_digits(sys);
  h->sliced.clear();
  spare_free(h);
  for (auto &kv : h->bufs)
    if (kv.first.find("oz_") != std::string::npos && kv.second.p) {
      cudaFree(kv.second.p);
      h->ws_bytes -= kv.second.n;
      kv.second = lgw_handle::Buf{};
    }
  h->ws_gen++;
  h->drop_graphs();
  return true;
}

// A workspace buffer of at least `bytes`.  optional (the digits of the FP64
// products): NULL where the device's memory does not allow it, and on a
// handle with a byte limit, which is kept for the buffers every call needs.
void *ws(lgw_handle *h, const std::string &name, size_t bytes, bool optional = false) {
  auto &b = h->bufs[h->ws_prefix + name];
  if (bytes == 0) bytes = 8;
  if (optional && h->ws_limit) return nullptr;
  if (b.n < bytes) {
    // the handle's byte limit is checked before anything is freed, so a
    // refused request leaves the workspace as it was
    if (h->ws_limit && h->ws_bytes - b.n + bytes > h->ws_limit) {
      set_err(h, LGW_ERR_OOM,
              "workspace limit: %s needs %zu bytes, the handle holds %zu of its %zu-byte limit",
              name.c_str(), bytes, h->ws_bytes, h->ws_limit);
      throw Fail{LGW_ERR_OOM};
    }
    if (b.p) {
      LGW_TRY_CUDA(h, cudaStreamSynchronize(h->stream));
      cudaFree(b.p);
      h->ws_bytes -= b.n;
      b.p = nullptr;
      b.n = 0;
    }
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation && h->spare_bytes != 0) {
      cudaGetLastError();
      spare_free(h);
      e = cudaMalloc(&p, bytes);
    }
    if (e == cudaErrorMemoryAllocation && !optional && drop_digits(h)) {
      cudaGetLastError();
      e = cudaMalloc(&p, bytes);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      if (optional) return nullptr;
      set_err(h, LGW_ERR_OOM, "cudaMalloc(%zu bytes) for %s failed: %s", bytes, name.c_str(),
              cudaGetErrorString(e));
      throw Fail{LGW_ERR_OOM};
    }
    b.p = p;
    b.n = bytes;
    h->ws_bytes += bytes;
    h->ws_gen++;
    h->drop_graphs();
  }
  return b.p;
}

template <class T>
T *wsT(lgw_handle *h, const std::string &name, size_t count) {
  return static_cast<T *>(ws(h, name, count * sizeof(T)));
}

bool is_device_ptr(const void *p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Device view of an input: the pointer itself, or a staged copy.
template <class T>
const T *in_dev(lgw_handle *h, const std::string &name, const T *p, size_t count) {
  if (!p || count == 0) return p;
  if (is_device_ptr(p)) return p;
  T *d = wsT<T>(h, name, count);
  LGW_TRY_CUDA(h, cudaMemcpyAsync(d, p, count * sizeof(T), cudaMemcpyHostToDevice, h->stream));
  return d;
}

// Host copy of a small array given on either side.
template <class T>
std::vector<T> to_host(lgw_handle *h, const T *p, size_t count) {
  std::vector<T> v(count);
  if (count == 0) return v;
  if (is_device_ptr(p)) {
    LGW_TRY_CUDA(h, cudaMemcpyAsync(v.data(), p, count * sizeof(T), cudaMemcpyDeviceToHost,
                                    h->stream));
    LGW_TRY_CUDA(h, cudaStreamSynchronize(h->stream));
  } else {
    std::memcpy(v.data(), p, count * sizeof(T));
  }
  return v;
}

// Output staging: compute into a device buffer, copy back if the caller's
// pointer is host memory.
template <class T>
struct OutBuf {
  T *user = nullptr;
  T *dev = nullptr;
  size_t count = 0;
  bool host = false;
  void init(lgw_handle *h, const std::string &name, T *p, size_t n) {
    user = p;
    count = n;
    if (!p) {
      dev = nullptr;
      return;
    }
    host = !is_device_ptr(p);
    dev = host ? wsT<T>(h, name, n) : p;
  }
  void finish(lgw_handle *h) {
    if (user && host && count)
      LGW_TRY_CUDA(h, cudaMemcpyAsync(user, dev, count * sizeof(T), cudaMemcpyDeviceToHost,
                                      h->stream));
  }
};

struct Timer {
  lgw_handle *h;
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> spans;
  cudaEvent_t open = nullptr;
  int open_cat = -1;
  explicit Timer(lgw_handle *hh) : h(hh) {}
  cudaEvent_t ev() {
    if (h->ev_used == h->ev_pool.size()) {
      cudaEvent_t e;
      LGW_TRY_CUDA(h, cudaEventCreate(&e));
      h->ev_pool.push_back(e);
    }
    return h->ev_pool[h->ev_used++];
  }
  // Close the running span (if any) and open one for category `cat`.
  void mark(int cat) {
    if (!h->timing) return;
    cudaEvent_t e = ev();
    LGW_TRY_CUDA(h, cudaEventRecord(e, h->stream));
    if (open) spans.push_back({open_cat, {open, e}});
    open = e;
    open_cat = cat;
  }
  void stop() {
    if (!h->timing || !open) return;
    cudaEvent_t e = ev();
    LGW_TRY_CUDA(h, cudaEventRecord(e, h->stream));
    spans.push_back({open_cat, {open, e}});
    open = nullptr;
  }
  void collect(double *acc, int ncat) {
    if (!h->timing) return;
    LGW_TRY_CUDA(h, cudaStreamSynchronize(h->stream));
    for (auto &s : spans) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, s.second.first, s.second.second);
      if (s.first >= 0 && s.first < ncat) acc[s.first] += ms;
    }
    spans.clear();
  }
};

enum Cat { C_START, C_GEMM1, C_GEMM2, C_DOTS, C_UPDATE, C_PASS2, C_NORM, C_SPEC, C_CF, C_QP, C_N };

void check_status(lgw_handle *h) {
  unsigned st = 0;
  LGW_TRY_CUDA(h, cudaMemcpyAsync(&st, h->d_status, sizeof st, cudaMemcpyDeviceToHost, h->stream));
  LGW_TRY_CUDA(h, cudaStreamSynchronize(h->stream));
  if (st & ST_TIMEOUT) {
    set_err(h, LGW_ERR_TIMEOUT, "a bounded device wait ran out");
    throw Fail{LGW_ERR_TIMEOUT};
  }
  if (st & ST_BAD_INPUT) {
    set_err(h, LGW_ERR_SHAPE, "a tridiagonal depth k_eff lies outside [0, k]");
    throw Fail{LGW_ERR_SHAPE};
  }
  if (st & ST_NOT_SPD) {
    set_err(h, LGW_ERR_NOT_SPD, "non-positive pair energy or Gauss node (C not positive definite)");
    throw Fail{LGW_ERR_NOT_SPD};
  }
  if (st & ST_NO_CONV) {
    set_err(h, LGW_ERR_NO_CONVERGENCE, "tridiagonal eigensolver or QP equation did not converge");
    throw Fail{LGW_ERR_NO_CONVERGENCE};
  }
}

// Replay the cached graph for `key`, capturing `body` into it first if it
// is not cached.  A failed capture runs `body` eagerly instead.
template <class F>
void run_graphed(lgw_handle *h, const std::string &key, F &&body) {
  cudaStream_t st = h->stream;
  auto it = h->graphs.find(key);
  if (it == h->graphs.end()) {
    if (h->graphs.size() >= 64) h->drop_graphs();
    // the caller's stream may be the legacy default stream, which cannot be
    // captured: record the launches on the handle's own stream (the graph is
    // then launched on the caller's stream, which orders it)
    if (!h->cap_stream)
      LGW_TRY_CUDA(h, cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    const int l0 = h->launches;
    LGW_TRY_CUDA(h, cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
    cudaGraph_t g = nullptr;
    h->stream = h->cap_stream;
    try {
      body();
    } catch (Fail &) {
      h->stream = st;
      cudaStreamEndCapture(h->cap_stream, &g);
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      throw;
    }
    h->stream = st;
    cudaError_t e = cudaStreamEndCapture(h->cap_stream, &g);
    cudaGraphExec_t ex = nullptr;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&ex, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      cudaGetLastError();
      h->launches = l0;
      body();
      return;
    }
    lgw_handle::Graph gr;
    gr.exec = ex;
    gr.launches = h->launches - l0;
    h->launches = l0;
    it = h->graphs.emplace(key, gr).first;
  }
  LGW_TRY_CUDA(h, cudaGraphLaunch(it->second.exec, st));
  h->launches += it->second.launches;
}

struct Opts {
  int k, precision, reorth, b_sub, qp_max_iter, use_graph, split, split32, qp_mode;
  double tol, qp_tol;
};

Opts resolve_opts(lgw_handle *h, const lgw_options *o, const SysDev &s) {
  if (!o) {
    set_err(h, LGW_ERR_ARG, "options pointer is NULL");
    throw Fail{LGW_ERR_ARG};
  }
  Opts r;
  r.k = o->k;
  r.precision = o->precision;
  r.reorth = o->reorth;
  r.b_sub = o->b_sub;
  r.qp_max_iter = o->qp_max_iter > 0 ? o->qp_max_iter : 50;
  r.use_graph = o->use_graph;
  r.qp_mode = o->qp_mode;
  if (r.qp_mode != 0 && r.qp_mode != 1) {
    set_err(h, LGW_ERR_ARG, "unknown qp_mode %d", o->qp_mode);
    throw Fail{LGW_ERR_ARG};
  }
  if (o->reorth_arith < LGW_RA_AUTO || o->reorth_arith > LGW_RA_SPLIT32) {
    set_err(h, LGW_ERR_ARG, "unknown reorthogonalisation arithmetic %d", o->reorth_arith);
    throw Fail{LGW_ERR_ARG};
  }
  r.split = o->reorth_arith == LGW_RA_SPLIT || o->reorth_arith == LGW_RA_SPLIT32 ||
            (o->reorth_arith == LGW_RA_AUTO && o->precision != LGW_FP64);
  r.split32 = o->reorth_arith == LGW_RA_SPLIT32;
  r.tol = o->breakdown_tol > 0 ? o->breakdown_tol : 1e-13;
  r.qp_tol = o->qp_tol > 0 ? o->qp_tol : 1e-10;
  if (r.k < 1 || r.k > s.n_vc) {
    set_err(h, LGW_ERR_ARG, "k = %d outside [1, n_vc = %d]", r.k, s.n_vc);
    throw Fail{LGW_ERR_ARG};
  }
  if (r.k > 4095) {
    set_err(h, LGW_ERR_UNSUPPORTED, "k = %d above the 4095-step limit of this build", r.k);
    throw Fail{LGW_ERR_UNSUPPORTED};
  }
  if (r.precision != LGW_FP64 && r.precision != LGW_BF16 && r.precision != LGW_FP8 &&
      r.precision != LGW_FP8_DEQ) {
    set_err(h, LGW_ERR_ARG, "unknown precision %d", r.precision);
    throw Fail{LGW_ERR_ARG};
  }
  if (r.reorth < LGW_REORTH_NONE || r.reorth > LGW_REORTH_DCGS) {
    set_err(h, LGW_ERR_ARG, "unknown reorthogonalisation mode %d", r.reorth);
    throw Fail{LGW_ERR_ARG};
  }
  if (r.b_sub < 0) {
    set_err(h, LGW_ERR_ARG, "b_sub < 0");
    throw Fail{LGW_ERR_ARG};
  }
  if (r.precision != LGW_FP64 && !tc_available()) {
    set_err(h, LGW_ERR_UNSUPPORTED, "tensor-core paths need an sm_103 device");
    throw Fail{LGW_ERR_UNSUPPORTED};
  }
  return r;
}

// E4M3 copies of L from src [nr][nc] (row stride ld) into s.
void make_fp8(lgw_handle *h, SysDev &s, const double *src, int ld, int nr, int nc) {
  const size_t n = (size_t)s.N * s.A;
  uint8_t *a = static_cast<uint8_t *>(sys_alloc(h, n));
  uint8_t *b = a ? static_cast<uint8_t *>(sys_alloc(h, n)) : nullptr;
  float *sc = b ? static_cast<float *>(sys_alloc(h, sizeof(float) * s.A)) : nullptr;
  if (!sc) {
    sys_free(h, a);
    sys_free(h, b);
    set_err(h, LGW_ERR_OOM, "device allocation for the E4M3 copies of L failed");
    throw Fail{LGW_ERR_OOM};
  }
  unsigned *colmax = wsT<unsigned>(h, "fp8_colmax", (size_t)s.A);
  launch_prepare_fp8(src, ld, nr, nc, s, colmax, a, b, sc, h->stream);
  check_launch(h, "prepare_fp8");
  s.L8 = a;
  s.L8t = b;
  s.sL = sc;
}

// Digits of L for the FP64 products (32 bytes per element of L), made on the
// first FP64 request, of L evened out along each contraction.  They may take a
// third of the free memory at most, and are given back when a workspace
// allocation fails (drop_digits); without them the products run on the CUDA
// cores, and the next request asks again.  None on a handle with a byte limit.
// One synchronisation, once.
void ensure_digits(lgw_handle *h, lgw_system *sys) {
  if (sys->oz_state != 0 || h->ws_limit) return;   // f64_work takes no buffers there
  SysDev &s = sys->s;
  if (sys->oz_buf) {   // of an attempt that ended in an error
    cudaDeviceSynchronize();
    free_digits(sys);
  }
  if (!s.L64 || !tc_available() || s.A > OZ_ROW_MAX) return;
  const size_t N = (size_t)s.N, A = (size_t)s.A;
  const size_t plane = OzOperand::digits(N, A / 64) * sizeof(uint16_t);
  const size_t rest = (2 * N + A) * sizeof(double) + (2 * (N + A) + 64) * sizeof(int);
  size_t fr = 0, tot = 0;
  LGW_TRY_CUDA(h, cudaMemGetInfo(&fr, &tot));
  if (2 * plane + rest > (fr + h->spare_bytes) / 3) return;
  void *p = sys_alloc(h, 2 * plane + rest);
  if (!p) return;
  sys->oz_buf = p;
  uint16_t *d = static_cast<uint16_t *>(p);
  double *x1 = reinterpret_cast<double *>(static_cast<uint8_t *>(p) + 2 * plane);   // 2^-s_vc
  double *xd = x1 + N, *ys = xd + N;
  int *e = reinterpret_cast<int *>(ys + A), *sx = e + N + A + 1, *sy = sx + N;
  const OzOperand a{d, e, s.N, s.A / 64};
  const OzOperand t{d + plane / sizeof(uint16_t), e + s.N, s.A, s.N / 64};
  unsigned *bad = reinterpret_cast<unsigned *>(e + N + A);
  cudaStream_t st = h->stream;
  LGW_TRY_CUDA(h, cudaMemsetAsync(e, 0, (N + A + 1) * sizeof(int), st));
  // L's scales by pair and by auxiliary function, then its digits on them: over
  // vc, L 2^s_vc meets x Delta^1/2 2^-s_vc, over mu, L 2^t_mu meets y 2^-t_mu
  launch_oz_max_both(s.L64, s.N, s.A, nullptr, nullptr, a.e, t.e, st);
  launch_oz_factors(OzBalance{a.e, s.N, s.dsq, sx, x1, xd},
                    OzBalance{t.e, s.A, nullptr, sy, ys, nullptr}, bad, st);
  launch_oz_max_both(s.L64, s.N, s.A, sy, sx, a.e, t.e, st);
  launch_oz_digits(s.L64, s.N, s.A, false, sy, a, st);
  launch_oz_digits(s.L64, s.N, s.A, true, sx, t, st);
  check_launch(h, "oz_slice(L)");
  h->launches--;   // the system's preparation, not this call's
  unsigned hb = 1;
  LGW_TRY_CUDA(h, cudaMemcpyAsync(&hb, bad, sizeof hb, cudaMemcpyDeviceToHost, st));
  LGW_TRY_CUDA(h, cudaStreamSynchronize(st));
  if (hb != 0) {
    free_digits(sys);
    sys->oz_state = -1;
    return;
  }
  s.ozA = a;
  s.ozT = t;
  s.ozx = xd;
  s.ozy = ys;
  sys->ozx_tda = x1;
  sys->oz_state = 1;
  h->sliced.push_back(sys);
  h->drop_graphs();   // captured without them
}

// The copies of L a request needs must exist; the E4M3 copies are made on
// the first FP8 request for a system that keeps its FP64 copy.
void ensure_copies(lgw_handle *h, const lgw_system *csys, const Opts &o) {
  const SysDev &cs = csys->s;
  if (o.precision == LGW_FP64 && !cs.L64) {
    set_err(h, LGW_ERR_UNSUPPORTED, "the system keeps no FP64 copy of L (LGW_SYS_NO_FP64)");
    throw Fail{LGW_ERR_UNSUPPORTED};
  }
  if (o.precision == LGW_BF16 && !cs.Lb) {
    set_err(h, LGW_ERR_UNSUPPORTED, "the system keeps no BF16 copy of L (LGW_SYS_NO_BF16)");
    throw Fail{LGW_ERR_UNSUPPORTED};
  }
  if (o.precision == LGW_FP64) ensure_digits(h, const_cast<lgw_system *>(csys));
  if ((o.precision != LGW_FP8 && o.precision != LGW_FP8_DEQ) || cs.L8) return;
  if (!cs.L64) {
    set_err(h, LGW_ERR_UNSUPPORTED, "no E4M3 copy of L and no FP64 copy to make it from");
    throw Fail{LGW_ERR_UNSUPPORTED};
  }
  lgw_system *sys = const_cast<lgw_system *>(csys);
  make_fp8(h, sys->s, cs.L64, cs.A, cs.N, cs.A);
}

struct ProbView {
  int n_t, n_m, n_freq, B;
  std::vector<int> targets, m_idx;
  const int *d_targets, *d_m_idx;
  const double *d_M, *d_V, *d_omega, *d_shift;
  double delta;
};

ProbView check_problem(lgw_handle *h, const SysDev &s, const lgw_problem *p) {
  if (!p) {
    set_err(h, LGW_ERR_ARG, "problem pointer is NULL");
    throw Fail{LGW_ERR_ARG};
  }
  ProbView v{};
  v.n_t = p->n_t;
  v.n_m = p->n_m;
  v.n_freq = p->n_freq;
  if (v.n_t < 0 || v.n_m < 0 || v.n_freq < 0 || (v.n_t > 0 && !p->targets) ||
      (v.n_m > 0 && !p->m_idx) || (v.n_freq > 0 && !p->omega)) {
    set_err(h, LGW_ERR_ARG, "negative size or missing targets/m_idx/omega");
    throw Fail{LGW_ERR_ARG};
  }
  if ((p->M == nullptr) == (p->V == nullptr)) {
    set_err(h, LGW_ERR_ARG, "exactly one of M and V must be given");
    throw Fail{LGW_ERR_ARG};
  }
  if (!(p->delta > 0.0)) {
    set_err(h, LGW_ERR_ARG, "delta must be > 0");
    throw Fail{LGW_ERR_ARG};
  }
  v.B = v.n_t * v.n_m;
  v.targets = to_host(h, p->targets, v.n_t);
  v.m_idx = to_host(h, p->m_idx, v.n_m);
  const int norb = s.n_v + s.n_c;
  for (int t : v.targets)
    if (t < 0 || t >= norb) {
      set_err(h, LGW_ERR_SHAPE, "target index %d outside [0, %d)", t, norb);
      throw Fail{LGW_ERR_SHAPE};
    }
  for (int m : v.m_idx)
    if (m < 0 || m >= norb) {
      set_err(h, LGW_ERR_SHAPE, "summed index %d outside [0, %d)", m, norb);
      throw Fail{LGW_ERR_SHAPE};
    }
  v.d_targets = in_dev(h, "in_targets", v.targets.data(), (size_t)v.n_t);
  v.d_m_idx = in_dev(h, "in_midx", v.m_idx.data(), (size_t)v.n_m);
  v.d_omega = in_dev(h, "in_omega", p->omega, (size_t)v.n_freq);
  v.d_shift = p->static_shift ? in_dev(h, "in_shift", p->static_shift, (size_t)v.n_t) : nullptr;
  v.d_M = p->M ? in_dev(h, "in_M", p->M, (size_t)v.B * s.n_aux) : nullptr;
  v.d_V = p->V ? in_dev(h, "in_V", p->V, (size_t)v.B * s.n_vc) : nullptr;
  v.delta = p->delta;
  return v;
}

// ---------------------------------------------------------------------------
// Lanczos over all start vectors, sub-batch by sub-batch.
// alpha/beta [B][k], beta0 [B], k_eff [B] are device arrays.
// ---------------------------------------------------------------------------
// Polynomial operator D = p_g(C) (the paper's form after Eq. 12): the
// Chebyshev interpolant of sqrt at the g+1 points of the first kind on
// [lo, hi], applied by Clenshaw's recurrence in S = a_s C + b_s I.
struct PolyOp {
  int g;
  double lo, hi, as, bs;
  std::vector<double> c;   // c_0 .. c_g
};

PolyOp make_poly(int g, double lo, double hi) {
  PolyOp p;
  p.g = g;
  p.lo = lo;
  p.hi = hi;
  p.as = 2.0 / (hi - lo);
  p.bs = -(hi + lo) / (hi - lo);
  const int n = g + 1;
  const double pi = 3.14159265358979323846;
  std::vector<double> f(n);
  for (int j = 0; j < n; ++j)
    f[j] = std::sqrt(0.5 * (hi + lo) + 0.5 * (hi - lo) * std::cos(pi * (j + 0.5) / n));
  p.c.assign(n, 0.0);
  for (int k = 0; k < n; ++k) {
    double acc = 0.0;
    for (int j = 0; j < n; ++j) acc += f[j] * std::cos(k * pi * (j + 0.5) / n);
    p.c[k] = 2.0 / n * acc;
  }
  p.c[0] *= 0.5;
  return p;
}

// ---------------------------------------------------------------------------
// FP64 contractions: on the tensor cores where the system holds digits of L
// and the operands' digits fit the workspace, else on the CUDA cores.
// ---------------------------------------------------------------------------
constexpr int F64_ROWS = 1024;   // vectors sliced at a time

struct F64Work {
  OzOperand x, y;        // digits of the vectors and of y = L^T (Delta^1/2 x); d NULL: none
  double *part = nullptr;
  size_t part_n = 0;     // doubles that `part` holds
};

// own: prefix of the buffers' names.  A recurrence takes its buffers once, so
// work of another width that runs between its sub-batches has names of its own
// (ws frees a buffer that has to grow).
F64Work f64_work(lgw_handle *h, const SysDev &s, int rows, const std::string &own = "") {
  F64Work f;
  // a contraction of one split writes its result, not partials
  const int splits = gemm1_f64_splits(s, rows);
  const size_t part = splits > 1 ? (size_t)splits * rows * s.A : 0;
  if (s.ozA.d) {
    const int r = std::min(rows, F64_ROWS);
    const size_t nx = OzOperand::digits(r, s.N / 64), ny = OzOperand::digits(r, s.A / 64);
    uint16_t *d = static_cast<uint16_t *>(ws(h, own + "oz_xy", (nx + ny) * sizeof(uint16_t), true));
    int *e = d ? static_cast<int *>(ws(h, own + "oz_e", 2 * (size_t)r * sizeof(int), true)) : nullptr;
    const size_t op = std::max(part, oz_part_rows(s.A, rows, F64_ROWS, s.N / 64) * s.A);
    double *pp = e ? static_cast<double *>(ws(h, own + "yp64", op * sizeof(double), true)) : nullptr;
    if (pp) {
      f.x = OzOperand{d, e, r, s.N / 64};
      f.y = OzOperand{d + nx, e + r, r, s.A / 64};
      f.x.scale = s.ozx;
      f.y.scale = s.ozy;
      f.part = pp;
      f.part_n = op;
      return f;
    }
  }
  if (part > 0) f.part = wsT<double>(h, own + "yp64", part);
  f.part_n = part;
  return f;
}

// No contraction writes more split partials than its work holds.
void check_part(lgw_handle *h, const F64Work &f, int splits, int rows, int A) {
  if ((size_t)splits * rows * A <= f.part_n) return;
  set_err(h, LGW_ERR_SHAPE, "%d splits of %d x %d partials exceed the %zu that were planned",
          splits, rows, A, f.part_n);
  throw Fail{LGW_ERR_SHAPE};
}

void oz_gemm(lgw_handle *h, const OzOperand &A, const OzOperand &B, int M, int Ncols, int splits,
             const OzOut &o, const char *what) {
  if (!launch_oz_gemm(A, B, M, Ncols, splits, o, h->d_status, h->stream)) {
    set_err(h, LGW_ERR_CUDA, "tensor map of %s failed", what);
    throw Fail{LGW_ERR_CUDA};
  }
  check_launch(h, what);
}

// Digits of the next step's vectors, for a producer of all of them at once.
OzOperand f64_next_digits(const SysDev &s, const F64Work &f, int Bs) {
  OzOperand x = f.x;
  if (!s.ozT.d || Bs > F64_ROWS) return OzOperand{};
  x.rows = Bs;
  return x;
}

// Y [rows][A] = (Delta^1/2 q) L; with digits, those of Y too (of the last
// F64_ROWS rows) for f64_contract2.  ready: the digits of Delta^1/2 q are in
// place (f64_next_digits).
void f64_contract1(lgw_handle *h, const SysDev &s, const F64Work &f, const double *q, int rows,
                   double *Y, bool ready = false) {
  cudaStream_t st = h->stream;
  if (!f.x.d || !s.ozT.d) {
    const int splits = gemm1_f64_splits(s, rows);
    if (splits > 1) check_part(h, f, splits, rows, s.A);
    launch_gemm1_f64(s, q, rows, splits > 1 ? f.part : Y, splits, st);
    check_launch(h, "gemm1_f64");
    if (splits == 1) return;
    launch_reduce_y_f64(f.part, splits, rows, s.A, Y, st);
    check_launch(h, "reduce_y_f64");
    return;
  }
  for (int r0 = 0; r0 < rows; r0 += F64_ROWS) {
    const int nr = std::min(F64_ROWS, rows - r0);
    OzOperand x = f.x, y = f.y;
    x.rows = y.rows = nr;
    if (!ready) {
      launch_oz_slice(q + (size_t)r0 * s.N, (size_t)s.N, nr, s.N, x.scale, false, x, st);
      check_launch(h, "oz_slice(x)");
    }
    const int splits = oz_splits(s.A, nr, s.N / 64);
    check_part(h, f, splits, nr, s.A);
    OzOut o;
    o.mode = OZ_PART;
    o.out = f.part;
    o.ldo = s.A;
    oz_gemm(h, s.ozT, x, s.A, nr, splits, o, "oz_gemm1");
    launch_oz_reduce(f.part, splits, nr, s.A, Y + (size_t)r0 * s.A, y, st);
    check_launch(h, "oz_reduce(y)");
  }
}

// The FP64 GEMM2 and its epilogue; fresh: Y comes straight from f64_contract1
// (its digits are in place).
void f64_contract2(lgw_handle *h, const SysDev &s, const F64Work &f, const double *Y, bool fresh,
                   int Bs, int epi, const double *q, const double *qprev, const double *betaj,
                   double *w, double *alpha_part) {
  cudaStream_t st = h->stream;
  if (!f.y.d || !s.ozA.d || Bs > F64_ROWS) {
    launch_gemm2_f64(s, Y, Bs, epi, q, qprev, betaj, w, alpha_part, st);
    check_launch(h, "gemm2_f64");
    return;
  }
  OzOperand y = f.y;
  y.rows = Bs;
  if (!fresh) {
    launch_oz_reduce(Y, 1, Bs, s.A, nullptr, y, st);
    check_launch(h, "oz_slice(y)");
  }
  OzOut o;
  o.mode = epi;
  o.out = w;
  o.ldo = s.N;
  o.Delta2 = s.Delta2;
  o.dsq = s.dsq;
  o.cd = s.cd;
  o.q = q;
  o.qprev = qprev;
  o.betaj = betaj;
  o.alpha_part = epi == EPI_START ? nullptr : alpha_part;
  oz_gemm(h, s.ozA, y, s.N, Bs, 1, o, "oz_gemm2");
}

// S [Ni][Nmu] += scale * X^T Y over R rows (X row stride ldx, Y row stride
// ldy), 1024 rows at a time on the tensor cores.  Rows need no balance here: of
// the pairs (X, Y) one holds unit vectors, bounded polynomials of C on them or
// images of those under L, or (Y, M) both scale with the vector's weight, so a
// row that is small in one factor is small in the sum.
void f64_atb(lgw_handle *h, const double *X, int ldx, const double *Y, int ldy, int R, int Ni,
             int Nmu, double *S, double scale = 1.0) {
  cudaStream_t st = h->stream;
  constexpr int RC = 1024;
  const int ra = std::max(128, round_up(Nmu, 16)), rb = std::max(64, round_up(Ni, 16));
  const int kb = (std::min(R, RC) + 63) / 64;
  const size_t na = OzOperand::digits(ra, kb), nb = OzOperand::digits(rb, kb);
  uint16_t *d = nullptr;
  int *e = nullptr;
  if (tc_available()) {
    d = static_cast<uint16_t *>(ws(h, "oz_atb", (na + nb) * sizeof(uint16_t), true));
    if (d) e = static_cast<int *>(ws(h, "oz_atb_e", (size_t)(ra + rb) * sizeof(int), true));
  }
  if (!e) {
    launch_atb_f64(X, ldx, Y, ldy, R, Ni, Nmu, S, st, scale);
    check_launch(h, "atb_f64");
    return;
  }
  for (int r0 = 0; r0 < R; r0 += RC) {
    const int nr = std::min(RC, R - r0), nkb = (nr + 63) / 64;
    const OzOperand a{d, e, ra, nkb}, b{d + na, e + ra, rb, nkb};
    launch_oz_slice(Y + (size_t)r0 * ldy, (size_t)ldy, nr, Nmu, nullptr, true, a, st);
    launch_oz_slice(X + (size_t)r0 * ldx, (size_t)ldx, nr, Ni, nullptr, true, b, st);
    check_launch(h, "oz_slice(atb)");
    OzOut o;
    o.mode = OZ_ADD;
    o.out = S;
    o.ldo = Nmu;
    o.scale = scale;
    oz_gemm(h, a, b, Nmu, Ni, 1, o, "oz_gemm(atb)");
  }
}

// B [n_pairs][n] = C [n_pairs][n] R [n][n], R lower triangular, 8192 pairs at a
// time on the tensor cores.
//
// The metric and C come in any normalisation of the auxiliary functions, one
// the inverse of the other, and every product counts.  Digits are relative to a
// row's largest element, so a function's scale in C, its largest |C_pk| over the
// pairs, is moved to row k of R first (an exact power of two): C's rows are then
// as even as they can be, and a column of R shows what its terms are worth.
// (Even rows of R would not do: column i starts in row i, and a large function
// before it would set the grid of C's rows.)  Tiles for which that is not enough
// find it out from the K blocks' exponents and use the FP64 pipe.
struct FitWork {
  OzOperand a, b;        // digits of R's columns and of C's rows; a.d NULL: none
  int *col = nullptr;    // largest exponent fields of C's columns
};
// The scales cost a pass over C, the shifts 10 us per 8192 rows of 1024, the
// tiles' look at the exponents hides behind their products.  For small C the
// pass runs beside the first diagonal block, else beside the factorisation with
// the digits of the first 8192 pairs, which takes as much off: 3.38 ms per call
// at 16384 pairs, n 1024, 3.37 to 3.40 without any of it; 1.48 against 1.50 at
// 6000 x 600, 338 us against 333 at 700 x 130, 129 against 123 at 512 x 64.  (All
// 16384 pairs' digits made beside the factorisation: 3.47 ms, the chain's blocks
// wait for a place.)
constexpr int FIT_PAIRS = 8192;

FitWork fit_work(lgw_handle *h, int n_pairs, int n) {
  FitWork f;
  const size_t nkb = (n + 63) / 64, ra = std::max(128, round_up(n, 16));
  const size_t rb = std::max(64, round_up(std::min(n_pairs, FIT_PAIRS), 16));
  const size_t na = OzOperand::digits(ra, nkb), nb = OzOperand::digits(rb, nkb);
  if (!tc_available() || n > OZ_ROW_MAX) return f;
  uint16_t *d = static_cast<uint16_t *>(ws(h, "oz_fit", (na + nb) * sizeof(uint16_t), true));
  const size_t nc = round_up(n, 64);
  int *e = d ? static_cast<int *>(ws(h, "oz_fit_e", (nc + ra + rb) * sizeof(int) +
                                                       (ra + rb) * nkb * sizeof(short), true))
             : nullptr;
  if (!e) return f;
  f.col = e;
  int *ea = f.col + nc, *eb = ea + ra;
  short *blk = reinterpret_cast<short *>(eb + rb);
  f.a = OzOperand{d, ea, (int)ra, (int)nkb, blk};
  f.b = OzOperand{d + na, eb, (int)rb, (int)nkb, blk + ra * nkb};
  return f;
}

void fit_slice(lgw_handle *h, const FitWork &f, const double *C, int n_pairs, int n, int p0,
               cudaStream_t st) {
  launch_oz_slice(C + (size_t)p0 * n, (size_t)n, std::min(FIT_PAIRS, n_pairs - p0), n, nullptr,
                  false, f.b, st, f.col);
  check_launch(h, "oz_slice(C)");
}

// What needs C alone: the scales and the first pairs' digits.
void fit_begin(lgw_handle *h, const FitWork &f, const double *C, int n_pairs, int n,
               cudaStream_t st) {
  launch_oz_col_max(C, (size_t)n, n_pairs, n, f.col, st);
  check_launch(h, "oz_col_max");
  fit_slice(h, f, C, n_pairs, n, 0, st);
}

void f64_fit(lgw_handle *h, const FitWork &f, const double *C, const double *R, int n_pairs,
             int n, double *B) {
  cudaStream_t st = h->stream;
  if (!f.a.d) {
    launch_gemm_nn_f64(C, R, n_pairs, n, n, B, st);
    check_launch(h, "gemm_nn_f64");
    return;
  }
  launch_oz_slice(R, (size_t)n, n, n, nullptr, true, f.a, st, nullptr, f.col);
  check_launch(h, "oz_slice(R)");
  for (int p0 = 0; p0 < n_pairs; p0 += FIT_PAIRS) {
    const int np = std::min(FIT_PAIRS, n_pairs - p0);
    if (p0 > 0) fit_slice(h, f, C, n_pairs, n, p0, st);
    OzOut o;
    o.mode = OZ_PART;
    o.out = B + (size_t)p0 * n;
    o.ldo = n;
    o.lower = true;   // column i of R starts in row i
    o.xa = R;
    o.xb = C + (size_t)p0 * n;
    o.ldxa = o.ldxb = o.K = n;
    oz_gemm(h, f.a, f.b, n, np, 1, o, "oz_gemm(fit)");
  }
}

// keep_basis stores all k + 1 FP64 basis vectors of a sub-batch (slot j of
// sub-batch row b at basis + (j * Bs + b) * N) whatever the reorthogonalisation
// mode; after_sub, if given, runs once each sub-batch's recurrence is done.
using SubBatchHook = std::function<void(const VecCtx &)>;
// after_step, if given, runs after the start (j = -1) and after each step j
// that ends with the plain normalisation (FP64 basis or ring; not the split
// basis), once q_{j+1} is in its slot.
using StepHook = std::function<void(const VecCtx &, int)>;

void run_lanczos(lgw_handle *h, const SysDev &s, const ProbView &pv, const Opts &o, double *alpha,
                 double *beta, double *beta0, int *k_eff, lgw_report *rep, double *tacc,
                 bool keep_basis = false, const SubBatchHook *after_sub = nullptr,
                 const PolyOp *poly = nullptr, const StepHook *after_step = nullptr) {
  // a reference: a graph capture redirects the launches to the capture stream
  cudaStream_t &st = h->stream;
  const int B = pv.B;
  const int k = o.k;
  if (B == 0) return;
  LGW_TRY_CUDA(h, cudaMemsetAsync(alpha, 0, sizeof(double) * B * k, st));
  LGW_TRY_CUDA(h, cudaMemsetAsync(beta, 0, sizeof(double) * B * k, st));
  const bool tc = o.precision != LGW_FP64;
  const bool fp8 = o.precision == LGW_FP8;
  const bool deq = o.precision == LGW_FP8_DEQ;
  int nsub_req = o.b_sub > 0 ? o.b_sub : std::min(B, 512);
  nsub_req = std::min(nsub_req, B);
  int Bs = round_up(nsub_req, PAD_VEC);
  if (tc) Bs = std::max(Bs, 64);
  const int N = s.N;
  const int nchunks = (N + VEC_CHUNK - 1) / VEC_CHUNK;
  const int kmax1 = k + 1;
  const bool reorth = o.reorth != LGW_REORTH_NONE;
  const bool split = reorth && o.split;
  // the delayed single-sweep Gram-Schmidt runs on the split basis; with the
  // FP64 basis the same request runs as CGS1K
  const bool dcgs = split && o.reorth == LGW_REORTH_DCGS;
  const bool full_basis = !split && (reorth || keep_basis);
  const int nslots = full_basis ? k + 1 : 3;

  VecCtx c{};
  c.N = N;
  c.Bs = Bs;
  c.nchunks = nchunks;
  c.k = k;
  c.kmax1 = kmax1;
  c.reorth = (o.reorth == LGW_REORTH_DCGS && !dcgs) ? (int)LGW_REORTH_CGS1K : o.reorth;
  c.ring = full_basis ? 0 : 1;
  c.nslots = nslots;
  c.tol = o.tol;
  c.Delta2 = s.Delta2;
  c.dsq = s.dsq;
  c.cd = s.cd;
  c.w = wsT<double>(h, "w", (size_t)Bs * N);
  c.basis = wsT<double>(h, split ? "ring" : "basis", (size_t)nslots * Bs * N);
  if (split) {
    c.bhi = wsT<float>(h, "basis_hi", (size_t)(k + 1) * Bs * N);
    c.blo = o.split32 ? nullptr : wsT<float>(h, "basis_lo", (size_t)(k + 1) * Bs * N);
  }
  c.dsqf = s.dsqf;
  c.d2lo = s.d2lo;
  // tensor cores without reorthogonalisation (the three-vector ring): the
  // slots and w as float pairs, the vector passes in double-float arithmetic
  c.pair = (tc && !reorth && !full_basis && poly == nullptr && s.d2lo != nullptr) ? 1 : 0;
  c.nalpha_f = c.pair ? wsT<float2>(h, "nalpha_f", (size_t)Bs) : nullptr;
  c.nbeta_f = c.pair ? wsT<float2>(h, "nbeta_f", (size_t)Bs) : nullptr;
  // float [Bs][N]: the split-basis epilogue output (c_K Delta^1/2 U) and, at
  // the start of each sub-batch, the tensor-core coupling vectors V = L M
  float *ucd_buf = tc ? wsT<float>(h, "ucd", (size_t)Bs * N) : nullptr;
  c.ucd = split ? ucd_buf : nullptr;
  c.ucd_pair = c.pair ? ucd_buf : nullptr;
  c.qscale = c.pair ? wsT<float2>(h, "qscale", (size_t)3 * Bs) : nullptr;
  c.xmax = c.pair ? wsT<unsigned>(h, "xmax", (size_t)Bs) : nullptr;
  c.d2f = s.d2f;
  c.kf = s.kf;
  c.n_yb = (s.A + 255) / 256;
  float *yy = (split && tc) ? wsT<float>(h, "yy_part", (size_t)Bs * c.n_yb) : nullptr;
  c.yy_part = yy;
  // the delayed sweep reads step j's partials and writes step j + 1's in
  // the same launch: two halves by step parity (the start writes half 0)
  c.dq2_part = (split && tc) ? wsT<float>(h, "dq2_part", (size_t)(dcgs ? 2 : 1) * Bs * nchunks)
                             : nullptr;
  c.xh = tc ? wsT<__nv_bfloat16>(h, "xh", (size_t)Bs * N) : nullptr;
  // alpha partials: per 2048-element chunk (tensor cores without
  // reorthogonalisation), per GEMM2 tile otherwise
  const bool tc_plain = tc && !reorth;
  c.n_mt = (tc_plain || poly) ? nchunks : (tc ? tc_n_mt(s) : N / F64_TILE);
  // chunks per block of the assembly, axpy and normalisation passes on the
  // tensor-core path without reorthogonalisation; 1 unless LGW_VEC_CPB (1 to
  // 64) asks otherwise (2, 4 and 8 measured within 3% of 1, bit-identical)
  c.cpb = 1;
  if (tc_plain) {
    if (const char *env = std::getenv("LGW_VEC_CPB"))
      c.cpb = std::max(1, std::min(64, std::atoi(env)));
  }
  c.alpha_part = wsT<double>(h, "alpha_part", (size_t)c.n_mt * Bs);
  c.dot_part = reorth ? wsT<double>(h, "dot_part", (size_t)Bs * nchunks * kmax1) : nullptr;
  c.h = reorth ? wsT<double>(h, "hcoef", (size_t)Bs * kmax1) : nullptr;
  c.norm_a = wsT<double>(h, "norm_a", (size_t)Bs * nchunks);
  c.norm_b = wsT<double>(h, "norm_b", (size_t)Bs * nchunks);
  c.norm_c = wsT<double>(h, "norm_c", (size_t)Bs * nchunks);
  c.flag2 = wsT<int>(h, "flag2", (size_t)Bs);
  c.amax = wsT<double>(h, "amax", (size_t)Bs);
  c.betaj = wsT<double>(h, "betaj", (size_t)Bs);
  c.sinv = wsT<double>(h, "sinv", (size_t)Bs);
  c.alpha = alpha;
  c.beta = beta;
  c.beta0 = beta0;
  c.k_eff = k_eff;
  c.n_second = wsT<int>(h, "n_second", 1);
  c.status = h->d_status;
  if (dcgs) {
    // the carried vector lives in ring slot 0 (where the start writes q_0);
    // FP64 contractions leave C w in the w buffer
    c.wv = slot_ptr(c, 0);
    c.uC = tc ? nullptr : c.w;
    c.hj_part = wsT<double>(h, "hj_part", (size_t)Bs * nchunks);
    c.gq = wsT<double>(h, "gq", (size_t)Bs * kmax1);
    c.p2_step = wsT<int>(h, "p2_step", (size_t)k);
  }
  LGW_TRY_CUDA(h, cudaMemsetAsync(c.n_second, 0, sizeof(int), st));
  LGW_TRY_CUDA(h, cudaMemsetAsync(c.flag2, 0, sizeof(int) * Bs, st));

  // contraction buffers
  double *Y64 = wsT<double>(h, "y64", (size_t)Bs * s.A);
  F64Work f64;
  if (!tc) f64 = f64_work(h, s, Bs);
  TcPlan *plan = nullptr;
  uint8_t *x8 = nullptr, *y8 = nullptr;
  uint16_t *x16 = nullptr, *y16 = nullptr;
  float *sx = nullptr, *ty = nullptr;
  float *Yp32 = nullptr;
  __nv_bfloat16 *Yh = nullptr;
  int splits_tc = 1;
  if (tc) {
    // the split count only depends on shapes; size the partials generously
    Yp32 = wsT<float>(h, "yp32", (size_t)64 * Bs * s.A);
    Yh = wsT<__nv_bfloat16>(h, "yh", (size_t)Bs * s.A);
    char err[256];
    plan = tc_plan_create(s, Bs, c.xh, Yp32, Yh, &splits_tc, err, sizeof err);
    if (!plan) {
      set_err(h, LGW_ERR_CUDA, "%s", err);
      throw Fail{LGW_ERR_CUDA};
    }
    if (!fp8 && !deq && !tc_plan_has_bf16(plan)) {
      tc_plan_destroy(plan);
      set_err(h, LGW_ERR_UNSUPPORTED, "BF16 contractions need the BF16 copies of L");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    if (deq) {
      x16 = wsT<uint16_t>(h, "x16", (size_t)Bs * N);
      y16 = wsT<uint16_t>(h, "y16", (size_t)Bs * s.A);
      sx = wsT<float>(h, "sx", (size_t)Bs);
      ty = wsT<float>(h, "ty", (size_t)Bs);
      if (!tc_plan_enable_deq(plan, s.L8t, s.L8, x16, y16, ty)) {
        tc_plan_destroy(plan);
        set_err(h, LGW_ERR_CUDA, "cuTensorMapEncodeTiled failed for the widened E4M3 operands");
        throw Fail{LGW_ERR_CUDA};
      }
    }
    if (fp8) {
      x8 = wsT<uint8_t>(h, "x8", (size_t)Bs * N);
      y8 = wsT<uint8_t>(h, "y8", (size_t)Bs * s.A);
      sx = wsT<float>(h, "sx", (size_t)Bs);
      ty = wsT<float>(h, "ty", (size_t)Bs);
      if (!tc_plan_enable_fp8(plan, s.L8t, s.L8, x8, y8, ty)) {
        tc_plan_destroy(plan);
        set_err(h, LGW_ERR_CUDA, "cuTensorMapEncodeTiled failed for the E4M3 operands");
        throw Fail{LGW_ERR_CUDA};
      }
    }
    if (!tc_plan_autotune(plan, ucd_buf, h->d_status, st, &splits_tc)) {
      tc_plan_destroy(plan);
      set_err(h, LGW_ERR_CUDA, "tensor-core tile autotuning failed");
      throw Fail{LGW_ERR_CUDA};
    }
  }
  struct PlanGuard {
    TcPlan *p;
    ~PlanGuard() {
      if (p) tc_plan_destroy(p);
    }
  } guard{plan};

  // use_graph: each sub-batch's launch sequence (start vectors and the k
  // steps) is captured once and replayed from the handle's graph cache
  const bool graph_mode = o.use_graph && after_sub == nullptr;
  const bool timing_saved = h->timing;
  if (graph_mode) h->timing = false;
  struct TimingRestore {
    lgw_handle *h;
    bool v;
    ~TimingRestore() { h->timing = v; }
  } timing_restore{h, timing_saved};
  // Clenshaw buffers of the polynomial operator
  double *pb[3] = {nullptr, nullptr, nullptr};
  double *pT = nullptr;
  if (poly) {
    for (int i = 0; i < 3; ++i)
      pb[i] = wsT<double>(h, "poly_b" + std::to_string(i), (size_t)Bs * N);
    if (!tc) pT = wsT<double>(h, "poly_t", (size_t)Bs * N);
  }
  // C b for the polynomial operator: FP64 product into pT, or the tensor
  // cores from c.xh = bf16(Delta^1/2 b) into ucd_buf
  auto apply_c = [&](const double *bsrc) {
    if (tc) {
      if (fp8) {
        launch_quant_x8(c.xh, Bs, N, x8, sx, st);
        check_launch(h, "quant_x8");
      } else if (deq) {
        launch_quant_x16(c.xh, Bs, N, x16, sx, st);
        check_launch(h, "quant_x16");
      }
      launch_gemm1_tc(plan, h->d_status, st);
      check_launch(h, "gemm1_tc");
      if (fp8)
        launch_reduce_y_fp8(Yp32, splits_tc, Bs, s.A, sx, s.sL, y8, ty, nullptr, 1, st);
      else if (deq)
        launch_reduce_y_f16(Yp32, splits_tc, Bs, s.A, sx, s.sL, y16, ty, nullptr, 1, st);
      else
        launch_reduce_y_bf16(Yp32, splits_tc, Bs, s.A, Yh, nullptr, st);
      check_launch(h, "reduce_y");
      launch_gemm2_tc_split(plan, ucd_buf, h->d_status, st);
      check_launch(h, "gemm2_tc");
    } else {
      f64_contract1(h, s, f64, bsrc, Bs, Y64);
      f64_contract2(h, s, f64, Y64, true, Bs, EPI_APPLY, bsrc, nullptr, nullptr, pT, nullptr);
    }
  };
  Timer tm(h);
  int nsub = 0;
  for (int vec0 = 0; vec0 < B; vec0 += nsub_req, ++nsub) {
    const int nvec = std::min(nsub_req, B - vec0);
    c.vec0 = vec0;
    c.nvec = nvec;
    auto sub_body = [&]() {
      // ---- start vectors b = Delta^1/2 V, V = L M (text after Eq. 8) ----
      tm.mark(C_START);
      if (dcgs) LGW_TRY_CUDA(h, cudaMemsetAsync(c.p2_step, 0, sizeof(int) * k, st));
      if (pv.d_M && tc && s.Lb) {
        // V = L M on the tensor cores in split BF16 (three products, FP32 sum)
        float *vf = ucd_buf;
        if (!launch_coupling_tc(plan, s, pv.d_M + (size_t)vec0 * s.n_aux, nvec, vf, h->d_status,
                                st)) {
          set_err(h, LGW_ERR_UNSUPPORTED, "tensor-core plan without the BF16 copies of L");
          throw Fail{LGW_ERR_UNSUPPORTED};
        }
        check_launch(h, "coupling_tc");
        launch_start_from_vf(c, vf, st);
        check_launch(h, "start_from_vf");
      } else if (pv.d_M) {
        if (!s.L64) {
          set_err(h, LGW_ERR_UNSUPPORTED, "start vectors from M need the BF16 or FP64 copy of L");
          throw Fail{LGW_ERR_UNSUPPORTED};
        }
        LGW_TRY_CUDA(h, cudaMemsetAsync(Y64, 0, sizeof(double) * Bs * s.A, st));
        LGW_TRY_CUDA(h, cudaMemcpy2DAsync(Y64, sizeof(double) * s.A, pv.d_M + (size_t)vec0 * s.n_aux,
                                          sizeof(double) * s.n_aux, sizeof(double) * s.n_aux, nvec,
                                          cudaMemcpyDeviceToDevice, st));
        f64_contract2(h, s, f64, Y64, false, Bs, EPI_START, nullptr, nullptr, nullptr, c.w,
                      nullptr);
        // padding rows of w (b >= nvec) hold L*0 = 0 already
        launch_norm_partials(c, c.w, c.norm_a, st);
        check_launch(h, "norm_partials");
      } else {
        launch_start_from_v(c, pv.d_V + (size_t)vec0 * s.n_vc, s.n_vc, s.n_vc, st);
        check_launch(h, "start_from_v");
      }
      if (c.pair) LGW_TRY_CUDA(h, cudaMemsetAsync(c.xmax, 0, sizeof(unsigned) * Bs, st));
      if (split)
        launch_start_split(c, st);
      else
        launch_normalize(c, 0, 1, nullptr, st);
      check_launch(h, "normalize(start)");
      if (after_step) (*after_step)(c, -1);
      bool x_ready = false;   // the digits of Delta^1/2 q_j are in place

      for (int j = 0; j < k; ++j) {
        const double *qj = slot_ptr(c, j);
        const double *qp = j > 0 ? slot_ptr(c, j - 1) : nullptr;
        // ---- C q_j through the two contractions (Eq. 4) ----
        tm.mark(C_GEMM1);
        if (poly) {
          // D q_j = p_g(C) q_j by Clenshaw; w = D q_j - beta_j q_{j-1}
          PolyStep ps{};
          ps.N = N;
          ps.q = qj;
          ps.Delta2 = s.Delta2;
          ps.dsqf = s.dsqf;
          ps.as = poly->as;
          ps.bs = poly->bs;
          ps.xh = tc ? c.xh : nullptr;
          ps.ck = poly->c[poly->g];
          ps.out = pb[0];
          tm.mark(C_UPDATE);
          launch_cheb_step(ps, nchunks, Bs, st);
          check_launch(h, "cheb_step");
          int i1 = 0, i2 = -1;
          for (int kk = poly->g - 1; kk >= 0; --kk) {
            tm.mark(C_GEMM1);
            apply_c(pb[i1]);
            tm.mark(C_UPDATE);
            ps.b1 = pb[i1];
            ps.b2 = i2 >= 0 ? pb[i2] : nullptr;
            ps.T = tc ? nullptr : pT;
            ps.ucd = tc ? ucd_buf : nullptr;
            ps.ck = poly->c[kk];
            if (kk > 0) {
              const int io = (i1 + 1) % 3;
              ps.out = pb[io];
              launch_cheb_step(ps, nchunks, Bs, st);
              check_launch(h, "cheb_step");
              i2 = i1;
              i1 = io;
            } else {
              ps.out = nullptr;
              ps.xh = nullptr;
              launch_cheb_final(ps, qp, c.betaj, c.w, c.alpha_part, nchunks, Bs, st);
              check_launch(h, "cheb_final");
            }
          }
        } else if (tc) {
          // the delayed Gram-Schmidt contracts the unnormalised carried
          // vector; 1/beta_j is applied to each column of the reduction
          const double *vscale = dcgs ? c.sinv : nullptr;
          if (fp8) {
            if (c.pair)
              launch_quant_x8_max(c.xh, Bs, N, c.xmax, x8, sx, st);
            else
              launch_quant_x8(c.xh, Bs, N, x8, sx, st, vscale);
            check_launch(h, "quant_x8");
          } else if (deq) {
            launch_quant_x16(c.xh, Bs, N, x16, sx, st, vscale);
            check_launch(h, "quant_x16");
          }
          launch_gemm1_tc(plan, h->d_status, st);
          check_launch(h, "gemm1_tc");
          if (fp8)
            launch_reduce_y_fp8(Yp32, splits_tc, Bs, s.A, sx, s.sL, y8, ty, yy, c.n_yb, st);
          else if (deq)
            launch_reduce_y_f16(Yp32, splits_tc, Bs, s.A, sx, s.sL, y16, ty, yy, c.n_yb, st);
          else
            launch_reduce_y_bf16(Yp32, splits_tc, Bs, s.A, Yh, yy, st, vscale);
          check_launch(h, "reduce_y");
          tm.mark(C_GEMM2);
          if (split) {
            launch_gemm2_tc_split(plan, const_cast<float *>(c.ucd), h->d_status, st);
          } else if (tc_plain) {
            // store-only FP32 epilogue; w and the alpha partials in FP64 on
            // the vector pass (an FP64 epilogue would serialise behind the
            // MMAs on the narrow FP64 pipe)
            launch_gemm2_tc_split(plan, ucd_buf, h->d_status, st);
            check_launch(h, "gemm2_tc");
            launch_assemble_w(c, j, ucd_buf, st);
          } else {
            launch_gemm2_tc(plan, EPI_LANCZOS, qj, qp, c.betaj, c.w, c.alpha_part, h->d_status,
                            st);
          }
          check_launch(h, tc_plain ? "assemble_w" : "gemm2_tc");
        } else if (dcgs) {
          // C w_{j-1} in FP64 with the partials of w . C w (alpha~ after
          // scaling by 1/beta_j^2)
          f64_contract1(h, s, f64, c.wv, Bs, Y64);
          tm.mark(C_GEMM2);
          f64_contract2(h, s, f64, Y64, true, Bs, EPI_APPLY, c.wv, nullptr, nullptr, c.w,
                        c.alpha_part);
        } else {
          f64_contract1(h, s, f64, qj, Bs, Y64, x_ready);
          tm.mark(C_GEMM2);
          f64_contract2(h, s, f64, Y64, true, Bs, EPI_LANCZOS, qj, qp, c.betaj, c.w,
                        c.alpha_part);
        }
        // ---- recurrence and reorthogonalisation ----
        tm.mark(C_DOTS);
        if (dcgs) {
          // one sweep over the basis: delayed update of q_j, w_j and its
          // projection coefficients; then beta_{j+1}, and the rare second pass
          launch_sweep_dcgs(c, j, st);
          check_launch(h, "sweep_dcgs");
          tm.mark(C_UPDATE);
          launch_reduce_dcgs(c, j, st);
          check_launch(h, "reduce_dcgs");
          tm.mark(C_PASS2);
          launch_pass2_dcgs(c, j, st);
          check_launch(h, "pass2_dcgs");
          continue;
        }
        if (split) {
          launch_dots_split(c, j, 1, st);
          check_launch(h, "dots_split");
          launch_reduce_dots_split(c, j, 1, st);
          check_launch(h, "reduce_dots_split");
          tm.mark(C_UPDATE);
          // q_{j+1} for the vectors that take no second pass, w' for the rest
          launch_update_split(c, j, 1, st);
          check_launch(h, "update_split");
          tm.mark(C_PASS2);
          launch_dots_split(c, j, 2, st);
          check_launch(h, "dots_split2");
          launch_reduce_dots_split(c, j, 2, st);
          check_launch(h, "reduce_dots_split2");
          launch_update_split(c, j, 2, st);
          check_launch(h, "update_split2");
          continue;
        }
        if (!tc) {
          const OzOperand xd = poly || j + 1 == k ? OzOperand{} : f64_next_digits(s, f64, Bs);
          if (launch_step_f64(c, j, xd, st)) {
            check_launch(h, "step_f64");
            x_ready = xd.d != nullptr;
            if (after_step) (*after_step)(c, j);
            continue;
          }
        }
        launch_alpha_reduce(c, j, st);
        check_launch(h, "alpha_reduce");
        launch_alpha_axpy(c, j, st);
        check_launch(h, "alpha_axpy");
        if (reorth) {
          launch_reduce_dots(c, j, 1, st);
          check_launch(h, "reduce_dots");
          tm.mark(C_UPDATE);
          launch_update(c, j, 1, st);
          check_launch(h, "update");
          tm.mark(C_PASS2);
          launch_second_pass_decide_j(c, j, st);
          check_launch(h, "second_pass_decide");
          launch_dots(c, j, 2, st);
          check_launch(h, "dots2");
          launch_reduce_dots(c, j, 2, st);
          check_launch(h, "reduce_dots2");
          launch_update(c, j, 2, st);
          check_launch(h, "update2");
        }
        tm.mark(C_NORM);
        launch_beta_vec(c, j, st);
        check_launch(h, "beta_vec");
        launch_normalize(c, j, 0, nullptr, st);
        check_launch(h, "normalize");
        if (after_step) (*after_step)(c, j);
      }
    };
    if (graph_mode) {
      char key[512];
      snprintf(key, sizeof key,
               "%s s%p B%d n%d v%d k%d p%d r%d sp%d s32%d t%.17g M%p V%p a%p b%p b0%p ke%p g%llu",
               h->ws_prefix.c_str(), (const void *)s.L64, Bs, nvec, vec0, k, o.precision,
               o.reorth, (int)split, o.split32, o.tol, (const void *)pv.d_M,
               (const void *)pv.d_V, (void *)alpha, (void *)beta, (void *)beta0, (void *)k_eff,
               h->ws_gen);
      run_graphed(h, key, sub_body);
    } else {
      sub_body();
    }
    if (after_sub) (*after_sub)(c);
  }
  tm.stop();
  if (rep) {
    tm.collect(tacc, C_N);
    int n2 = 0;
    LGW_TRY_CUDA(h, cudaMemcpy(&n2, c.n_second, sizeof(int), cudaMemcpyDeviceToHost));
    rep->n_second_pass = n2;
    rep->n_sub_batches = nsub;
    rep->b_sub = Bs;
    rep->gemm1_splits = tc ? splits_tc
                           : (f64.x.d ? oz_splits(s.A, Bs, s.N / 64) : gemm1_f64_splits(s, Bs));
  }
}

// Interval [x_lo, x_hi] around the spectrum of C for the polynomial form:
// x_lo = min Delta^2 (a bound: C = Delta^2 + a positive semidefinite term);
// x_hi = the largest Ritz value of k_est Lanczos steps (BF16 tensor-core
// contractions when the system has them, else FP64; CGS2) from a hash start
// vector, plus the last beta, the residual norm of that step.  Synchronous.
void estimate_interval(lgw_handle *h, const SysDev &s, int k_est, double &lo, double &hi) {
  cudaStream_t &st = h->stream;
  Opts o{};
  o.k = std::max(1, std::min(k_est, s.n_vc));
  o.precision = (s.Lb && tc_available()) ? LGW_BF16 : LGW_FP64;
  o.reorth = LGW_REORTH_CGS2;
  o.b_sub = 1;
  o.qp_max_iter = 50;
  o.split = o.precision != LGW_FP64;
  o.tol = 1e-13;
  o.qp_tol = 1e-10;
  const bool timing = h->timing;
  h->timing = false;
  double *vec = wsT<double>(h, "iv_vec", (size_t)s.n_vc);
  launch_interval(nullptr, s.n_vc, s.n_vc, nullptr, nullptr, nullptr, nullptr, vec,
                  0x5EEDull, true, st);
  check_launch(h, "hash_vector");
  ProbView pv{};
  pv.n_t = 1;
  pv.n_m = 1;
  pv.B = 1;
  pv.d_V = vec;
  pv.delta = 1.0;
  double *a = wsT<double>(h, "iv_alpha", (size_t)o.k);
  double *b = wsT<double>(h, "iv_beta", (size_t)o.k);
  double *b0 = wsT<double>(h, "iv_beta0", 1);
  int *ke = wsT<int>(h, "iv_keff", 1);
  run_lanczos(h, s, pv, o, a, b, b0, ke, nullptr, nullptr);
  double *out = wsT<double>(h, "iv_out", 2);
  launch_interval(s.Delta2, s.n_vc, s.N, a, b, ke, out, nullptr, 0, false, st);
  check_launch(h, "interval");
  double hv[2];
  LGW_TRY_CUDA(h, cudaMemcpyAsync(hv, out, sizeof hv, cudaMemcpyDeviceToHost, st));
  LGW_TRY_CUDA(h, cudaStreamSynchronize(st));
  h->timing = timing;
  lo = hv[0];
  hi = hv[1];
  if (!(lo > 0.0) || !(hi > lo)) {
    set_err(h, LGW_ERR_NOT_SPD, "spectral interval estimate [%g, %g] is not positive", lo, hi);
    throw Fail{LGW_ERR_NOT_SPD};
  }
}

// Band Lanczos over the request's targets (band width p = n_t): one
// recurrence per summed orbital g, started from [b_{t,g} over t].  Outputs
// the banded T, R0 and the step counts: Tb [G][k][p+1], R0 [G][p][p],
// keff [G] (device).  FP64 basis, CGS2; FP64 or BF16 contractions.
void run_band(lgw_handle *h, const SysDev &s, const ProbView &pv, const Opts &o, double *Tb,
              double *R0, int *keff, double *tacc) {
  cudaStream_t &st = h->stream;
  const int p = pv.n_t, G = pv.n_m, k = o.k;
  const bool tc = o.precision != LGW_FP64;
  int nsub_req = o.b_sub > 0 ? std::min(o.b_sub, G) : std::min(G, 512);
  int Bs = round_up(nsub_req, PAD_VEC);
  if (tc) Bs = std::max(Bs, 64);
  const int N = s.N;
  const int nchunks = (N + VEC_CHUNK - 1) / VEC_CHUNK;
  const int kmax1 = k + 1;
  LGW_TRY_CUDA(h, cudaMemsetAsync(Tb, 0, sizeof(double) * (size_t)G * k * (p + 1), st));
  LGW_TRY_CUDA(h, cudaMemsetAsync(R0, 0, sizeof(double) * (size_t)G * p * p, st));
  LGW_TRY_CUDA(h, cudaMemsetAsync(keff, 0, sizeof(int) * (size_t)G, st));
  BandCtx bc{};
  VecCtx &c = bc.c;
  c.N = N;
  c.Bs = Bs;
  c.nchunks = nchunks;
  c.k = k;
  c.kmax1 = kmax1;
  c.reorth = LGW_REORTH_CGS2;
  c.ring = 0;
  c.nslots = k;
  c.tol = o.tol;
  c.Delta2 = s.Delta2;
  c.dsq = s.dsq;
  c.cd = s.cd;
  c.dsqf = s.dsqf;
  c.d2f = s.d2f;
  c.kf = s.kf;
  c.w = wsT<double>(h, "w", (size_t)Bs * N);
  c.basis = wsT<double>(h, "basis", (size_t)k * Bs * N);
  c.xh = tc ? wsT<__nv_bfloat16>(h, "xh", (size_t)Bs * N) : nullptr;
  c.dot_part = wsT<double>(h, "dot_part", (size_t)Bs * nchunks * kmax1);
  c.h = wsT<double>(h, "hcoef", (size_t)Bs * kmax1);
  c.norm_a = wsT<double>(h, "norm_a", (size_t)Bs * nchunks);
  c.norm_b = wsT<double>(h, "norm_b", (size_t)Bs * nchunks);
  c.norm_c = wsT<double>(h, "norm_c", (size_t)Bs * nchunks);
  c.status = h->d_status;
  bc.p = p;
  bc.G = G;
  bc.nv = wsT<int>(h, "band_nv", (size_t)Bs);
  bc.act = wsT<int>(h, "band_act", (size_t)Bs);
  bc.newrow = wsT<int>(h, "band_newrow", (size_t)Bs);
  bc.inv = wsT<double>(h, "band_inv", (size_t)Bs);
  bc.scale = wsT<double>(h, "band_scale", (size_t)Bs);
  bc.tmax = wsT<double>(h, "band_tmax", (size_t)Bs);
  bc.hsum = wsT<double>(h, "band_hsum", (size_t)Bs * kmax1);
  bc.Tb = Tb;
  bc.R0 = R0;
  bc.keff = keff;
  bc.xq = tc ? nullptr : wsT<double>(h, "band_xq", (size_t)Bs * N);

  double *Y64 = wsT<double>(h, "y64", (size_t)Bs * s.A);
  F64Work f64;
  if (!tc) f64 = f64_work(h, s, Bs);
  float *ucd_buf = tc ? wsT<float>(h, "ucd", (size_t)Bs * N) : nullptr;
  TcPlan *plan = nullptr;
  float *Yp32 = nullptr;
  __nv_bfloat16 *Yh = nullptr;
  int splits_tc = 1;
  if (tc) {
    Yp32 = wsT<float>(h, "yp32", (size_t)64 * Bs * s.A);
    Yh = wsT<__nv_bfloat16>(h, "yh", (size_t)Bs * s.A);
    char err[256];
    plan = tc_plan_create(s, Bs, c.xh, Yp32, Yh, &splits_tc, err, sizeof err);
    if (!plan) {
      set_err(h, LGW_ERR_CUDA, "%s", err);
      throw Fail{LGW_ERR_CUDA};
    }
    if (!tc_plan_has_bf16(plan)) {
      tc_plan_destroy(plan);
      set_err(h, LGW_ERR_UNSUPPORTED, "BF16 contractions need the BF16 copies of L");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    if (!tc_plan_autotune(plan, ucd_buf, h->d_status, st, &splits_tc)) {
      tc_plan_destroy(plan);
      set_err(h, LGW_ERR_CUDA, "tensor-core tile autotuning failed");
      throw Fail{LGW_ERR_CUDA};
    }
  }
  struct PlanGuard {
    TcPlan *p;
    ~PlanGuard() {
      if (p) tc_plan_destroy(p);
    }
  } guard{plan};
  Timer tm(h);
  for (int vec0 = 0; vec0 < G; vec0 += nsub_req) {
    const int nvec = std::min(nsub_req, G - vec0);
    c.vec0 = vec0;
    c.nvec = nvec;
    launch_band_init(bc, st);
    check_launch(h, "band_init");
    // ---- the start block, one target's vectors at a time (text after Eq. 8) ----
    for (int a = 0; a < p; ++a) {
      tm.mark(C_START);
      const size_t row0 = (size_t)a * G + vec0;
      if (pv.d_M && tc) {
        if (!launch_coupling_tc(plan, s, pv.d_M + row0 * s.n_aux, nvec, ucd_buf, h->d_status, st)) {
          set_err(h, LGW_ERR_UNSUPPORTED, "tensor-core plan without the BF16 copies of L");
          throw Fail{LGW_ERR_UNSUPPORTED};
        }
        check_launch(h, "coupling_tc");
        launch_start_from_vf(c, ucd_buf, st);
        check_launch(h, "start_from_vf");
      } else if (pv.d_M) {
        if (!s.L64) {
          set_err(h, LGW_ERR_UNSUPPORTED, "start vectors from M need the BF16 or FP64 copy of L");
          throw Fail{LGW_ERR_UNSUPPORTED};
        }
        LGW_TRY_CUDA(h, cudaMemsetAsync(Y64, 0, sizeof(double) * Bs * s.A, st));
        LGW_TRY_CUDA(h, cudaMemcpy2DAsync(Y64, sizeof(double) * s.A, pv.d_M + row0 * s.n_aux,
                                          sizeof(double) * s.n_aux, sizeof(double) * s.n_aux,
                                          nvec, cudaMemcpyDeviceToDevice, st));
        f64_contract2(h, s, f64, Y64, false, Bs, EPI_START, nullptr, nullptr, nullptr, c.w,
                      nullptr);
      } else {
        launch_start_from_v(c, pv.d_V + row0 * s.n_vc, s.n_vc, s.n_vc, st);
        check_launch(h, "start_from_v");
      }
      tm.mark(C_DOTS);
      launch_band_activate(bc, 0, a, st);
      h->launches += launch_band_append(bc, 0, a, st);
      check_launch(h, "band_append(start)");
    }
    // ---- k steps: C q_j, projected out of all of the group's vectors ----
    for (int j = 0; j < k; ++j) {
      tm.mark(C_GEMM1);
      launch_band_activate(bc, 1, j, st);
      launch_band_operand(bc, j, st);
      check_launch(h, "band_operand");
      if (tc) {
        launch_gemm1_tc(plan, h->d_status, st);
        check_launch(h, "gemm1_tc");
        launch_reduce_y_bf16(Yp32, splits_tc, Bs, s.A, Yh, nullptr, st);
        check_launch(h, "reduce_y");
        tm.mark(C_GEMM2);
        launch_gemm2_tc_split(plan, ucd_buf, h->d_status, st);
        check_launch(h, "gemm2_tc");
        launch_band_assemble(bc, j, ucd_buf, st);
        check_launch(h, "band_assemble");
      } else {
        f64_contract1(h, s, f64, bc.xq, Bs, Y64);
        tm.mark(C_GEMM2);
        f64_contract2(h, s, f64, Y64, true, Bs, EPI_APPLY, bc.xq, nullptr, nullptr, c.w, nullptr);
      }
      tm.mark(C_DOTS);
      h->launches += launch_band_append(bc, 1, j, st);
      check_launch(h, "band_append");
    }
    launch_band_finish(bc, st);
    check_launch(h, "band_finish");
  }
  tm.stop();
  if (tacc) tm.collect(tacc, C_N);
}

void run_sigma(lgw_handle *h, const SysDev &s, const ProbView &pv, const Opts &o,
               const double *alpha, const double *beta, const double *beta0, const int *k_eff,
               double *sigma, double *e_qp, double *z_qp, lgw_report *rep, double *tacc,
               int cfmode = 0) {
  // cfmode 0: spectral map of C's tridiagonals (Omega-space fractions);
  // 1: D = p_g(C)'s own tridiagonal, (G(zeta) - G(0)) / z; 2: A's own
  // tridiagonal (Tamm-Dancoff), -eta G(zeta)
  const bool poly = cfmode != 0;
  cudaStream_t st = h->stream;
  const int B = pv.B, k = o.k;
  Timer tm(h);
  JacobiBufs jb;
  jb.a = wsT<double>(h, "jac_a", (size_t)std::max(B, 1) * k);
  jb.b2 = wsT<double>(h, "jac_b2", (size_t)std::max(B, 1) * k);
  jb.w0 = wsT<double>(h, "jac_w0", (size_t)std::max(B, 1));
  jb.n = wsT<int>(h, "jac_n", (size_t)std::max(B, 1));
  unsigned long long *mt = wsT<unsigned long long>(h, "min_theta", 1);
  const double big = 1e300;
  unsigned long long bigbits;
  std::memcpy(&bigbits, &big, sizeof big);
  LGW_TRY_CUDA(h, cudaMemcpyAsync(mt, &bigbits, sizeof bigbits, cudaMemcpyHostToDevice, st));
  tm.mark(C_SPEC);
  if (B > 0 && poly) {
    // the fractions run on D = p_g(C)'s own tridiagonal (no spectral map)
    jb.poles = 0;
    jb.a = const_cast<double *>(alpha);
    jb.g0 = cfmode == 1 ? wsT<double>(h, "jac_g0", (size_t)B) : nullptr;
    launch_poly_prep(alpha, beta, beta0, k_eff, B, k, jb, h->d_status, st);
    check_launch(h, "poly_prep");
  } else if (B > 0) {
    launch_spectral_impl(alpha, beta, beta0, k_eff, B, k, jb, mt, h->d_status, st);
    check_launch(h, "spectral");
  }
  CfProblem cp{};
  cp.n_t = pv.n_t;
  cp.n_m = pv.n_m;
  cp.n_freq = pv.n_freq;
  cp.k = k;
  cp.targets = pv.d_targets;
  cp.m_idx = pv.d_m_idx;
  cp.eps = s.eps;
  cp.n_v = s.n_v;
  cp.omega = pv.d_omega;
  cp.delta = pv.delta;
  cp.shift = pv.d_shift;
  cp.qp_mode = o.qp_mode;
  tm.mark(C_CF);
  double *sig = sigma ? sigma : wsT<double>(h, "sigma_tmp", (size_t)std::max(1, pv.n_t * pv.n_freq * 2));
  const int S = cf_slices(cp);
  double *part = S > 1 ? wsT<double>(h, "cf_part", (size_t)S * pv.n_t * pv.n_freq * 2) : nullptr;
  const int ncf = launch_cf_grid(cp, jb, sig, part, S, st);
  if (ncf > 0) check_launch(h, "cf_grid");
  if (ncf > 1) check_launch(h, "cf_reduce");
  tm.mark(C_QP);
  if (e_qp && pv.n_t > 0) {
    launch_qp(cp, jb, sig, o.qp_max_iter, o.qp_tol, e_qp, z_qp, h->d_status, st);
    check_launch(h, "qp");
  }
  tm.stop();
  if (rep) {
    tm.collect(tacc, C_N);
    unsigned long long bits = 0;
    LGW_TRY_CUDA(h, cudaMemcpy(&bits, mt, sizeof bits, cudaMemcpyDeviceToHost));
    double mtv;
    std::memcpy(&mtv, &bits, sizeof mtv);
    rep->min_theta = mtv;
  }
}

void fill_report_common(lgw_handle *h, const SysDev &s, const ProbView &pv, const Opts &o,
                        const int *k_eff_dev, lgw_report *rep, const double *tacc) {
  if (!rep) return;
  rep->ms_start = tacc[C_START];
  rep->ms_gemm1 = tacc[C_GEMM1];
  rep->ms_gemm2 = tacc[C_GEMM2];
  rep->ms_dots = tacc[C_DOTS];
  rep->ms_update = tacc[C_UPDATE];
  rep->ms_pass2 = tacc[C_PASS2];
  rep->ms_normalize = tacc[C_NORM];
  rep->ms_spectral = tacc[C_SPEC];
  rep->ms_cf = tacc[C_CF];
  rep->ms_qp = tacc[C_QP];
  rep->n_vectors = pv.B;
  std::vector<int> ke(pv.B);
  if (pv.B) {
    LGW_TRY_CUDA(h, cudaMemcpy(ke.data(), k_eff_dev, sizeof(int) * pv.B, cudaMemcpyDeviceToHost));
  }
  int kmin = o.k, kmax = 0;
  double elems = 0.0;
  for (int x : ke) {
    kmin = std::min(kmin, x);
    kmax = std::max(kmax, x);
    elems += (double)s.n_vc * (double)x * (double)(x + 1) / 2.0;
  }
  rep->k_min = pv.B ? kmin : 0;
  rep->k_max = kmax;
  rep->gemm_flops = 4.0 * s.n_vc * (double)s.n_aux * (double)pv.B * (double)o.k;
  rep->reorth_elems = o.reorth != LGW_REORTH_NONE ? elems : 0.0;
}

lgw_status guard_handle(lgw_handle *h) {
  if (!h) return LGW_ERR_ARG;
  cudaError_t e = cudaSetDevice(h->device);
  if (e != cudaSuccess) return set_err(h, LGW_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(e));
  h->last = LGW_OK;
  h->msg.clear();
  return LGW_OK;
}

}  // namespace

// ===========================================================================
// exported C ABI
// ===========================================================================
namespace {
// x_lo = x_hi = 0 asks the library for the interval (estimate_interval,
// kept with the system after its first estimate).
const PolyOp *poly_arg(lgw_handle *h, const lgw_system *sys, const lgw_poly *pp, PolyOp &store) {
  if (!pp) return nullptr;
  double lo = pp->x_lo, hi = pp->x_hi;
  if (pp->g >= 1 && pp->g <= 256 && lo == 0.0 && hi == 0.0) {
    lgw_system *ms = const_cast<lgw_system *>(sys);
    if (!ms->ivl_ok) {
      estimate_interval(h, sys->s, 32, ms->ivl_lo, ms->ivl_hi);
      ms->ivl_ok = true;
    }
    lo = ms->ivl_lo;
    hi = ms->ivl_hi;
  }
  if (pp->g < 1 || pp->g > 256 || !(lo > 0.0) || !(hi > lo)) {
    set_err(h, LGW_ERR_ARG, "polynomial: need 1 <= g <= 256 and 0 < x_lo < x_hi (or both 0)");
    throw Fail{LGW_ERR_ARG};
  }
  store = make_poly(pp->g, lo, hi);
  return &store;
}

// A stretch of work beside the handle's stream, on the first lane: it starts
// after what the stream holds so far, and the stream goes on after it from
// join() (or the destructor: also when an exception passes).  Off: the stream.
struct SideStream {
  lgw_handle *h;
  cudaStream_t st;
  cudaEvent_t ev = nullptr;
  SideStream(lgw_handle *h_, bool on) : h(h_), st(h_->stream) {
    if (!on) return;
    if (h->lanes.empty()) {
      cudaStream_t l;
      LGW_TRY_CUDA(h, cudaStreamCreateWithFlags(&l, cudaStreamNonBlocking));
      h->lanes.push_back(l);
    }
    LGW_TRY_CUDA(h, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    if (cudaEventRecord(ev, h->stream) != cudaSuccess ||
        cudaStreamWaitEvent(h->lanes[0], ev, 0) != cudaSuccess) {
      cudaEventDestroy(ev);
      ev = nullptr;
      cudaGetLastError();
      return;   // on the stream itself
    }
    st = h->lanes[0];
  }
  SideStream(const SideStream &) = delete;
  void join() {
    if (!ev) return;
    if (cudaEventRecord(ev, st) != cudaSuccess || cudaStreamWaitEvent(h->stream, ev, 0) != cudaSuccess)
      cudaStreamSynchronize(st);
    cudaEventDestroy(ev);
    ev = nullptr;
  }
  ~SideStream() { join(); }
};

// Tamm-Dancoff view of a system: the same copies of L with Delta^1/2 -> 1,
// Delta^2 -> Delta, c_K Delta^1/2 -> c_K / 2 (refreshed on every use, so
// copies made later, such as the E4M3 ones, are seen).
const SysDev &tda_view(lgw_handle *h, const lgw_system *csys) {
  lgw_system *sys = const_cast<lgw_system *>(csys);
  const SysDev &s = sys->s;
  if (!sys->tda_buf) {
    const size_t N = (size_t)s.N;
    void *buf = sys_alloc(h, N * (2 * sizeof(double) + 4 * sizeof(float)));
    if (!buf) {
      set_err(h, LGW_ERR_OOM, "device allocation for the Tamm-Dancoff view failed");
      throw Fail{LGW_ERR_OOM};
    }
    sys->tda_buf = buf;
    double *ones = static_cast<double *>(buf), *cd = ones + N;
    float *onesf = reinterpret_cast<float *>(cd + N), *d2f = onesf + N, *cdf = d2f + N;
    launch_tda_view(s.Delta, s.n_vc, s.N, 0.5 * s.kf, ones, cd, onesf, d2f, cdf + N, cdf,
                    h->stream);
    check_launch(h, "tda_view");
  }
  const size_t N = (size_t)s.N;
  double *ones = static_cast<double *>(sys->tda_buf), *cd = ones + N;
  float *onesf = reinterpret_cast<float *>(cd + N), *d2f = onesf + N, *cdf = d2f + N;
  SysDev &t = sys->tda;
  t = s;
  t.kf = 0.5 * s.kf;
  t.dsq = ones;
  t.ozx = sys->ozx_tda;
  t.Delta2 = s.Delta;
  t.cd = cd;
  t.dsqf = onesf;
  t.d2f = d2f;
  t.d2lo = cdf + N;
  t.cdf = cdf;
  return t;
}

lgw_status sigma_c_impl(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                        const lgw_options *o, const lgw_poly *pp, double *sigma, double *e_qp,
                        double *z_qp, lgw_report *rep, bool tda = false) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h) return set_err(h, LGW_ERR_ARG, "bad system handle");
  try {
    cudaStream_t st = h->stream;
    h->launches = 0;
    h->ev_used = 0;
    h->timing = rep != nullptr;
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    if (rep) {
      std::memset(rep, 0, sizeof *rep);
      LGW_TRY_CUDA(h, cudaEventCreate(&t0));
      LGW_TRY_CUDA(h, cudaEventCreate(&t1));
      LGW_TRY_CUDA(h, cudaEventRecord(t0, st));
    }
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, sys->s);
    ensure_copies(h, sys, op);
    PolyOp pstore;
    const PolyOp *poly = poly_arg(h, sys, pp, pstore);
    if (poly) {
      // Lanczos on D = p_g(C) keeps the FP64 basis
      op.split = 0;
      op.split32 = 0;
    }
    const SysDev &s = tda ? tda_view(h, sys) : sys->s;
    ProbView pv = check_problem(h, s, p);
    double tacc[C_N] = {0};
    double *alpha = wsT<double>(h, "co_alpha", (size_t)std::max(1, pv.B) * op.k);
    double *beta = wsT<double>(h, "co_beta", (size_t)std::max(1, pv.B) * op.k);
    double *beta0 = wsT<double>(h, "co_beta0", (size_t)std::max(1, pv.B));
    int *ke = wsT<int>(h, "co_keff", (size_t)std::max(1, pv.B));
    OutBuf<double> sg, e, z;
    sg.init(h, "out_sigma", sigma, (size_t)pv.n_t * pv.n_freq * 2);
    e.init(h, "out_eqp", e_qp, (size_t)pv.n_t);
    z.init(h, "out_zqp", z_qp, (size_t)pv.n_t);
    run_lanczos(h, s, pv, op, alpha, beta, beta0, ke, rep, tacc, false, nullptr, poly);
    run_sigma(h, s, pv, op, alpha, beta, beta0, ke, sg.dev, e.dev, z.dev, rep, tacc,
              poly != nullptr ? 1 : (tda ? 2 : 0));
    sg.finish(h);
    e.finish(h);
    z.finish(h);
    if (rep) {
      LGW_TRY_CUDA(h, cudaEventRecord(t1, st));
      LGW_TRY_CUDA(h, cudaEventSynchronize(t1));
      float ms = 0.f;
      cudaEventElapsedTime(&ms, t0, t1);
      cudaEventDestroy(t0);
      cudaEventDestroy(t1);
      fill_report_common(h, s, pv, op, ke, rep, tacc);
      if (poly) rep->gemm_flops *= poly->g;
      rep->ms_total = ms;
      rep->gpu_launches = h->launches;
    }
    check_status(h);
    h->timing = false;
  } catch (Fail &f) {
    h->timing = false;
    return f.st;
  }
  return LGW_OK;
}
// Exact reverse mode of one sub-batch's three-term recurrence (FP64, no
// reorthogonalisation), segment by segment from the last: each segment
// [s0, s0 + ci) is recomputed from its checkpoint (q_{s0-1}, q_s0) with the
// forward's own kernels (breakdown test off: the recorded depths stand),
// then taken back step by step (k_rev_*: one dot pass, one scalar step, one
// elementwise pass, and C ubar_j through the FP64 contractions).  SC
// accumulates sum_j (ubar_j (L^T D q_j)^T + q_j (L^T D ubar_j)^T) = 2 G D L;
// then y = dF/db, SB += y M^T and the diagonal terms of dDelta.
//
// Polynomial form (poly != NULL: the recurrence runs on D = p_g(C)): each
// product D x is Clenshaw's recurrence in S = a_s C + b_s I (g products with
// C).  Taking step j back needs D ubar_j and the pairs through which dF/dD
// reaches C: Clenshaw on q_j is redone (b_1..b_g and their L^T D b_k), then
// the reverse recurrence bbar_1 = S u, bbar_k = 2 S bbar_{k-1} - bbar_{k-2}
// (u = bbar_0 = ubar_j) gives D u = c_0 u + sum_k c_k bbar_k and
//   dF/dC += a_s u b_1^T + 2 a_s sum_{k=1}^{g-1} bbar_k b_{k+1}^T.
void reverse_sweep(lgw_handle *h, const SysDev &s, const ProbView &pv, const Opts &op,
                   const VecCtx &c, const AdjCtx &a, const double *ckpt, int ci, double *SC,
                   double *SB, double *dD, double *gdeps, const PolyOp *poly) {
  cudaStream_t &st = h->stream;
  const int Bs = c.Bs, N = c.N, A = s.A, k = op.k;
  const size_t BN = (size_t)Bs * N, BA = (size_t)Bs * A;
  const int cs = std::min(ci, k), nseg = (k + ci - 1) / ci;
  double *seg = wsT<double>(h, "rev_seg", (size_t)(cs + 2) * BN);
  double *useg = wsT<double>(h, "rev_useg", (size_t)cs * BN);
  double *yseg = wsT<double>(h, "rev_yseg", (size_t)cs * BA);
  double *ybseg = wsT<double>(h, "rev_ybseg", (size_t)cs * BA);
  const F64Work f64 = f64_work(h, s, Bs);   // the recurrence's own: same width
  double *Y = wsT<double>(h, "adj_Y", BN);
  RevCtx r{};
  r.N = N;
  r.Bs = Bs;
  r.nvec = c.nvec;
  r.vec0 = c.vec0;
  r.k = k;
  r.nchunks = c.nchunks;
  r.seg = seg;
  r.qbar = wsT<double>(h, "rev_qbar", 3 * BN);
  double *cu = wsT<double>(h, "rev_cu", BN);
  r.cu = cu;
  r.useg = useg;
  r.Gd = wsT<double>(h, "adj_Gd", BN);
  // on D = p_g(C) the pairs of the reverse Clenshaw recurrence give diag(dF/dC)
  r.gd_from_steps = poly ? 0 : 1;
  r.dpart = wsT<double>(h, "rev_dpart", (size_t)Bs * c.nchunks * 6);
  r.coef = wsT<double>(h, "rev_coef", (size_t)Bs * 8);
  r.bbar = wsT<double>(h, "rev_bbar", (size_t)Bs * k);
  r.Gam = a.Gam;
  r.ay = a.ay;
  r.alpha = a.alpha;
  r.beta = a.beta;
  r.beta0 = a.beta0;
  r.k_eff = a.k_eff;
  LGW_TRY_CUDA(h, cudaMemsetAsync(r.qbar, 0, sizeof(double) * 3 * BN, st));
  LGW_TRY_CUDA(h, cudaMemsetAsync(cu, 0, sizeof(double) * BN, st));
  LGW_TRY_CUDA(h, cudaMemsetAsync(r.Gd, 0, sizeof(double) * BN, st));
  launch_rev_init(r, st);
  check_launch(h, "rev_init");
  // polynomial form: Clenshaw vectors b_k (slot k - 1), their L^T D b_k, the
  // reverse vectors bbar_1..bbar_g (slot k - 1) and L^T D bbar_{k-1}
  const int g = poly ? poly->g : 0;
  double *fb = nullptr, *fy = nullptr, *rb = nullptr, *ry = nullptr, *T = nullptr,
         *apart = nullptr, *zeros = nullptr;
  if (poly) {
    fb = wsT<double>(h, "rev_fb", (size_t)g * BN);
    fy = wsT<double>(h, "rev_fy", (size_t)g * BA);
    rb = wsT<double>(h, "rev_rb", (size_t)g * BN);
    ry = wsT<double>(h, "rev_ry", (size_t)g * BA);
    T = wsT<double>(h, "rev_T", BN);
    apart = wsT<double>(h, "rev_apart", (size_t)c.nchunks * Bs);
    zeros = wsT<double>(h, "rev_zeros", (size_t)Bs);
    LGW_TRY_CUDA(h, cudaMemsetAsync(zeros, 0, sizeof(double) * Bs, st));
  }
  // T = C x with L^T D x into yout (FP64 contractions)
  auto apply_c = [&](const double *x, double *yout) {
    f64_contract1(h, s, f64, x, Bs, yout);
    f64_contract2(h, s, f64, yout, true, Bs, EPI_APPLY, x, nullptr, nullptr, T, nullptr);
  };
  auto fbk = [&](int k) { return fb + (size_t)(k - 1) * BN; };
  auto rbk = [&](int k) { return rb + (size_t)(k - 1) * BN; };
  // Clenshaw on x: b_g .. b_1 into fb and L^T D b_k into fy; with w given,
  // also the Lanczos step's w = D x - beta_j q_{j-1} and its alpha partials
  auto clenshaw = [&](const double *x, const double *qprev, const double *betaj, double *w,
                      double *alpha_part) {
    PolyStep ps{};
    ps.N = N;
    ps.q = x;
    ps.Delta2 = s.Delta2;
    ps.dsqf = s.dsqf;
    ps.as = poly->as;
    ps.bs = poly->bs;
    ps.ck = poly->c[g];
    ps.out = fbk(g);
    launch_cheb_step(ps, c.nchunks, Bs, st);
    check_launch(h, "cheb_step(reverse)");
    for (int kk = g - 1; kk >= 0; --kk) {
      apply_c(fbk(kk + 1), fy + (size_t)kk * BA);
      ps.b1 = fbk(kk + 1);
      ps.b2 = kk + 2 <= g ? fbk(kk + 2) : nullptr;
      ps.T = T;
      ps.ck = poly->c[kk];
      if (kk > 0) {
        ps.out = fbk(kk);
        launch_cheb_step(ps, c.nchunks, Bs, st);
        check_launch(h, "cheb_step(reverse)");
      } else if (w) {
        ps.out = nullptr;
        launch_cheb_final(ps, qprev, betaj, w, alpha_part, c.nchunks, Bs, st);
        check_launch(h, "cheb_final(reverse)");
      }
    }
  };
  // the recomputation window: q_j at slot j - (s0 - 1) of seg
  VecCtx rc = c;
  rc.ring = 0;
  rc.basis = seg;
  rc.nslots = cs + 2;
  rc.tol = 0.0;
  for (int sg = nseg - 1; sg >= 0; --sg) {
    const int s0 = sg * ci, e = std::min(s0 + ci, k), n = e - s0;
    LGW_TRY_CUDA(h, cudaMemcpyAsync(seg, ckpt + (size_t)sg * 2 * BN, sizeof(double) * 2 * BN,
                                    cudaMemcpyDeviceToDevice, st));
    rc.slot0 = s0 - 1;
    r.s0 = s0;
    launch_rev_set_betaj(r, rc.betaj, st);
    check_launch(h, "rev_set_betaj");
    bool x_ready = false;
    for (int j = s0; j < e; ++j) {
      const double *qj = slot_ptr(rc, j);
      const double *qp = j > 0 ? slot_ptr(rc, j - 1) : nullptr;
      if (poly) {
        clenshaw(qj, qp, rc.betaj, rc.w, rc.alpha_part);
      } else {
        double *yj = yseg + (size_t)(j - s0) * BA;
        f64_contract1(h, s, f64, qj, Bs, yj, x_ready);
        f64_contract2(h, s, f64, yj, true, Bs, EPI_LANCZOS, qj, qp, rc.betaj, rc.w, rc.alpha_part);
      }
      const OzOperand xd = poly || j + 1 == e ? OzOperand{} : f64_next_digits(s, f64, Bs);
      if (launch_step_f64(rc, j, xd, st)) {
        check_launch(h, "step_f64(recompute)");
        x_ready = xd.d != nullptr;
        continue;
      }
      launch_alpha_reduce(rc, j, st);
      check_launch(h, "alpha_reduce(recompute)");
      launch_alpha_axpy(rc, j, st);
      check_launch(h, "alpha_axpy(recompute)");
      launch_beta_vec(rc, j, st);
      check_launch(h, "beta_vec(recompute)");
      launch_normalize(rc, j, 0, nullptr, st);
      check_launch(h, "normalize(recompute)");
    }
    for (int j = e - 1; j >= s0; --j) {
      launch_rev_step(r, j, st);
      check_launch(h, "rev_step");
      const double *uj = useg + (size_t)(j - s0) * BN;
      if (!poly) {
        double *ybj = ybseg + (size_t)(j - s0) * BA;
        f64_contract1(h, s, f64, uj, Bs, ybj);
        f64_contract2(h, s, f64, ybj, true, Bs, EPI_APPLY, uj, nullptr, nullptr, cu, nullptr);
        continue;
      }
      // Clenshaw vectors of q_j, then the reverse recurrence from u = ubar_j
      clenshaw(slot_ptr(rc, j), nullptr, nullptr, nullptr, nullptr);
      PolyStep ps{};
      ps.N = N;
      ps.q = uj;
      ps.Delta2 = s.Delta2;
      ps.dsqf = s.dsqf;
      ps.as = poly->as;
      ps.bs = poly->bs;
      ps.ck = 0.0;
      apply_c(uj, ry);
      ps.b1 = uj;
      ps.T = T;
      launch_cheb_final(ps, nullptr, zeros, rbk(1), apart, c.nchunks, Bs, st);   // S u
      check_launch(h, "cheb_final(reverse S u)");
      for (int kk = 2; kk <= g; ++kk) {
        apply_c(rbk(kk - 1), ry + (size_t)(kk - 1) * BA);
        ps.b1 = rbk(kk - 1);
        ps.b2 = kk == 2 ? uj : rbk(kk - 2);
        ps.out = rbk(kk);
        launch_cheb_step(ps, c.nchunks, Bs, st);
        check_launch(h, "cheb_step(reverse)");
      }
      // D u for qbar_j (added by the next step's first pass)
      launch_rev_axpby(cu, poly->c[0], uj, 0.0, BN, st);
      for (int kk = 1; kk <= g; ++kk) launch_rev_axpby(cu, poly->c[kk], rbk(kk), 1.0, BN, st);
      check_launch(h, "rev_axpby");
      // pairs (a_s: u, b_1) and (2 a_s: bbar_k, b_{k+1}), k = 1 .. g-1
      const double as = poly->as;
      launch_rev_gd(r.Gd, as, uj, fbk(1), BN, st);
      for (int kk = 1; kk < g; ++kk) launch_rev_gd(r.Gd, 2.0 * as, rbk(kk), fbk(kk + 1), BN, st);
      check_launch(h, "rev_gd");
      f64_atb(h, uj, N, fy, A, Bs, N, A, SC, as);
      f64_atb(h, fbk(1), N, ry, A, Bs, N, A, SC, as);
      if (g > 1) {
        f64_atb(h, rbk(1), N, fy + BA, A, (g - 1) * Bs, N, A, SC, 2.0 * as);
        f64_atb(h, fbk(2), N, ry + BA, A, (g - 1) * Bs, N, A, SC, 2.0 * as);
      }
    }
    if (poly) continue;
    f64_atb(h, useg, N, yseg, A, n * Bs, N, A, SC);
    f64_atb(h, seg + BN, N, ybseg, A, n * Bs, N, A, SC);
  }
  const double *q0 = ckpt + BN;
  launch_rev_finish(r, q0, Y, st);
  check_launch(h, "rev_finish");
  if (SB) {
    f64_atb(h, Y, N, pv.d_M + (size_t)c.vec0 * s.n_aux, s.n_aux, c.nvec, N, s.n_aux, SB);
  }
  launch_adj_accumulate(a, s.Delta, BasisRef{q0, nullptr, nullptr}, Y, r.Gd, dD, gdeps, st);
  check_launch(h, "adj_accumulate");
}
}  // namespace

extern "C" {

const char *lgw_status_string(lgw_status s) {
  switch (s) {
    case LGW_OK: return "ok";
    case LGW_ERR_ARG: return "invalid argument";
    case LGW_ERR_SHAPE: return "inconsistent shape or index";
    case LGW_ERR_CUDA: return "CUDA error";
    case LGW_ERR_OOM: return "out of device memory";
    case LGW_ERR_NOT_SPD: return "Casida matrix or Gauss node not positive";
    case LGW_ERR_NO_CONVERGENCE: return "no convergence";
    case LGW_ERR_TIMEOUT: return "device wait timed out";
    case LGW_ERR_UNSUPPORTED: return "unsupported option";
  }
  return "unknown status";
}

lgw_status lgw_create(lgw_handle **out, int device, void *cuda_stream) {
  if (!out) return LGW_ERR_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return LGW_ERR_ARG;
  }
  if (cudaSetDevice(device) != cudaSuccess) return LGW_ERR_CUDA;
  lgw_handle *h = new lgw_handle();
  h->device = device;
  h->stream = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMalloc(&h->d_status, sizeof(unsigned)) != cudaSuccess) {
    cudaGetLastError();
    delete h;
    return LGW_ERR_OOM;
  }
  cudaMemset(h->d_status, 0, sizeof(unsigned));
  *out = h;
  return LGW_OK;
}

lgw_status lgw_destroy(lgw_handle *h) {
  if (!h) return LGW_OK;
  cudaSetDevice(h->device);
  cudaStreamSynchronize(h->stream);
  h->drop_graphs();
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  for (auto l : h->lanes) cudaStreamDestroy(l);
  for (auto &kv : h->bufs)
    if (kv.second.p) cudaFree(kv.second.p);
  spare_free(h);
  for (auto e : h->ev_pool) cudaEventDestroy(e);
  if (h->d_status) cudaFree(h->d_status);
  delete h;
  return LGW_OK;
}

lgw_status lgw_set_workspace_limit(lgw_handle *h, size_t bytes) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  h->ws_limit = bytes;
  if (bytes) drop_digits(h);   // and the spare blocks
  return LGW_OK;
}

lgw_status lgw_workspace_bytes(lgw_handle *h, size_t *bytes) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!bytes) return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_workspace_bytes");
  *bytes = h->ws_bytes;
  return LGW_OK;
}

lgw_status lgw_release_workspace(lgw_handle *h) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (cudaStreamSynchronize(h->stream) != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "stream synchronisation before the release failed");
  drop_digits(h);   // and the spare blocks
  h->drop_graphs();
  for (auto &kv : h->bufs)
    if (kv.second.p) cudaFree(kv.second.p);
  h->bufs.clear();
  h->ws_bytes = 0;
  h->ws_gen++;
  return LGW_OK;
}

lgw_status lgw_selftest_bounded_wait(lgw_handle *h, int32_t arrive, double seconds) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!(seconds >= 1e-4 && seconds <= 2.0))
    return set_err(h, LGW_ERR_ARG, "self-test wait must lie in [1e-4, 2] s");
  int khz = 0;
  if (cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, h->device) != cudaSuccess || khz <= 0)
    return set_err(h, LGW_ERR_CUDA, "clock rate query failed");
  const long long cycles = (long long)(seconds * (double)khz * 1e3);
  cudaStream_t st = h->stream;
  if (cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st) != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "status reset failed");
  launch_wait_selftest(arrive != 0, cycles, h->d_status, st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "self-test launch failed: %s", cudaGetErrorString(e));
  unsigned stw = 0;
  if (cudaMemcpyAsync(&stw, h->d_status, sizeof stw, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "self-test status read failed");
  if (stw & ST_TIMEOUT)
    return set_err(h, LGW_ERR_TIMEOUT, "a bounded device wait ran out (self-test, %.3g s)",
                   seconds);
  return LGW_OK;
}

lgw_status lgw_last_error(lgw_handle *h, char *buf, size_t n) {
  if (!h) return LGW_ERR_ARG;
  if (buf && n) {
    std::strncpy(buf, h->msg.c_str(), n - 1);
    buf[n - 1] = '\0';
  }
  return h->last;
}

lgw_status lgw_prepare_system(lgw_handle *h, const lgw_system_desc *d, lgw_system **out) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!d || !out || !d->eps || !d->L) return set_err(h, LGW_ERR_ARG, "NULL descriptor field");
  if (d->n_v < 1 || d->n_c < 1 || d->n_aux < 1)
    return set_err(h, LGW_ERR_ARG, "n_v, n_c, n_aux must be >= 1");
  // the 32 x 32 transpose tiles of the operand copies use grid.y = N / 32
  if ((int64_t)d->n_v * d->n_c > (int64_t)65535 * 32)
    return set_err(h, LGW_ERR_SHAPE, "n_v * n_c above 2097120");
  if (!(d->kernel_factor >= 0.0)) return set_err(h, LGW_ERR_ARG, "kernel_factor must be >= 0");
  *out = nullptr;
  lgw_system *sys = new lgw_system();
  sys->h = h;
  SysDev &s = sys->s;
  s.n_v = d->n_v;
  s.n_c = d->n_c;
  s.n_aux = d->n_aux;
  s.n_vc = d->n_v * d->n_c;
  s.N = round_up(s.n_vc, PAD_VC);
  s.A = round_up(s.n_aux, PAD_AUX);
  s.kf = d->kernel_factor;
  std::vector<void *> allocs;
  auto alloc = [&](size_t bytes) -> void * {
    void *p = sys_alloc(h, bytes);
    if (p) allocs.push_back(p);
    return p;
  };
  const int flags = d->flags;
  if ((flags & ~(LGW_SYS_NO_FP64 | LGW_SYS_NO_BF16 | LGW_SYS_FP8)) != 0 ||
      ((flags & LGW_SYS_NO_FP64) && (flags & LGW_SYS_NO_BF16))) {
    delete sys;
    return set_err(h, LGW_ERR_ARG, "bad system flags 0x%x", flags);
  }
  const bool keep64 = !(flags & LGW_SYS_NO_FP64), keep16 = !(flags & LGW_SYS_NO_BF16);
  const int norb = s.n_v + s.n_c;
  s.eps = (double *)alloc(sizeof(double) * norb);
  s.Delta = (double *)alloc(sizeof(double) * s.N);
  s.dsq = (double *)alloc(sizeof(double) * s.N);
  s.Delta2 = (double *)alloc(sizeof(double) * s.N);
  s.cd = (double *)alloc(sizeof(double) * s.N);
  s.dsqf = (float *)alloc(sizeof(float) * s.N);
  s.d2f = (float *)alloc(2 * sizeof(float) * s.N);   // d2f, then d2lo
  s.d2lo = s.d2f ? s.d2f + s.N : nullptr;
  s.cdf = (float *)alloc(sizeof(float) * s.N);
  bool ok = s.eps && s.Delta && s.dsq && s.Delta2 && s.cd && s.dsqf && s.d2f && s.cdf;
  if (ok && keep64) ok = (s.L64 = (double *)alloc(sizeof(double) * (size_t)s.N * s.A)) != nullptr;
  if (ok && keep16) {
    s.Lb = (__nv_bfloat16 *)alloc(sizeof(__nv_bfloat16) * (size_t)s.N * s.A);
    s.Ltb = (__nv_bfloat16 *)alloc(sizeof(__nv_bfloat16) * (size_t)s.N * s.A);
    s.Lb_lo = (__nv_bfloat16 *)alloc(sizeof(__nv_bfloat16) * (size_t)s.N * s.A);
    ok = s.Lb && s.Ltb && s.Lb_lo;
  }
  if (!ok) {
    for (void *p : allocs) sys_free(h, p);
    delete sys;
    return set_err(h, LGW_ERR_OOM, "device allocation for the system failed");
  }
  try {
    cudaStream_t st = h->stream;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    if (is_device_ptr(d->eps))
      LGW_TRY_CUDA(h, cudaMemcpyAsync(s.eps, d->eps, sizeof(double) * norb, cudaMemcpyDeviceToDevice, st));
    else
      LGW_TRY_CUDA(h, cudaMemcpyAsync(s.eps, d->eps, sizeof(double) * norb, cudaMemcpyHostToDevice, st));
    const double *Lsrc = in_dev(h, "in_L", d->L, (size_t)s.n_vc * s.n_aux);
    launch_pair_energies(s, st);
    check_launch(h, "pair_energies");
    launch_check_delta(s, h->d_status, st);
    check_launch(h, "check_delta");
    if (keep64) {
      launch_pad_L(Lsrc, s, st);
      check_launch(h, "pad_L");
    }
    if (keep16) {
      launch_quantize_L(Lsrc, s.n_aux, s.n_vc, s.n_aux, s, st);
      check_launch(h, "quantize_L");
    }
    if (!keep64 || (flags & LGW_SYS_FP8)) make_fp8(h, s, Lsrc, s.n_aux, s.n_vc, s.n_aux);
    check_status(h);
  } catch (Fail &f) {
    cudaStreamSynchronize(h->stream);
    for (void *p : allocs) sys_free(h, p);
    sys_free(h, s.L8);
    sys_free(h, s.L8t);
    sys_free(h, s.sL);
    delete sys;
    return f.st;
  }
  *out = sys;
  return LGW_OK;
}

lgw_status lgw_release_system(lgw_system *sys) {
  if (!sys) return LGW_OK;
  cudaSetDevice(sys->h->device);
  cudaStreamSynchronize(sys->h->stream);
  // cached graphs may reference this system's buffers
  sys->h->drop_graphs();
  SysDev &s = sys->s;
  void *ps[] = {s.eps,  s.Delta, s.dsq, s.Delta2, s.cd,  s.dsqf,
                s.d2f, s.cdf,   s.L64, s.Lb,     s.Ltb, s.Lb_lo};
  for (void *p : ps) sys_free(sys->h, p);
  sys_free(sys->h, sys->Ltb_lo);
  sys_free(sys->h, sys->tda_buf);
  if (sys->oz_buf) {
    free_digits(sys);
    auto &v = sys->h->sliced;
    v.erase(std::remove(v.begin(), v.end(), sys), v.end());
  }
  sys_free(sys->h, s.L8);
  sys_free(sys->h, s.L8t);
  sys_free(sys->h, s.sL);
  delete sys;
  return LGW_OK;
}

lgw_status lgw_apply_casida(lgw_handle *h, const lgw_system *sys, int32_t n_vec, const double *X,
                            double *Y, int32_t precision) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || n_vec < 0 || (n_vec > 0 && (!X || !Y)))
    return set_err(h, LGW_ERR_ARG, "bad arguments to lgw_apply_casida");
  if (n_vec == 0) return LGW_OK;
  if (precision != LGW_FP64 && precision != LGW_BF16 && precision != LGW_FP8 &&
      precision != LGW_FP8_DEQ)
    return set_err(h, LGW_ERR_ARG, "bad precision");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    const bool tc = precision != LGW_FP64;
    const bool fp8 = precision == LGW_FP8;
    const bool deq = precision == LGW_FP8_DEQ;
    if (tc && !tc_available()) {
      set_err(h, LGW_ERR_UNSUPPORTED, "tensor-core paths need an sm_103 device");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    {
      Opts oa{};
      oa.precision = precision;
      ensure_copies(h, sys, oa);
    }
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    const double *Xd = in_dev(h, "ap_xin", X, (size_t)n_vec * s.n_vc);
    OutBuf<double> Yo;
    Yo.init(h, "ap_yout", Y, (size_t)n_vec * s.n_vc);
    int Bs = round_up(n_vec, PAD_VEC);
    if (tc) Bs = std::max(Bs, 64);
    double *xp = wsT<double>(h, "ap_x", (size_t)Bs * s.N);
    double *wp = wsT<double>(h, "ap_w", (size_t)Bs * s.N);
    LGW_TRY_CUDA(h, cudaMemsetAsync(xp, 0, sizeof(double) * Bs * s.N, st));
    LGW_TRY_CUDA(h, cudaMemcpy2DAsync(xp, sizeof(double) * s.N, Xd, sizeof(double) * s.n_vc,
                                      sizeof(double) * s.n_vc, n_vec, cudaMemcpyDeviceToDevice, st));
    double *Y64 = wsT<double>(h, "y64", (size_t)Bs * s.A);
    if (tc) {
      __nv_bfloat16 *xh = wsT<__nv_bfloat16>(h, "ap_xh", (size_t)Bs * s.N);
      float *yp = wsT<float>(h, "ap_yp32", (size_t)64 * Bs * s.A);
      __nv_bfloat16 *yh = wsT<__nv_bfloat16>(h, "ap_yh", (size_t)Bs * s.A);
      launch_scale_rows_to_bf16(xp, s.dsq, Bs, s.N, xh, st);
      check_launch(h, "scale_rows_to_bf16");
      char err[256];
      int splits = 1;
      TcPlan *plan = tc_plan_create(s, Bs, xh, yp, yh, &splits, err, sizeof err);
      if (!plan) {
        set_err(h, LGW_ERR_CUDA, "%s", err);
        throw Fail{LGW_ERR_CUDA};
      }
      uint8_t *x8 = nullptr, *y8 = nullptr;
      float *sx = nullptr, *ty = nullptr;
      if (fp8) {
        x8 = wsT<uint8_t>(h, "ap_x8", (size_t)Bs * s.N);
        y8 = wsT<uint8_t>(h, "ap_y8", (size_t)Bs * s.A);
        sx = wsT<float>(h, "ap_sx", (size_t)Bs);
        ty = wsT<float>(h, "ap_ty", (size_t)Bs);
        if (!tc_plan_enable_fp8(plan, s.L8t, s.L8, x8, y8, ty)) {
          tc_plan_destroy(plan);
          set_err(h, LGW_ERR_CUDA, "cuTensorMapEncodeTiled failed for the E4M3 operands");
          throw Fail{LGW_ERR_CUDA};
        }
        launch_quant_x8(xh, Bs, s.N, x8, sx, st);
        check_launch(h, "quant_x8");
      }
      uint16_t *x16 = nullptr, *y16 = nullptr;
      if (deq) {
        x16 = wsT<uint16_t>(h, "ap_x16", (size_t)Bs * s.N);
        y16 = wsT<uint16_t>(h, "ap_y16", (size_t)Bs * s.A);
        sx = wsT<float>(h, "ap_sx", (size_t)Bs);
        ty = wsT<float>(h, "ap_ty", (size_t)Bs);
        if (!tc_plan_enable_deq(plan, s.L8t, s.L8, x16, y16, ty)) {
          tc_plan_destroy(plan);
          set_err(h, LGW_ERR_CUDA, "cuTensorMapEncodeTiled failed for the widened E4M3 operands");
          throw Fail{LGW_ERR_CUDA};
        }
        launch_quant_x16(xh, Bs, s.N, x16, sx, st);
        check_launch(h, "quant_x16");
      }
      launch_gemm1_tc(plan, h->d_status, st);
      check_launch(h, "gemm1_tc");
      if (fp8)
        launch_reduce_y_fp8(yp, splits, Bs, s.A, sx, s.sL, y8, ty, nullptr, 1, st);
      else if (deq)
        launch_reduce_y_f16(yp, splits, Bs, s.A, sx, s.sL, y16, ty, nullptr, 1, st);
      else
        launch_reduce_y_bf16(yp, splits, Bs, s.A, yh, nullptr, st);
      check_launch(h, "reduce_y");
      launch_gemm2_tc(plan, EPI_APPLY, xp, nullptr, nullptr, wp, nullptr, h->d_status, st);
      check_launch(h, "gemm2_tc");
      LGW_TRY_CUDA(h, cudaStreamSynchronize(st));
      tc_plan_destroy(plan);
    } else {
      const F64Work f64 = f64_work(h, s, Bs);
      f64_contract1(h, s, f64, xp, Bs, Y64);
      f64_contract2(h, s, f64, Y64, true, Bs, EPI_APPLY, xp, nullptr, nullptr, wp, nullptr);
    }
    LGW_TRY_CUDA(h, cudaMemcpy2DAsync(Yo.dev, sizeof(double) * s.n_vc, wp, sizeof(double) * s.N,
                                      sizeof(double) * s.n_vc, n_vec, cudaMemcpyDeviceToDevice, st));
    Yo.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_lanczos_coeffs(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                              const lgw_options *o, double *alpha, double *beta, double *beta0,
                              int32_t *k_eff) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !alpha || !beta || !beta0 || !k_eff)
    return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_lanczos_coeffs");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, s);
    ensure_copies(h, sys, op);
    ProbView pv = check_problem(h, s, p);
    OutBuf<double> a, b, b0;
    OutBuf<int32_t> ke;
    a.init(h, "out_alpha", alpha, (size_t)pv.B * op.k);
    b.init(h, "out_beta", beta, (size_t)pv.B * op.k);
    b0.init(h, "out_beta0", beta0, (size_t)pv.B);
    ke.init(h, "out_keff", k_eff, (size_t)pv.B);
    h->timing = false;
    run_lanczos(h, s, pv, op, a.dev, b.dev, b0.dev, ke.dev, nullptr, nullptr);
    a.finish(h);
    b.finish(h);
    b0.finish(h);
    ke.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_sigma_from_coeffs(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                                 const lgw_options *o, const double *alpha, const double *beta,
                                 const double *beta0, const int32_t *k_eff, double *sigma,
                                 double *e_qp, double *z_qp) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !alpha || !beta || !beta0 || !k_eff)
    return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_sigma_from_coeffs");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, s);
    ProbView pv = check_problem(h, s, p);
    const double *da = in_dev(h, "in_alpha", alpha, (size_t)pv.B * op.k);
    const double *db = in_dev(h, "in_beta", beta, (size_t)pv.B * op.k);
    const double *db0 = in_dev(h, "in_beta0", beta0, (size_t)pv.B);
    const int *dke = in_dev(h, "in_keff", k_eff, (size_t)pv.B);
    OutBuf<double> sg, e, z;
    sg.init(h, "out_sigma", sigma, (size_t)pv.n_t * pv.n_freq * 2);
    e.init(h, "out_eqp", e_qp, (size_t)pv.n_t);
    z.init(h, "out_zqp", z_qp, (size_t)pv.n_t);
    h->timing = false;
    run_sigma(h, s, pv, op, da, db, db0, dke, sg.dev, e.dev, z.dev, nullptr, nullptr);
    sg.finish(h);
    e.finish(h);
    z.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_sigma_c(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                       const lgw_options *o, double *sigma, double *e_qp, double *z_qp,
                       lgw_report *rep) {
  return sigma_c_impl(h, sys, p, o, nullptr, sigma, e_qp, z_qp, rep);
}

lgw_status lgw_sigma_c_tda(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                           const lgw_options *o, double *sigma, double *e_qp, double *z_qp,
                           lgw_report *rep) {
  return sigma_c_impl(h, sys, p, o, nullptr, sigma, e_qp, z_qp, rep, true);
}

lgw_status lgw_sigma_offdiag(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                             const lgw_options *o, int32_t n_pairs, const int32_t *pairs,
                             double *sigma_od) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || n_pairs < 0 || (n_pairs > 0 && (!pairs || !sigma_od)))
    return set_err(h, LGW_ERR_ARG, "bad arguments to lgw_sigma_offdiag");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    h->timing = false;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, s);
    ensure_copies(h, sys, op);
    ProbView pv = check_problem(h, s, p);
    if (n_pairs == 0) return LGW_OK;
    std::vector<int> hp = to_host(h, pairs, (size_t)2 * n_pairs);
    for (int x : hp)
      if (x < 0 || x >= pv.n_t) {
        set_err(h, LGW_ERR_SHAPE, "pair index %d outside [0, n_t = %d)", x, pv.n_t);
        throw Fail{LGW_ERR_SHAPE};
      }
    // virtual request: rows 2i, 2i+1 = factors of t + t' and t - t' (pair i)
    ProbView pv2 = pv;
    pv2.n_t = 2 * n_pairs;
    pv2.B = pv2.n_t * pv.n_m;
    pv2.targets.assign(pv2.n_t, 0);
    for (int i = 0; i < n_pairs; ++i) pv2.targets[2 * i] = pv2.targets[2 * i + 1] = pv.targets[hp[2 * i]];
    pv2.d_targets = in_dev(h, "od_targets", pv2.targets.data(), (size_t)pv2.n_t);
    const int *dpairs = in_dev(h, "od_pairs", hp.data(), hp.size());
    pv2.d_shift = nullptr;
    if (pv.d_M) {
      double *M2 = wsT<double>(h, "od_M", (size_t)pv2.B * s.n_aux);
      launch_pol_rows(pv.d_M, pv.n_m, s.n_aux, dpairs, n_pairs, M2, st);
      check_launch(h, "pol_rows");
      pv2.d_M = M2;
    } else {
      double *V2 = wsT<double>(h, "od_V", (size_t)pv2.B * s.n_vc);
      launch_pol_rows(pv.d_V, pv.n_m, s.n_vc, dpairs, n_pairs, V2, st);
      check_launch(h, "pol_rows");
      pv2.d_V = V2;
    }
    double *alpha = wsT<double>(h, "co_alpha", (size_t)pv2.B * op.k);
    double *beta = wsT<double>(h, "co_beta", (size_t)pv2.B * op.k);
    double *beta0 = wsT<double>(h, "co_beta0", (size_t)pv2.B);
    int *ke = wsT<int>(h, "co_keff", (size_t)pv2.B);
    double *sig2 = wsT<double>(h, "od_sigma", (size_t)pv2.n_t * pv.n_freq * 2);
    run_lanczos(h, s, pv2, op, alpha, beta, beta0, ke, nullptr, nullptr);
    run_sigma(h, s, pv2, op, alpha, beta, beta0, ke, sig2, nullptr, nullptr, nullptr, nullptr);
    OutBuf<double> out;
    out.init(h, "out_sigma_od", sigma_od, (size_t)n_pairs * pv.n_freq * 2);
    launch_pol_combine(sig2, n_pairs, pv.n_freq, out.dev, st);
    check_launch(h, "pol_combine");
    out.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_spectral_interval(lgw_handle *h, const lgw_system *sys, int32_t k, double *x_lo,
                                 double *x_hi) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !x_lo || !x_hi)
    return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_spectral_interval");
  if (k < 1 || k > 4095) return set_err(h, LGW_ERR_ARG, "k = %d outside [1, 4095]", k);
  if (!sys->s.L64 && !sys->s.Lb)
    return set_err(h, LGW_ERR_UNSUPPORTED, "the interval needs the FP64 or the BF16 copy of L");
  try {
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), h->stream));
    h->timing = false;
    estimate_interval(h, sys->s, k, *x_lo, *x_hi);
    check_status(h);
    if (k == 32) {   // the estimate lgw_sigma_c_poly uses when asked for one
      lgw_system *ms = const_cast<lgw_system *>(sys);
      ms->ivl_lo = *x_lo;
      ms->ivl_hi = *x_hi;
      ms->ivl_ok = true;
    }
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_sigma_band(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                          const lgw_options *o, double *sigma, lgw_report *rep) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !sigma) return set_err(h, LGW_ERR_ARG, "bad arguments to lgw_sigma_band");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    h->launches = 0;
    h->ev_used = 0;
    h->timing = rep != nullptr;
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    if (rep) {
      std::memset(rep, 0, sizeof *rep);
      LGW_TRY_CUDA(h, cudaEventCreate(&t0));
      LGW_TRY_CUDA(h, cudaEventCreate(&t1));
      LGW_TRY_CUDA(h, cudaEventRecord(t0, st));
    }
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, s);
    if (op.precision == LGW_FP8 || op.precision == LGW_FP8_DEQ) {
      set_err(h, LGW_ERR_UNSUPPORTED, "band Lanczos runs FP64 or BF16 contractions");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    if (op.k > 512) {
      set_err(h, LGW_ERR_UNSUPPORTED, "band Lanczos: k = %d above its 512-step limit", op.k);
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    ensure_copies(h, sys, op);
    ProbView pv = check_problem(h, s, p);
    const int P = pv.n_t, G = pv.n_m, F = pv.n_freq, k = op.k;
    if (P < 1 || P > 8) {
      set_err(h, LGW_ERR_UNSUPPORTED, "band Lanczos: n_t = %d targets, 1..8 supported", P);
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    OutBuf<double> out;
    out.init(h, "out_sigma_band", sigma, (size_t)P * P * F * 2);
    double tacc[C_N] = {0};
    if (G > 0 && F > 0) {
      double *Tb = wsT<double>(h, "band_T", (size_t)G * k * (P + 1));
      double *R0 = wsT<double>(h, "band_R0", (size_t)G * P * P);
      int *keff = wsT<int>(h, "band_keff", (size_t)G);
      run_band(h, s, pv, op, Tb, R0, keff, rep ? tacc : nullptr);
      // polarisation vectors of the small problem: e_a, then e_a +- e_b
      const int nx = P + P * (P - 1);
      std::vector<double> xs((size_t)nx * P, 0.0);
      for (int a = 0; a < P; ++a) xs[(size_t)a * P + a] = 1.0;
      int q = 0;
      for (int a = 0; a < P; ++a)
        for (int b = a + 1; b < P; ++b, ++q) {
          double *xp = &xs[(size_t)(P + 2 * q) * P], *xm = xp + P;
          xp[a] = xm[a] = 1.0;
          xp[b] = 1.0;
          xm[b] = -1.0;
        }
      const double *dxs = in_dev(h, "band_xs", xs.data(), xs.size());
      const int Bx = nx * G;
      double *a2 = wsT<double>(h, "co_alpha", (size_t)Bx * k);
      double *b2 = wsT<double>(h, "co_beta", (size_t)Bx * k);
      double *b02 = wsT<double>(h, "co_beta0", (size_t)Bx);
      int *ke2 = wsT<int>(h, "co_keff", (size_t)Bx);
      double *scr = wsT<double>(h, "band_small", (size_t)Bx * (k + 2) * k);
      launch_band_small(Tb, R0, keff, G, k, P, dxs, nx, op.tol, scr, a2, b2, b02, ke2, st);
      check_launch(h, "band_small");
      ProbView pv3 = pv;
      pv3.n_t = nx;
      pv3.B = Bx;
      pv3.d_targets = nullptr;
      pv3.d_shift = nullptr;
      double *sigx = wsT<double>(h, "band_sigx", (size_t)nx * F * 2);
      run_sigma(h, s, pv3, op, a2, b2, b02, ke2, sigx, nullptr, nullptr, rep, tacc);
      launch_band_combine(sigx, P, F, out.dev, st);
      check_launch(h, "band_combine");
    } else if (out.dev) {
      LGW_TRY_CUDA(h, cudaMemsetAsync(out.dev, 0, sizeof(double) * (size_t)P * P * F * 2, st));
    }
    out.finish(h);
    if (rep) {
      LGW_TRY_CUDA(h, cudaEventRecord(t1, st));
      LGW_TRY_CUDA(h, cudaEventSynchronize(t1));
      float ms = 0.f;
      cudaEventElapsedTime(&ms, t0, t1);
      cudaEventDestroy(t0);
      cudaEventDestroy(t1);
      rep->ms_total = ms;
      rep->ms_start = tacc[C_START];
      rep->ms_gemm1 = tacc[C_GEMM1];
      rep->ms_gemm2 = tacc[C_GEMM2];
      rep->ms_dots = tacc[C_DOTS];
      rep->ms_spectral = tacc[C_SPEC];
      rep->ms_cf = tacc[C_CF];
      rep->n_vectors = G;
      rep->gemm_flops = 4.0 * s.n_vc * (double)s.n_aux * (double)G * (double)k;
      rep->gpu_launches = h->launches;
      rep->k_min = rep->k_max = k;
    }
    check_status(h);
    h->timing = false;
  } catch (Fail &f) {
    h->timing = false;
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_sigma_c_poly(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                            const lgw_options *o, const lgw_poly *poly, double *sigma,
                            double *e_qp, double *z_qp, lgw_report *rep) {
  if (!poly) return h ? set_err(h, LGW_ERR_ARG, "polynomial descriptor is NULL") : LGW_ERR_ARG;
  return sigma_c_impl(h, sys, p, o, poly, sigma, e_qp, z_qp, rep);
}

lgw_status lgw_lanczos_coeffs_poly(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                                   const lgw_options *o, const lgw_poly *pp, double *alpha,
                                   double *beta, double *beta0, int32_t *k_eff) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !pp || !alpha || !beta || !beta0 || !k_eff)
    return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_lanczos_coeffs_poly");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, s);
    ensure_copies(h, sys, op);
    PolyOp pstore;
    const PolyOp *poly = poly_arg(h, sys, pp, pstore);
    op.split = 0;
    op.split32 = 0;
    ProbView pv = check_problem(h, s, p);
    OutBuf<double> a, b, b0;
    OutBuf<int32_t> ke;
    a.init(h, "out_alpha", alpha, (size_t)pv.B * op.k);
    b.init(h, "out_beta", beta, (size_t)pv.B * op.k);
    b0.init(h, "out_beta0", beta0, (size_t)pv.B);
    ke.init(h, "out_keff", k_eff, (size_t)pv.B);
    h->timing = false;
    run_lanczos(h, s, pv, op, a.dev, b.dev, b0.dev, ke.dev, nullptr, nullptr, false, nullptr,
                poly);
    a.finish(h);
    b.finish(h);
    b0.finish(h);
    ke.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_sigma_c_batched(lgw_handle *h, int32_t n_sys, const lgw_system *const *systems,
                               const lgw_problem *problems, const lgw_options *o,
                               double *const *sigma, double *const *e_qp, double *const *z_qp,
                               lgw_report *rep) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (n_sys < 0 || (n_sys > 0 && (!systems || !problems || !sigma || !e_qp)))
    return set_err(h, LGW_ERR_ARG, "bad arguments to lgw_sigma_c_batched");
  for (int i = 0; i < n_sys; ++i)
    if (!systems[i] || systems[i]->h != h)
      return set_err(h, LGW_ERR_ARG, "bad system handle at index %d", i);
  if (rep) std::memset(rep, 0, sizeof *rep);
  if (n_sys == 0) return LGW_OK;
  const cudaStream_t caller = h->stream;
  // every exit restores the caller's stream and the default workspace names; one
  // that leaves before the lanes are joined waits for what they still run (the
  // caller may release those systems next)
  struct Restore {
    lgw_handle *h;
    cudaStream_t st;
    bool joined = false;
    ~Restore() {
      h->stream = st;
      h->ws_prefix.clear();
      h->timing = false;
      if (!joined)
        for (cudaStream_t l : h->lanes) cudaStreamSynchronize(l);
    }
  } restore{h, caller};
  try {
    h->launches = 0;
    h->ev_used = 0;
    h->timing = false;
    cudaEvent_t t0 = nullptr, t1 = nullptr, fork = nullptr;
    if (rep) {
      LGW_TRY_CUDA(h, cudaEventCreate(&t0));
      LGW_TRY_CUDA(h, cudaEventCreate(&t1));
      LGW_TRY_CUDA(h, cudaEventRecord(t0, caller));
    }
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), caller));
    // systems are independent: up to 4 run at once, system i on lane i % 4
    const int S = std::min(n_sys, 4);
    while ((int)h->lanes.size() < S) {
      cudaStream_t l;
      LGW_TRY_CUDA(h, cudaStreamCreateWithFlags(&l, cudaStreamNonBlocking));
      h->lanes.push_back(l);
    }
    LGW_TRY_CUDA(h, cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
    LGW_TRY_CUDA(h, cudaEventRecord(fork, caller));
    for (int l = 0; l < S; ++l) LGW_TRY_CUDA(h, cudaStreamWaitEvent(h->lanes[l], fork, 0));
    struct Done {
      int B, k, n_vc, n_aux, reorth;
      const int *ke;
    };
    std::vector<Done> done;
    for (int i = 0; i < n_sys; ++i) {
      const int lane = i % S;
      h->stream = h->lanes[lane];
      h->ws_prefix = "lane" + std::to_string(lane) + "/";
      const SysDev &s = systems[i]->s;
      Opts op = resolve_opts(h, o, s);
      ensure_copies(h, systems[i], op);
      ProbView pv = check_problem(h, s, &problems[i]);
      double *alpha = wsT<double>(h, "co_alpha", (size_t)std::max(1, pv.B) * op.k);
      double *beta = wsT<double>(h, "co_beta", (size_t)std::max(1, pv.B) * op.k);
      double *beta0 = wsT<double>(h, "co_beta0", (size_t)std::max(1, pv.B));
      int *ke = wsT<int>(h, "co_keff" + std::to_string(i), (size_t)std::max(1, pv.B));
      OutBuf<double> sg, e, z;
      sg.init(h, "out_sigma", sigma[i], (size_t)pv.n_t * pv.n_freq * 2);
      e.init(h, "out_eqp", e_qp[i], (size_t)pv.n_t);
      z.init(h, "out_zqp", z_qp ? z_qp[i] : nullptr, (size_t)pv.n_t);
      run_lanczos(h, s, pv, op, alpha, beta, beta0, ke, nullptr, nullptr);
      run_sigma(h, s, pv, op, alpha, beta, beta0, ke, sg.dev, e.dev, z.dev, nullptr, nullptr);
      sg.finish(h);
      e.finish(h);
      z.finish(h);
      done.push_back({pv.B, op.k, s.n_vc, s.n_aux, op.reorth, ke});
    }
    h->stream = caller;
    h->ws_prefix.clear();
    for (int l = 0; l < S; ++l) {
      LGW_TRY_CUDA(h, cudaEventRecord(fork, h->lanes[l]));
      LGW_TRY_CUDA(h, cudaStreamWaitEvent(caller, fork, 0));
    }
    restore.joined = true;
    cudaEventDestroy(fork);
    if (rep) {
      LGW_TRY_CUDA(h, cudaEventRecord(t1, caller));
      LGW_TRY_CUDA(h, cudaEventSynchronize(t1));
      float ms = 0.f;
      cudaEventElapsedTime(&ms, t0, t1);
      cudaEventDestroy(t0);
      cudaEventDestroy(t1);
      rep->ms_total = ms;
      rep->gpu_launches = h->launches;
      int kmin = 1 << 30, kmax = 0;
      for (const Done &d : done) {
        std::vector<int> kv(d.B);
        if (d.B)
          LGW_TRY_CUDA(h, cudaMemcpy(kv.data(), d.ke, sizeof(int) * d.B, cudaMemcpyDeviceToHost));
        for (int x : kv) {
          kmin = std::min(kmin, x);
          kmax = std::max(kmax, x);
          if (d.reorth != LGW_REORTH_NONE)
            rep->reorth_elems += (double)d.n_vc * (double)x * (double)(x + 1) / 2.0;
        }
        rep->n_vectors += d.B;
        rep->gemm_flops += 4.0 * d.n_vc * (double)d.n_aux * (double)d.B * (double)d.k;
      }
      rep->k_min = rep->n_vectors ? kmin : 0;
      rep->k_max = kmax;
      rep->n_sub_batches = n_sys;
    }
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

static lgw_status backward_impl(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                                const lgw_options *o, const double *dE, double *dL,
                                double *deps, bool tda, const lgw_poly *pp = nullptr) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !dE) return set_err(h, LGW_ERR_ARG, "NULL argument to the backward call");
  try {
    cudaStream_t st = h->stream;
    h->timing = false;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    Opts op = resolve_opts(h, o, sys->s);
    ensure_copies(h, sys, op);
    const SysDev &s = tda ? tda_view(h, sys) : sys->s;
    if (op.qp_mode != 0) {
      set_err(h, LGW_ERR_UNSUPPORTED, "the adjoint differentiates the graphical QP solution (qp_mode 0)");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    // FP64 contractions without reorthogonalisation: the exact reverse mode
    // of the three-term recurrence, recomputed from Krylov checkpoints;
    // otherwise the Krylov form over the stored basis
    const bool exact = op.reorth == LGW_REORTH_NONE && op.precision == LGW_FP64;
    const int ci = (o->ckpt_every > 0) ? o->ckpt_every : 16;
    if (o->ckpt_every < 0) {
      set_err(h, LGW_ERR_ARG, "ckpt_every < 0");
      throw Fail{LGW_ERR_ARG};
    }
    // the polynomial form is differentiated exactly only (the Krylov form
    // would need the eigenvectors of C behind p_g); its interval is held fixed
    PolyOp pstore;
    const PolyOp *poly = poly_arg(h, sys, pp, pstore);
    if (poly && !exact) {
      set_err(h, LGW_ERR_UNSUPPORTED,
              "the polynomial form's adjoint needs FP64 contractions without reorthogonalisation");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    if (poly) {
      op.split = 0;
      op.split32 = 0;
    }
    // the adjoint contracts with the stored Krylov basis: FP64 (FP64 mode)
    // or the split float pair (BF16 mode with split arithmetic); the split
    // basis needs reorthogonalisation (otherwise the FP64 basis is kept)
    if (op.reorth == LGW_REORTH_NONE || op.precision == LGW_FP64) {
      op.split = 0;
      op.split32 = 0;
    }
    if (op.k > adj_max_k()) {
      set_err(h, LGW_ERR_UNSUPPORTED, "k = %d above the %d-step limit of the adjoint", op.k,
              adj_max_k());
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    if (!s.L64 || (op.precision != LGW_FP64 && !s.Ltb)) {
      set_err(h, LGW_ERR_UNSUPPORTED,
              "the adjoint needs the FP64 copy of L (and the BF16 copies for BF16/FP8)");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    ProbView pv = check_problem(h, s, p);
    const int B = pv.B, k = op.k, N = s.N, A = s.A;
    const double *d_dE = in_dev(h, "in_dE", dE, (size_t)pv.n_t);
    OutBuf<double> oL, oe;
    oL.init(h, "out_dL", dL, (size_t)s.n_vc * s.n_aux);
    oe.init(h, "out_deps", deps, (size_t)(s.n_v + s.n_c));
    double *gdeps = wsT<double>(h, "adj_deps", (size_t)(s.n_v + s.n_c));
    LGW_TRY_CUDA(h, cudaMemsetAsync(gdeps, 0, sizeof(double) * (s.n_v + s.n_c), st));
    if (B == 0 || pv.n_t == 0) {
      if (oL.dev) LGW_TRY_CUDA(h, cudaMemsetAsync(oL.dev, 0, sizeof(double) * s.n_vc * s.n_aux, st));
      if (pv.n_t > 0) {
        // no summed orbitals: E_t = eps_t + s_t, Z_t = 1
        std::vector<double> one(pv.n_t, 1.0);
        double *Z1 = wsT<double>(h, "adj_Z", (size_t)pv.n_t);
        LGW_TRY_CUDA(h, cudaMemcpyAsync(Z1, one.data(), sizeof(double) * pv.n_t,
                                        cudaMemcpyHostToDevice, st));
        double *dD = wsT<double>(h, "adj_dDelta", (size_t)N);
        LGW_TRY_CUDA(h, cudaMemsetAsync(dD, 0, sizeof(double) * N, st));
        launch_adj_deps(dD, s.n_v, s.n_c, pv.d_targets, pv.n_t, Z1, d_dE, gdeps, st);
        check_launch(h, "adj_deps");
      }
      if (oe.dev)
        LGW_TRY_CUDA(h, cudaMemcpyAsync(oe.dev, gdeps, sizeof(double) * (s.n_v + s.n_c),
                                        cudaMemcpyDeviceToDevice, st));
      oL.finish(h);
      oe.finish(h);
      LGW_TRY_CUDA(h, cudaStreamSynchronize(st));
      return LGW_OK;
    }
    const bool tc = op.precision != LGW_FP64;
    // sub-batch: the caller's b_sub, else as many vectors as fit in half of
    // the free device memory (plus what the handle already holds)
    {
      size_t fr = 0, tot = 0;
      LGW_TRY_CUDA(h, cudaMemGetInfo(&fr, &tot));
      size_t held = 0;
      for (auto &kv : h->bufs) held += kv.second.n;
      const int cs = std::min(ci, k), nseg = (k + ci - 1) / ci;
      // exact form: checkpoints, the recomputation window, ubar_j, the qbar ring
      // and row buffers, plus (polynomial form) Clenshaw's 2 g + 1 vectors
      const int gp = poly ? poly->g : 0;
      const double per_vec =
          exact ? 8.0 * (2 * nseg + 2 * cs + 12 + 2 * gp + 1) * N + 16.0 * (cs + gp) * A +
                      40.0 * k * k
                : 8.0 * (k + 1) * N + (tc ? 4.0 * k * N : 0.0) + 20.0 * k * A + 48.0 * N +
                      40.0 * k * k;
      const double budget = 0.5 * (double)(fr + held);
      int fit = (int)std::min<double>(budget / per_vec, 1 << 20);
      fit = std::max(PAD_VEC, fit / PAD_VEC * PAD_VEC);
      if (op.b_sub <= 0) op.b_sub = std::min(B, fit);
    }
    const int bsub = std::min(op.b_sub, B);
    const bool one_pass = bsub >= B;
    if (tc && !sys->Ltb_lo) {
      lgw_system *ms = const_cast<lgw_system *>(sys);
      ms->Ltb_lo = static_cast<__nv_bfloat16 *>(
          sys_alloc(h, sizeof(__nv_bfloat16) * (size_t)N * A));
      if (!ms->Ltb_lo) {
        set_err(h, LGW_ERR_OOM, "device allocation for the low half of L^T failed");
        throw Fail{LGW_ERR_OOM};
      }
      launch_split_t(BasisRef{s.L64, nullptr, nullptr}, N, A, A, nullptr, ms->Ltb_lo, st);
      check_launch(h, "split_t(L lo)");
    }
    // coefficients of the forward pass
    double *alpha = wsT<double>(h, "co_alpha", (size_t)B * k);
    double *beta = wsT<double>(h, "co_beta", (size_t)B * k);
    double *beta0 = wsT<double>(h, "co_beta0", (size_t)B);
    int *ke = wsT<int>(h, "co_keff", (size_t)B);
    double *E = wsT<double>(h, "adj_E", (size_t)pv.n_t);
    double *Z = wsT<double>(h, "adj_Z", (size_t)pv.n_t);
    // accumulators
    double *SC = wsT<double>(h, "adj_SC", (size_t)N * A);
    double *SB = pv.d_M ? wsT<double>(h, "adj_SB", (size_t)N * s.n_aux) : nullptr;
    double *dD = wsT<double>(h, "adj_dDelta", (size_t)N);
    LGW_TRY_CUDA(h, cudaMemsetAsync(SC, 0, sizeof(double) * N * A, st));
    if (SB) LGW_TRY_CUDA(h, cudaMemsetAsync(SB, 0, sizeof(double) * N * s.n_aux, st));
    LGW_TRY_CUDA(h, cudaMemsetAsync(dD, 0, sizeof(double) * N, st));

    auto forward_sigma = [&]() {
      run_sigma(h, s, pv, op, alpha, beta, beta0, ke, nullptr, E, Z, nullptr, nullptr,
                poly ? 1 : (tda ? 2 : 0));
    };
    // Krylov checkpoints of the exact mode: (q_{s0-1}, q_s0) at every segment
    // start s0 = 0, ci, 2 ci, ... (q_{-1} = 0), copied out of the forward's
    // three-vector ring
    const int nseg = (k + ci - 1) / ci;
    double *ckpt = nullptr;
    StepHook keep_ckpt = [&](const VecCtx &c, int j) {
      const size_t BN = (size_t)c.Bs * c.N;
      if (j < 0) {
        ckpt = wsT<double>(h, "rev_ckpt", (size_t)nseg * 2 * BN);
        LGW_TRY_CUDA(h, cudaMemsetAsync(ckpt, 0, sizeof(double) * BN, st));
        LGW_TRY_CUDA(h, cudaMemcpyAsync(ckpt + BN, slot_ptr(c, 0), sizeof(double) * BN,
                                        cudaMemcpyDeviceToDevice, st));
        return;
      }
      const int nx = j + 1;
      if (nx % ci != 0 || nx >= k) return;
      double *dst = ckpt + (size_t)(nx / ci) * 2 * BN;
      LGW_TRY_CUDA(h, cudaMemcpyAsync(dst, slot_ptr(c, j), sizeof(double) * BN,
                                      cudaMemcpyDeviceToDevice, st));
      LGW_TRY_CUDA(h, cudaMemcpyAsync(dst + BN, slot_ptr(c, nx), sizeof(double) * BN,
                                      cudaMemcpyDeviceToDevice, st));
    };
    SubBatchHook adjoint = [&](const VecCtx &c) {
      if (one_pass) forward_sigma();
      const int Bs = c.Bs;
      const BasisRef qb = op.split ? BasisRef{nullptr, c.bhi, c.blo}
                                   : BasisRef{c.basis, nullptr, nullptr};
      AdjCtx a{};
      a.N = N;
      a.Bs = Bs;
      a.nvec = c.nvec;
      a.vec0 = c.vec0;
      a.k = k;
      a.n_m = pv.n_m;
      a.n_v = s.n_v;
      a.alpha = alpha;
      a.beta = beta;
      a.beta0 = beta0;
      a.k_eff = ke;
      a.E = E;
      a.Z = Z;
      a.dE = d_dE;
      a.eps = s.eps;
      a.m_idx = pv.d_m_idx;
      a.delta = pv.delta;
      const size_t kk = (size_t)k * k;
      a.theta = wsT<double>(h, "adj_theta", (size_t)Bs * k);
      a.V = wsT<double>(h, "adj_V", (size_t)Bs * kk);
      a.Phi = wsT<double>(h, "adj_Phi", (size_t)Bs * kk);
      a.X = wsT<double>(h, "adj_X", (size_t)Bs * kk);
      a.ay = wsT<double>(h, "adj_ay", (size_t)Bs * k);
      a.Gam = wsT<double>(h, "adj_Gam", (size_t)Bs * kk);
      a.Gamf = tc ? wsT<float>(h, "adj_Gamf", (size_t)Bs * kk) : nullptr;
      a.dz = wsT<double>(h, "adj_dz", (size_t)Bs);
      a.status = h->d_status;
      a.tda = tda ? 1 : 0;
      a.poly = poly ? 1 : 0;
      // The eigenvectors take one block per vector and a serial chain (25 ms at
      // 128 vectors, k 120) that leaves the chip idle: on the tensor-core path
      // what does not need them runs beside them, P = Q^T D L and the transposed
      // split of Q (7.5 ms, of which 7.2 are saved), where a block still fits
      // beside a tile of the GEMM (24 KB).
      const int rows = k * Bs;
      const bool beside = tc && !exact && (size_t)6 * k * sizeof(double) <= (size_t)20 * 1024;
      double *P = nullptr, *R = nullptr;
      __nv_bfloat16 *Shi = nullptr, *Slo = nullptr, *Rhi = nullptr, *Rlo = nullptr;
      auto products_of_q = [&](cudaStream_t ss) {
        // P = Q^T D L: three split-BF16 products, FP64 sums of 16384-long chunks;
        // then the transposed split of Q in the same buffers
        char err[256];
        launch_split_scaled(qb, rows, N, s.dsq, Shi, Slo, ss);
        check_launch(h, "split_scaled(D Q)");
        // Ltb is K-block-major; the adjoint's own Ltb_lo is row-major
        const __nv_bfloat16 *pa[3] = {s.Ltb, s.Ltb, sys->Ltb_lo};
        const int pk[3] = {1, 1, 0};
        const __nv_bfloat16 *pb[3] = {Shi, Slo, Shi};
        if (!tc_gemm_f64out(3, pa, pk, pb, A, rows, N, 16384, P, A, 0, h->d_status, ss, err,
                            sizeof err)) {
          set_err(h, LGW_ERR_CUDA, "%s", err);
          throw Fail{LGW_ERR_CUDA};
        }
        check_launch(h, "tc_gemm_f64out(P)");
        launch_split_t(qb, rows, N, N, Shi, Slo, ss);
        check_launch(h, "split_t(Q)");
      };
      if (!exact) {
        P = wsT<double>(h, "adj_P", (size_t)rows * A);
        R = wsT<double>(h, "adj_R", (size_t)rows * A);
        if (tc) {
          Shi = wsT<__nv_bfloat16>(h, "adj_Shi", (size_t)rows * N);
          Slo = wsT<__nv_bfloat16>(h, "adj_Slo", (size_t)rows * N);
          Rhi = wsT<__nv_bfloat16>(h, "adj_Rhi", (size_t)rows * A);
          Rlo = wsT<__nv_bfloat16>(h, "adj_Rlo", (size_t)rows * A);
        }
      }
      {
        // the eigenvectors stay on the stream and so start first, a block per SM
        SideStream side(h, beside);
        launch_eig_full(a, st);
        check_launch(h, "eig_full");
        if (tc && !exact) products_of_q(side.st);
        side.join();
      }
      launch_adj_coeffs(a, st);
      check_launch(h, "adj_coeffs");
      if (exact) {
        reverse_sweep(h, s, pv, op, c, a, ckpt, ci, SC, SB, dD, gdeps, poly);
        return;
      }
      double *Y = wsT<double>(h, "adj_Y", (size_t)Bs * N);
      double *Gd = wsT<double>(h, "adj_Gd", (size_t)Bs * N);
      if (tc)
        launch_adj_rows_f32(a, qb, Y, Gd, st);
      else
        launch_adj_rows(a, qb, Y, Gd, st);
      check_launch(h, "adj_rows");
      if (tc) {
        char err[256];
        launch_gamma_p(a, P, A, R, st);
        check_launch(h, "gamma_p");
        // SC += Q R  (M = N_aux, N = N_vc, K = k Bs, transposed split operands)
        launch_split_t(BasisRef{R, nullptr, nullptr}, rows, A, A, Rhi, Rlo, st);
        check_launch(h, "split_t(R)");
        const __nv_bfloat16 *qa[3] = {Rhi, Rhi, Rlo};
        const __nv_bfloat16 *qb[3] = {Shi, Slo, Shi};
        if (!tc_gemm_f64out(3, qa, nullptr, qb, A, N, rows, 16384, SC, A, 1, h->d_status, st, err,
                            sizeof err)) {
          set_err(h, LGW_ERR_CUDA, "%s", err);
          throw Fail{LGW_ERR_CUDA};
        }
        check_launch(h, "tc_gemm_f64out(SC)");
      } else {
        // P = Q^T D L over the k * Bs basis rows (FP64 GEMM1), R = Gam P
        f64_contract1(h, s, f64_work(h, s, rows, "adj_"), c.basis, rows, P);
        launch_gamma_p(a, P, A, R, st);
        check_launch(h, "gamma_p");
        f64_atb(h, c.basis, N, R, A, rows, N, A, SC);
      }
      // SB += Y^T M
      if (SB) {
        f64_atb(h, Y, N, pv.d_M + (size_t)c.vec0 * s.n_aux, s.n_aux, c.nvec, N, s.n_aux, SB);
      }
      launch_adj_accumulate(a, s.Delta, qb, Y, Gd, dD, gdeps, st);
      check_launch(h, "adj_accumulate");
    };
    // the exact mode keeps only the three-vector ring and the checkpoints
    const bool keep = !exact;
    const StepHook *sh = exact ? &keep_ckpt : nullptr;
    if (one_pass) {
      run_lanczos(h, s, pv, op, alpha, beta, beta0, ke, nullptr, nullptr, keep, &adjoint, poly,
                  sh);
    } else {
      run_lanczos(h, s, pv, op, alpha, beta, beta0, ke, nullptr, nullptr, false, nullptr, poly);
      forward_sigma();
      run_lanczos(h, s, pv, op, alpha, beta, beta0, ke, nullptr, nullptr, keep, &adjoint, poly,
                  sh);
    }
    double *dLdev = oL.dev ? oL.dev : wsT<double>(h, "adj_dL", (size_t)s.n_vc * s.n_aux);
    // the exact mode accumulates SC = sum_j (ubar_j y_j^T + q_j ybar_j^T) = 2 G D L
    launch_adj_dL(s.L64, s.dsq, SC, SB, A, s.n_vc, s.n_aux, exact ? 0.5 * s.kf : s.kf, dLdev, dD,
                  tda ? 1 : 0, st);
    check_launch(h, "adj_dL");
    launch_adj_deps(dD, s.n_v, s.n_c, pv.d_targets, pv.n_t, Z, d_dE, gdeps, st);
    check_launch(h, "adj_deps");
    if (oe.dev)
      LGW_TRY_CUDA(h, cudaMemcpyAsync(oe.dev, gdeps, sizeof(double) * (s.n_v + s.n_c),
                                      cudaMemcpyDeviceToDevice, st));
    oL.finish(h);
    oe.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_sigma_c_backward(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                                const lgw_options *o, const double *dE, double *dL,
                                double *deps) {
  return backward_impl(h, sys, p, o, dE, dL, deps, false);
}

lgw_status lgw_sigma_c_tda_backward(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                                    const lgw_options *o, const double *dE, double *dL,
                                    double *deps) {
  return backward_impl(h, sys, p, o, dE, dL, deps, true);
}

lgw_status lgw_sigma_c_poly_backward(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                                     const lgw_options *o, const lgw_poly *poly, const double *dE,
                                     double *dL, double *deps) {
  if (!poly) return set_err(h, LGW_ERR_ARG, "NULL polynomial to lgw_sigma_c_poly_backward");
  return backward_impl(h, sys, p, o, dE, dL, deps, false, poly);
}

lgw_status lgw_sigma_x(lgw_handle *h, const lgw_system *sys, const lgw_problem *p,
                       double *sigma_x) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !sigma_x) return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_sigma_x");
  try {
    const SysDev &s = sys->s;
    cudaStream_t st = h->stream;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    ProbView pv = check_problem(h, s, p);
    if (!pv.d_M) {
      set_err(h, LGW_ERR_UNSUPPORTED, "the exchange self-energy needs the pair factors M");
      throw Fail{LGW_ERR_UNSUPPORTED};
    }
    OutBuf<double> out;
    out.init(h, "out_sigma_x", sigma_x, (size_t)pv.n_t);
    launch_sigma_x(pv.d_M, pv.n_t, pv.n_m, s.n_aux, pv.d_m_idx, s.n_v, out.dev, st);
    if (pv.n_t > 0) check_launch(h, "sigma_x");
    out.finish(h);
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

lgw_status lgw_fit_factors(lgw_handle *h, int32_t n_pairs, int32_t n_aux, const double *C,
                           const double *metric, double *B) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (n_pairs < 0 || n_aux < 1 || (n_pairs > 0 && (!C || !B)) || !metric)
    return set_err(h, LGW_ERR_ARG, "bad arguments to lgw_fit_factors");
  try {
    cudaStream_t st = h->stream;
    LGW_TRY_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st));
    const double *Vd = in_dev(h, "in_metric", metric, (size_t)n_aux * n_aux);
    double *R = wsT<double>(h, "fit_R", (size_t)n_aux * n_aux);
    const double *Cd = nullptr;
    OutBuf<double> out;
    FitWork f;
    if (n_pairs > 0) {
      Cd = in_dev(h, "in_fitC", C, (size_t)n_pairs * n_aux);
      out.init(h, "out_fitB", B, (size_t)n_pairs * n_aux);
      f = fit_work(h, n_pairs, n_aux);
    }
    {
      // the factorisation is a serial chain that leaves the chip idle: what
      // needs C alone runs beside it, the first pairs' digits too where they
      // take longer than the fork and join, else the scales only
      const bool fork = f.a.d && (size_t)n_pairs * n_aux >= (size_t)1 << 21;
      ColMax cm;
      if (f.a.d && !fork) cm = ColMax{Cd, n_pairs, f.col};
      launch_fit_init(Vd, n_aux, R, cm.col, round_up(n_aux, 64), st);
      check_launch(h, "fit_init");
      SideStream side(h, fork);
      if (fork) fit_begin(h, f, Cd, n_pairs, n_aux, side.st);
      h->launches += launch_cholesky(R, n_aux, h->d_status, st, cm);
      check_launch(h, "cholesky");
      side.join();
      if (cm.col) fit_slice(h, f, Cd, n_pairs, n_aux, 0, st);
    }
    if (n_pairs > 0) {
      f64_fit(h, f, Cd, R, n_pairs, n_aux, out.dev);
      out.finish(h);
    }
    check_status(h);
  } catch (Fail &f) {
    return f.st;
  }
  return LGW_OK;
}

}  // extern "C"

// ===========================================================================
// Allocation-free variant of lgw_sigma_from_coeffs.
//
// Some callers cannot let a library allocate device memory while they run:
// services that hand the library a fixed device-memory budget at start-up,
// or latency-bound loops where cudaMalloc/cudaFree would synchronise the
// device and stall other streams.  This entry point performs the spectral
// map, the continued fractions on the grid and the QP solve with all of its
// scratch in one file-scope device array of fixed size; the caller passes
// inputs and outputs as device pointers.
// ===========================================================================
namespace {

// 2^21 doubles = 16 MiB on every device that loads the library, held until
// the process exits.  Layout per call: poles [B][k], weights [B][k], w0 [B],
// depth [B] (ints, rounded up), 3 B k doubles that are not used (they keep
// the accepted sizes what they were), one word for the smallest Gauss node.
constexpr size_t kNoallocDoubles = (size_t)1 << 21;
static __device__ __align__(256) double g_noalloc_scratch[kNoallocDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double *g_noalloc_addr[kMaxDevices] = {nullptr};

// Sets the Gauss-node minimum word and checks every target / summed index
// and every depth k_eff against [0, k].  It only reads the index arrays;
// the caller reads the status word before launching anything that
// dereferences an index.
__global__ void k_noalloc_prologue(unsigned long long *min_theta_bits, const int *targets, int n_t,
                                   const int *m_idx, int n_m, int norb, const int *k_eff, int B,
                                   int k, unsigned *status) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *min_theta_bits = 0x7FEFFFFFFFFFFFFFull;   // largest finite double
  if (i < n_t && (targets[i] < 0 || targets[i] >= norb)) atomicOr(status, ST_BAD_INPUT);
  if (i < n_m && (m_idx[i] < 0 || m_idx[i] >= norb)) atomicOr(status, ST_BAD_INPUT);
  if (i < B && (k_eff[i] < 0 || k_eff[i] > k)) atomicOr(status, ST_BAD_INPUT);
}

// Device memory of device `dev` (managed memory counts as any device's).
bool is_device_ptr_on(const void *p, int dev) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type == cudaMemoryTypeManaged) return true;
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

size_t noalloc_doubles_needed(size_t B, size_t k) {
  return 2 * B * k + B + (B + 1) / 2 + 3 * B * k + 1;
}

}  // namespace

extern "C" lgw_status lgw_sigma_from_coeffs_noalloc(lgw_handle *h, const lgw_system *sys,
                                                    const lgw_problem *p, const lgw_options *o,
                                                    const double *alpha, const double *beta,
                                                    const double *beta0, const int32_t *k_eff,
                                                    double *sigma, double *e_qp, double *z_qp) {
  lgw_status g = guard_handle(h);
  if (g != LGW_OK) return g;
  if (!sys || sys->h != h || !p || !o || !alpha || !beta || !beta0 || !k_eff || !sigma ||
      !e_qp)
    return set_err(h, LGW_ERR_ARG, "NULL argument to lgw_sigma_from_coeffs_noalloc");
  const SysDev &s = sys->s;
  const int n_t = p->n_t, n_m = p->n_m, n_freq = p->n_freq, k = o->k;
  if (n_t < 1 || n_m < 1 || n_freq < 1 || !p->targets || !p->m_idx || !p->omega)
    return set_err(h, LGW_ERR_ARG, "noalloc: n_t, n_m, n_freq must be >= 1 with their arrays");
  if (k < 1 || k > s.n_vc) return set_err(h, LGW_ERR_ARG, "noalloc: k outside [1, n_vc]");
  if (k > 4095)
    return set_err(h, LGW_ERR_UNSUPPORTED, "noalloc: k = %d above the 4095-step limit", k);
  if (o->qp_mode != 0 && o->qp_mode != 1)
    return set_err(h, LGW_ERR_ARG, "noalloc: unknown qp_mode %d", o->qp_mode);
  if (!(p->delta > 0.0)) return set_err(h, LGW_ERR_ARG, "noalloc: delta must be > 0");
  const void *dev_ptrs[] = {alpha, beta, beta0, k_eff, sigma, e_qp, p->targets, p->m_idx,
                            p->omega};
  for (const void *q : dev_ptrs)
    if (!is_device_ptr_on(q, h->device))
      return set_err(h, LGW_ERR_ARG, "noalloc: every array must be device memory of device %d",
                     h->device);
  if ((z_qp && !is_device_ptr_on(z_qp, h->device)) ||
      (p->static_shift && !is_device_ptr_on(p->static_shift, h->device)))
    return set_err(h, LGW_ERR_ARG, "noalloc: every array must be device memory of device %d",
                   h->device);
  const size_t B = (size_t)n_t * (size_t)n_m;
  if (noalloc_doubles_needed(B, (size_t)k) > kNoallocDoubles)
    return set_err(h, LGW_ERR_UNSUPPORTED,
                   "noalloc: n_t*n_m*(5k+2) exceeds the %zu-double static scratch (B=%zu, k=%d)",
                   kNoallocDoubles, B, k);
  if (h->device < 0 || h->device >= kMaxDevices)
    return set_err(h, LGW_ERR_UNSUPPORTED, "noalloc: device index beyond %d", kMaxDevices);

  // One-time set-up per device: host code cannot use the array's name as a
  // device address, so fetch the address with that device current.
  double *base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[h->device]) {
      void *ptr = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
      if (e != cudaSuccess)
        return set_err(h, LGW_ERR_CUDA, "noalloc: cudaGetSymbolAddress failed: %s",
                       cudaGetErrorString(e));
      g_noalloc_addr[h->device] = static_cast<double *>(ptr);
    }
    base = g_noalloc_addr[h->device];
  }
  JacobiBufs jb;
  jb.a = base;
  jb.b2 = jb.a + B * k;
  jb.w0 = jb.b2 + B * k;
  jb.n = reinterpret_cast<int *>(jb.w0 + B);
  double *work = jb.w0 + B + (B + 1) / 2;
  unsigned long long *mt = reinterpret_cast<unsigned long long *>(work + 3 * B * k);

  cudaStream_t st = h->stream;
  if (cudaMemsetAsync(h->d_status, 0, sizeof(unsigned), st) != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "noalloc: status reset failed");
  // Index check first, and its verdict read back before any kernel that
  // dereferences an index (eps[m], eps[t], the k_eff-deep rows) is queued.
  const size_t nmax = std::max<size_t>(std::max(n_t, n_m), B);
  launch_pdl(k_noalloc_prologue, dim3((unsigned)((nmax + 255) / 256)), dim3(256), 0, st, mt,
             p->targets, n_t, p->m_idx, n_m, s.n_v + s.n_c, k_eff, (int)B, k, h->d_status);
  {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
      return set_err(h, LGW_ERR_CUDA, "noalloc: index check launch failed: %s",
                     cudaGetErrorString(e));
    unsigned stw = 0;
    if (cudaMemcpyAsync(&stw, h->d_status, sizeof stw, cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return set_err(h, LGW_ERR_CUDA, "noalloc: status read failed");
    if (stw & ST_BAD_INPUT)
      return set_err(h, LGW_ERR_SHAPE,
                     "noalloc: orbital index outside [0, n_v + n_c) or k_eff outside [0, k]");
  }
  launch_spectral_impl(alpha, beta, beta0, k_eff, (int)B, k, jb, mt, h->d_status, st);
  CfProblem cp{};
  cp.n_t = n_t;
  cp.n_m = n_m;
  cp.n_freq = n_freq;
  cp.k = k;
  cp.targets = p->targets;
  cp.m_idx = p->m_idx;
  cp.eps = s.eps;
  cp.n_v = s.n_v;
  cp.omega = p->omega;
  cp.delta = p->delta;
  cp.shift = p->static_shift;
  cp.qp_mode = o->qp_mode;
  launch_cf_grid(cp, jb, sigma, nullptr, 1, st);
  const int qp_iter = o->qp_max_iter > 0 ? o->qp_max_iter : 50;
  const double qp_tol = o->qp_tol > 0 ? o->qp_tol : 1e-10;
  launch_qp(cp, jb, sigma, qp_iter, qp_tol, e_qp, z_qp, h->d_status, st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "noalloc: kernel launch failed: %s", cudaGetErrorString(e));
  unsigned stw = 0;
  if (cudaMemcpyAsync(&stw, h->d_status, sizeof stw, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return set_err(h, LGW_ERR_CUDA, "noalloc: status read failed");
  if (stw & ST_TIMEOUT) return set_err(h, LGW_ERR_TIMEOUT, "a bounded device wait ran out");
  if (stw & ST_NOT_SPD) return set_err(h, LGW_ERR_NOT_SPD, "non-positive Gauss node");
  if (stw & ST_NO_CONV)
    return set_err(h, LGW_ERR_NO_CONVERGENCE, "tridiagonal eigensolver or QP did not converge");
  return LGW_OK;
}
