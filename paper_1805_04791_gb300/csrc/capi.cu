// extern "C" entry points of include/vie.h: argument checks, handle life
// cycle and dispatch to the set-up, apply and solver translation units.
#include <chrono>
#include <cmath>
#include <cstring>
#include <mutex>
#include <set>
#include <utility>
#include <string>

#include "vie_internal.h"

namespace vie {

static thread_local std::string g_last_error;

static std::mutex g_cfg_mutex;
static std::set<std::pair<int, const void*>> g_cfg_done;

bool kernel_configured(const void* kernel) {
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(g_cfg_mutex);
  return g_cfg_done.count({dev, kernel}) != 0;
}

void kernel_mark_configured(const void* kernel) {
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(g_cfg_mutex);
  g_cfg_done.insert({dev, kernel});
}

void set_error(const std::string& msg) { g_last_error = msg; }

// Device memory comes from one pool per device, which keeps up to a thirty-second
// of the device (kPoolShare) mapped when problems are destroyed: mapping and
// unmapping cost about 1 ms a gigabyte each way, a fifth of a request at 192^3
// (whole request 118 -> 99 ms at 192^3, 6.4 -> 5.1 ms at 64^3).  The pool gives
// everything unused back when one of the library's allocations fails (which is
// then tried again), when a problem is destroyed while less than an eighth of
// the device is free, and when the caller asks for it (vie_release_memory): another
// allocator in the process cannot take what the pool keeps.  Pools are made once per device and live as long as the
// process; the CUDA calls on them are thread-safe and stream-ordered.
static const int kPoolShare = 32, kPoolDevices = 64;
static std::mutex g_pool_mutex;
static cudaMemPool_t g_pool[kPoolDevices] = {nullptr};
static bool g_pool_tried[kPoolDevices] = {false};

// The pool of the current device; nullptr (the device's default pool) if it cannot be made.
static cudaMemPool_t device_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kPoolDevices) return nullptr;
  std::lock_guard<std::mutex> g(g_pool_mutex);
  if (g_pool_tried[dev]) return g_pool[dev];
  g_pool_tried[dev] = true;
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.handleTypes = cudaMemHandleTypeNone;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  size_t freeb = 0, total = 0;
  if (cudaMemGetInfo(&freeb, &total) == cudaSuccess && cudaMemPoolCreate(&pool, &props) == cudaSuccess) {
    uint64_t keep = total / kPoolShare;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess) {
      g_pool[dev] = pool;
      return pool;
    }
    cudaMemPoolDestroy(pool);
  }
  cudaGetLastError();
  return nullptr;
}

cudaError_t dalloc(void** p, size_t bytes, cudaStream_t st) {
  *p = nullptr;
  if (bytes == 0) bytes = 256;
  cudaMemPool_t pool = device_pool();
  if (!pool) return cudaMallocAsync(p, bytes, st);
  cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (e != cudaErrorMemoryAllocation || cudaStreamIsCapturing(st, &cap) != cudaSuccess ||
      cap != cudaStreamCaptureStatusNone)
    return e;
  cudaGetLastError();
  cudaStreamSynchronize(st);  // what was freed on this stream is unused now
  cudaMemPoolTrimTo(pool, 0);
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

void dfree(void* p, cudaStream_t st) {
  if (p) cudaFreeAsync(p, st);
}

size_t pool_unused() {
  cudaMemPool_t pool = device_pool();
  uint64_t reserved = 0, used = 0;
  if (!pool || cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess)
    return 0;
  return reserved > used ? (size_t)(reserved - used) : 0;
}

static void pool_give_back() {
  size_t freeb = 0, total = 0;
  cudaMemPool_t pool = device_pool();
  if (pool && cudaMemGetInfo(&freeb, &total) == cudaSuccess && freeb < total / 8) cudaMemPoolTrimTo(pool, 0);
}

// Pinned host blocks of the solver-state mirrors: one size, at most kPinnedKept of
// them kept for the next problem (allocating and freeing one takes 0.3 ms).
static const size_t kPinnedKept = 16;
static std::vector<void*> g_pinned;

cudaError_t pinned_take(void** p) {
  {
    std::lock_guard<std::mutex> g(g_pool_mutex);
    if (!g_pinned.empty()) {
      *p = g_pinned.back();
      g_pinned.pop_back();
      return cudaSuccess;
    }
  }
  return cudaMallocHost(p, kPinnedBytes);
}

void pinned_give(void* p) {
  {
    std::lock_guard<std::mutex> g(g_pool_mutex);
    if (g_pinned.size() < kPinnedKept) {
      g_pinned.push_back(p);
      return;
    }
  }
  cudaFreeHost(p);
}

vie_status cuda_fail(cudaError_t e, const char* what) {
  cudaGetLastError();  // the runtime keeps it for the next check otherwise, which would report it again
  g_last_error = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? VIE_ENOMEM : VIE_ECUDA;
}

bool ranges_overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t pa = (uintptr_t)a, pb = (uintptr_t)b;
  return pa < pb + nb && pb < pa + na;
}

size_t grid_vec_bytes(const vie_problem* P, int c, int nrhs, size_t elem) {
  return elem * (size_t)nrhs * (size_t)c * (size_t)P->n * (size_t)P->n * (size_t)P->n;
}

// Grid sizes: any n in [4, 512].  2n and 3n that factor into the codelet
// radices (2, 3, 5, 7, 11) take direct transforms, others Bluestein's; an
// allocation that fails returns VIE_ENOMEM.
static bool valid_size(int n) { return n >= 4 && n <= 512; }

int conv_half(int n) {
  for (int m = n;; ++m) {
    int r = m;
    for (int p : {2, 3, 5, 7, 11})
      while (r % p == 0) r /= p;
    if (r == 1) return m;
  }
}

static void free_set(KernelSet& k, cudaStream_t st) {
  dfree(k.oct64, st);
  dfree(k.oct32, st);
  dfree(k.octdf, st);
  k.oct64 = nullptr;
  k.oct32 = nullptr;
  k.octdf = nullptr;
}

static void free_problem(vie_problem* P) {
  if (!P) return;
  cudaStream_t st = P->stream;
  // steps of a solve, on whatever stream, write to the buffers and to the pinned block;
  // each is followed by one of these events or runs on cap_stream
  if (P->cap_stream) cudaStreamSynchronize(P->cap_stream);
  for (cudaEvent_t e : P->arn_ev)
    if (e) cudaEventSynchronize(e);
  void* ptrs[] = {P->tw64, P->tw32, P->He64, P->He32, P->Hm64, P->Hm32, P->twdf, P->Hedf, P->Hmdf,
                  P->base_oct, P->ws.buf, P->ks.buf, P->dflag};
  for (void* q : ptrs) dfree(q, st);
  free_set(P->kapply, st);
  free_set(P->keval, st);
  cudaStreamSynchronize(st);
  for (cudaEvent_t e : P->prof.ev) cudaEventDestroy(e);
  for (cudaEvent_t e : P->arn_ev)
    if (e) cudaEventDestroy(e);
  if (P->arn_host) pinned_give(P->arn_host);
  for (cudaGraphExec_t g : P->graph_exec)
    if (g) cudaGraphExecDestroy(g);
  for (cudaEvent_t e : P->cap_ev)
    if (e) cudaEventDestroy(e);
  if (P->cap_stream) cudaStreamDestroy(P->cap_stream);
  delete P;
  pool_give_back();
}

}  // namespace vie

using namespace vie;

extern "C" {

const char* vie_last_error(void) { return g_last_error.c_str(); }

vie_status vie_problem_create(int kind, int n, double lo, double hi, double omega, const void* eps, const void* mu,
                              void* stream, vie_problem** out) {
  g_last_error.clear();
  if (!out) {
    set_error("out is NULL");
    return VIE_EINVAL;
  }
  *out = nullptr;
  if (kind < VIE_LAPLACE || kind > VIE_MAXWELL) {
    set_error("unknown kind");
    return VIE_EINVAL;
  }
  if (!valid_size(n)) {
    set_error("n must be in [4, 512]");
    return VIE_EINVAL;
  }
  if (!(hi > lo) || !std::isfinite(lo) || !std::isfinite(hi)) {
    set_error("box must satisfy lo < hi");
    return VIE_EINVAL;
  }
  if (!(omega >= 0.0) || !std::isfinite(omega)) {
    set_error("omega must be finite and >= 0");
    return VIE_EINVAL;
  }
  if (kind != VIE_LAPLACE && omega == 0.0) {
    set_error("Helmholtz/Maxwell need omega > 0 (use a tiny omega for the quasi-static limit)");
    return VIE_EINVAL;
  }
  if (!eps) {
    set_error("eps is NULL");
    return VIE_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const auto t_start = std::chrono::steady_clock::now();
  vie_problem* P = new vie_problem();
  P->kind = kind;
  P->n = n;
  P->has_mu = (kind == VIE_MAXWELL && mu != nullptr) ? 1 : 0;
  P->ncomp = P->has_mu ? 6 : 3;
  P->lo = lo;
  P->hi = hi;
  P->D = hi - lo;
  P->h = P->D / n;
  P->L = std::sqrt(3.0) * P->D;
  P->omega = kind == VIE_LAPLACE ? 0.0 : omega;
  cudaGetDevice(&P->device);
  P->stream = st;
  P->nk = conv_half(n);
  if (!make_line_plan(2 * P->nk, &P->planM) || P->planM.Q != P->planM.M) {
    delete P;
    set_error("bad FFT size");
    return VIE_EINVAL;
  }
  vie_status s = VIE_OK;
  cudaError_t e = dalloc((void**)&P->dflag, sizeof(int) * 4, st);
  if (e != cudaSuccess) s = cuda_fail(e, "cudaMalloc(flag)");
  if (s == VIE_OK) s = make_line_table(P->planM, &P->tw64, &P->tw32, st);
  if (s == VIE_OK) s = build_medium(P, eps, mu, st);
  if (s == VIE_OK) s = build_kernels(P, st);
  if (s == VIE_OK) {
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) s = cuda_fail(e, "vie_problem_create");
  }
  if (s != VIE_OK) {
    free_problem(P);
    return s;
  }
  P->t_precompute = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count();
  *out = P;
  return VIE_OK;
}

int vie_problem_ncomp(const vie_problem* P) { return P ? P->ncomp : 0; }

vie_status vie_apply(vie_problem* P, const void* x, void* y, int precision, int nrhs, void* stream) {
  if (!P || !x || !y || nrhs < 1 || (precision != VIE_FP64 && precision != VIE_FP32 && precision != VIE_DF64)) {
    set_error("vie_apply: bad argument");
    return VIE_EINVAL;
  }
  const size_t vb = grid_vec_bytes(P, P->ncomp, nrhs, precision == VIE_FP32 ? sizeof(float2) : sizeof(double2));
  if (ranges_overlap(x, vb, y, vb)) {
    set_error("vie_apply: x and y must not overlap");
    return VIE_EINVAL;
  }
  return run_apply(P, P->kapply, x, y, precision, nrhs, true, (cudaStream_t)stream);
}

vie_status vie_rhs_plane_wave(vie_problem* P, const double* d, const double* p, int nrhs, void* rhs_out,
                              void* stream) {
  if (!P || !d || !rhs_out || nrhs < 1 || (P->kind == VIE_MAXWELL && !p)) {
    set_error("vie_rhs_plane_wave: bad argument");
    return VIE_EINVAL;
  }
  // a plane wave needs a unit propagation direction (|d| fixes the wavenumber w |d|)
  // and, for Maxwell, a transverse polarisation (d . p = 0, else E_in is not a
  // solution of the free-space equations); Laplace's d is the field E0 itself
  for (int r = 0; r < nrhs && P->kind != VIE_LAPLACE; ++r) {
    const double* dr = d + 3 * (size_t)r;
    const double dn = std::sqrt(dr[0] * dr[0] + dr[1] * dr[1] + dr[2] * dr[2]);
    if (!(std::fabs(dn - 1.0) <= 1e-8)) {
      set_error("vie_rhs_plane_wave: d must be a unit vector");
      return VIE_EINVAL;
    }
    if (P->kind == VIE_MAXWELL) {
      const double* pr = p + 3 * (size_t)r;
      const double pn = std::sqrt(pr[0] * pr[0] + pr[1] * pr[1] + pr[2] * pr[2]);
      const double dp = dr[0] * pr[0] + dr[1] * pr[1] + dr[2] * pr[2];
      if (!std::isfinite(pn) || !(std::fabs(dp) <= 1e-8 * pn)) {
        set_error("vie_rhs_plane_wave: p must be finite and perpendicular to d");
        return VIE_EINVAL;
      }
    }
  }
  return run_rhs(P, d, p, nrhs, rhs_out, (cudaStream_t)stream);
}

vie_status vie_solve(vie_problem* P, const void* rhs, void* J, const vie_solve_opts* opt, vie_solve_info* info,
                     void* stream) {
  if (!P || !rhs || !J || !opt || opt->nrhs < 1 || opt->restart < 1 || opt->restart > 200 || !(opt->tol > 0) ||
      opt->max_inner < 1 || opt->max_outer < 0 ||
      (opt->mode == VIE_SOLVE_MIXED && !(opt->inner_tol > 0 && opt->inner_tol < 1)) ||
      (opt->mode != VIE_SOLVE_FP64 && opt->mode != VIE_SOLVE_MIXED && opt->mode != VIE_SOLVE_BICGSTAB) ||
      (opt->check_fp64 != 0 && opt->check_fp64 != 1)) {
    set_error("vie_solve: bad argument");
    return VIE_EINVAL;
  }
  const size_t vb = grid_vec_bytes(P, P->ncomp, opt->nrhs, sizeof(double2));
  if (ranges_overlap(rhs, vb, J, vb)) {
    set_error("vie_solve: rhs and J must not overlap");
    return VIE_EINVAL;
  }
  return run_solve(P, rhs, J, opt, info, (cudaStream_t)stream);
}

vie_status vie_eval_scattered(vie_problem* P, const void* J, void* field_out, int nrhs, void* stream) {
  if (!P || !J || !field_out || nrhs < 1) {
    set_error("vie_eval_scattered: bad argument");
    return VIE_EINVAL;
  }
  if (ranges_overlap(J, grid_vec_bytes(P, P->ncomp, nrhs, sizeof(double2)), field_out,
                     grid_vec_bytes(P, P->kind == VIE_MAXWELL ? 6 : 1, nrhs, sizeof(double2)))) {
    set_error("vie_eval_scattered: J and field_out must not overlap");
    return VIE_EINVAL;
  }
  vie_status s = build_eval_kernels(P, (cudaStream_t)stream);
  if (s != VIE_OK) return s;
  return run_apply(P, P->keval, J, field_out, VIE_FP64, nrhs, false, (cudaStream_t)stream);
}

size_t vie_problem_bytes(int kind, int n, int nrhs, int restart, int has_mu) {
  if (n < 1 || nrhs < 1 || restart < 1) return 0;
  const bool mx = kind == VIE_MAXWELL, mu = mx && has_mu;
  const size_t N = (size_t)n * n * n, nk = (size_t)conv_half(n), media = mu ? 2 : 1;
  const size_t O = nk + 1, O3 = O * O * O, S = 3 * (size_t)n / 2 + 1;
  const int c = mu ? 6 : 3, narr = mu ? 9 : 6, nfield = mx ? 9 : 3;
  const size_t medium = 144 * N * media + 64 * 1024;  // H: 6 entries, FP64 + FP32; flags, line table
  const size_t bases = 16 * O3 * 4;
  // set-up scratch (compute_symbols): two line-operator buffers, the table of G^, line tables
  const size_t scratch = 32 * (S * S * O + S * O * O) + 48 * S * S + 1080 * 2 * (size_t)n;
  // a mixed solve of nrhs right-hand sides: kernels, double-word copies, Krylov workspace
  const size_t solve = medium + bases + 40 * O3 * narr + 96 * N * media + krylov_bytes((long long)(c * N), restart, nrhs);
  // the scattered field after it: set-up of the base that the operator does not need,
  // beside the solve's workspace; then its kernels and its own (E and H: six components)
  const size_t base = solve + apply_workspace_bytes(n, (int)nk, c, nrhs, VIE_FP64) + (mu ? 0 : scratch);
  const size_t field = solve + 24 * O3 * nfield + apply_workspace_bytes(n, (int)nk, mx ? 6 : 3, nrhs, VIE_FP64);
  return std::max(medium + bases + scratch, std::max(base, field));
}

vie_status vie_tune(vie_problem* P, int precision, int* variant, void* stream) {
  if (!P || !variant || (precision != VIE_FP64 && precision != VIE_FP32 && precision != VIE_DF64)) {
    set_error("vie_tune: bad argument");
    return VIE_EINVAL;
  }
  return tune_apply(P, P->kapply, precision, variant, (cudaStream_t)stream);
}

vie_status vie_profile_begin(vie_problem* P, int cap) {
  if (!P || cap < 1 || cap > 100000) {
    set_error("vie_profile_begin: bad argument");
    return VIE_EINVAL;
  }
  Profiler& pf = P->prof;
  const size_t need = (size_t)cap * (kProfSlots + 1);
  while (pf.ev.size() < need) {
    cudaEvent_t e;
    VIE_CK(cudaEventCreate(&e));
    pf.ev.push_back(e);
  }
  pf.on = true;
  pf.cap = cap;
  pf.count = 0;
  return VIE_OK;
}

vie_status vie_profile_end(vie_problem* P, double* ms, int nslots, int* count) {
  if (!P || !ms || nslots < 0) {
    set_error("vie_profile_end: bad argument");
    return VIE_EINVAL;
  }
  Profiler& pf = P->prof;
  VIE_CK(cudaDeviceSynchronize());
  for (int k = 0; k < nslots; ++k) ms[k] = 0.0;
  for (int a = 0; a < pf.count; ++a) {
    cudaEvent_t* ev = &pf.ev[(size_t)a * (kProfSlots + 1)];
    for (int k = 0; k < kProfSlots && k < nslots; ++k) {
      float t = 0.f;
      VIE_CK(cudaEventElapsedTime(&t, ev[k], ev[k + 1]));
      ms[k] += t;
    }
  }
  if (count) *count = pf.count;
  pf.on = false;
  pf.count = 0;
  return VIE_OK;
}

vie_status vie_problem_destroy(vie_problem* P) {
  free_problem(P);
  return VIE_OK;
}

vie_status vie_release_memory(void) {
  std::vector<void*> blocks;
  {
    std::lock_guard<std::mutex> g(g_pool_mutex);
    blocks.swap(g_pinned);
  }
  for (void* p : blocks) cudaFreeHost(p);
  cudaMemPool_t pool = device_pool();
  if (pool) VIE_CK(cudaMemPoolTrimTo(pool, 0));
  return VIE_OK;
}

}  // extern "C"
