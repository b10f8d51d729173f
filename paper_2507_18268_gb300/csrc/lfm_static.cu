// Allocation-free PCG solve (lfm_pcg_solve_static in include/lapfoam.h).
//
// Some callers cannot allocate device memory: a plug-in running inside a host code whose
// memory manager owns every device buffer, or a real-time loop that must not call an
// allocator once it has started. This entry point serves them: the caller passes the LDU
// system and the solution vector in device memory it already owns, and every piece of
// working memory the solve needs lives in one file-scope device array declared below.
//
// The array is fixed at load time (every GPU that loads the library holds it until the
// process exits) and shared by all calls: each call re-initialises what must start at zero,
// and two calls whose kernels overlap on a GPU would race on it, so callers must order
// their calls (one stream, or explicit synchronisation).
//
// The solve is the same diagonal-preconditioned CG with the normFactor residual as the
// step kernels, run by a team of CTAs in one cooperative launch (lfm_device.cuh): the
// face-to-cell lists are rebuilt from owner/neighbour on every call (the owned faces by the
// jumps of the sorted owner array, the neighbour-side ones by counting + per-cell sort), then
// the CG recurrence runs with a barrier per pass. The largest systems are bound by latency: a
// pass touches at most 6 MB, all of it in L2, so it costs its dependent loads and its barrier.
// One cell per thread and as many CTAs as that needs, at most one per SM, keep both short.
// 64,000 cells, 6 iterations: 2.97 ms with one CTA of 1,024 threads (63 cells a thread, the
// lists built by one SM), 0.16 ms now.
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <mutex>

#include <cuda_runtime.h>

#include "lfm_device.cuh"
#include "lfm_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr uint64_t kTimeoutNs = 2000000000ull;  // of one barrier wait
constexpr int32_t kMaxCells = lfm::kStaticMaxCells;
constexpr int32_t kMaxFaces = lfm::kStaticMaxFaces;

// Byte layout of the scratch array.
constexpr size_t align256(size_t v) { return (v + 255) / 256 * 256; }
constexpr size_t kOffR = 0;
constexpr size_t kOffW = kOffR + align256(8 * (size_t)kMaxCells);
constexpr size_t kOffP = kOffW + align256(8 * (size_t)kMaxCells);
constexpr size_t kOffQ = kOffP + align256(8 * (size_t)kMaxCells);
constexpr size_t kOffRD = kOffQ + align256(8 * (size_t)kMaxCells);
constexpr size_t kOffOwnStart = kOffRD + align256(8 * (size_t)kMaxCells);
constexpr size_t kOffLoStart = kOffOwnStart + align256(4 * ((size_t)kMaxCells + 1));
constexpr size_t kOffLoFill = kOffLoStart + align256(4 * ((size_t)kMaxCells + 1));
constexpr size_t kOffLosort = kOffLoFill + align256(4 * (size_t)kMaxCells);
constexpr size_t kOffLoOther = kOffLosort + align256(4 * (size_t)kMaxFaces);
constexpr size_t kOffCtaSum = kOffLoOther + align256(4 * (size_t)kMaxFaces);
constexpr size_t kOffPartials = kOffCtaSum + align256(4 * (size_t)lfm::kTeamCap);
constexpr size_t kOffStats = kOffPartials + align256(2 * lfm::kMaxSums * sizeof(double) * (size_t)lfm::kTeamCap);
constexpr size_t kOffReason = kOffStats + align256(sizeof(lfm_step_stats));
constexpr size_t kOffSync = kOffReason + align256(2 * sizeof(int32_t));
constexpr size_t kScratchBytes = kOffSync + align256(sizeof(lfm::SyncWords));

// Why the kernel rejected the addressing (first int of the reason words; the second holds a
// face or cell id).
enum Reason { kBadNone = 0, kBadFace = 1, kBadOrder = 2, kBadDegree = 3 };

static __device__ __align__(256) unsigned char g_static_scratch[kScratchBytes];

struct Scratch {
  double *r, *w, *p, *q, *rD;
  int32_t *own_start, *lo_start, *lo_fill, *losort, *lo_other;
  int32_t* cta_sum;  // neighbour-side faces of each CTA's cells
  double* partials;
  lfm_step_stats* stats;
  int32_t* reason;  // [2] Reason and the offending face or cell
  lfm::SyncWords* sync;
};

__device__ __forceinline__ Scratch carve(unsigned char* base) {
  Scratch s;
  s.r = reinterpret_cast<double*>(base + kOffR);
  s.w = reinterpret_cast<double*>(base + kOffW);
  s.p = reinterpret_cast<double*>(base + kOffP);
  s.q = reinterpret_cast<double*>(base + kOffQ);
  s.rD = reinterpret_cast<double*>(base + kOffRD);
  s.own_start = reinterpret_cast<int32_t*>(base + kOffOwnStart);
  s.lo_start = reinterpret_cast<int32_t*>(base + kOffLoStart);
  s.lo_fill = reinterpret_cast<int32_t*>(base + kOffLoFill);
  s.losort = reinterpret_cast<int32_t*>(base + kOffLosort);
  s.lo_other = reinterpret_cast<int32_t*>(base + kOffLoOther);
  s.cta_sum = reinterpret_cast<int32_t*>(base + kOffCtaSum);
  s.partials = reinterpret_cast<double*>(base + kOffPartials);
  s.stats = reinterpret_cast<lfm_step_stats*>(base + kOffStats);
  s.reason = reinterpret_cast<int32_t*>(base + kOffReason);
  s.sync = reinterpret_cast<lfm::SyncWords*>(base + kOffSync);
  return s;
}

__device__ __forceinline__ bool conv_test(double res, double init_res, double tol, double rel_tol) {
  return res < tol || (rel_tol > 0.0 && res < rel_tol * init_res);
}

// Row c of A v from the per-call lists: neighbour-side faces, then owned faces.
__device__ __forceinline__ double row(const Scratch& s, int c, const int32_t* __restrict__ neighbour,
                                      const double* __restrict__ diag, const double* __restrict__ upper,
                                      const double* v) {
  double acc = diag[c] * v[c];
  for (int i = s.lo_start[c]; i < s.lo_start[c + 1]; ++i) acc = fma(upper[s.losort[i]], v[s.lo_other[i]], acc);
  for (int f = s.own_start[c]; f < s.own_start[c + 1]; ++f) acc = fma(upper[f], v[neighbour[f]], acc);
  return acc;
}

// The first reason wins; its second word is the face or cell it names.
__device__ __forceinline__ void reject(const Scratch& s, int why, int32_t id) {
  if (atomicCAS(&s.reason[0], 0, why) == 0) s.reason[1] = id;
}

__global__ void __launch_bounds__(kThreads) static_pcg_kernel(
    unsigned char* scratch, int32_t N, int32_t F, const int32_t* __restrict__ owner,
    const int32_t* __restrict__ neighbour, const double* __restrict__ diag, const double* __restrict__ upper,
    const double* __restrict__ source, double* __restrict__ x, double tol, double rel_tol, int32_t max_iter,
    int32_t min_iter) {
  using namespace lfm;
  constexpr int B = kThreads;
  __shared__ TeamShared<B> sh;
  __shared__ int32_t s_warp[B / 32], s_base;
  const Scratch s = carve(scratch);
  const Team tm{(int)gridDim.x, (int)blockIdx.x, s.sync, s.partials, kTimeoutNs};
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) team_join(tm, sh);
  int chunk = (N + tm.size - 1) / tm.size;
  chunk = (chunk + 31) & ~31;
  const int c0 = min(N, tm.rank * chunk), c1 = min(N, c0 + chunk);
  const int f_first = tm.rank * B + tid, f_step = tm.size * B;

  // ---- face-to-cell lists ---------------------------------------------------------------
  // Nothing read from owner/neighbour is used as an address before it has been checked; a
  // rejected system leaves x untouched.
  for (int f = f_first; f < F; f += f_step) {
    const int32_t o = owner[f], n = neighbour[f];
    const int bad = (o < 0 || n <= o || n >= N) ? kBadFace : (f > 0 && owner[f - 1] > o) ? kBadOrder : kBadNone;
    if (bad) reject(s, bad, f);
  }
  for (int c = c0 + tid; c < c1; c += B) s.lo_fill[c] = 0;
  if (!team_barrier<B>(tm, sh)) return;
  if (ld_volatile_i32(s.reason) != 0) {
    if (tm.rank == 0 && tid == 0) s.stats->status = LFM_EINVAL;
    return;
  }
  // own_start[c] = first face with owner >= c: the faces are sorted by owner, so each jump of
  // owner (and the two ends) sets the cells it passes
  if (F == 0) {
    for (int c = c0 + tid; c <= (c1 == N ? N : c1 - 1); c += B) s.own_start[c] = 0;
  }
  for (int f = f_first; f <= F && F > 0; f += f_step) {
    const int32_t from = f > 0 ? owner[f - 1] + 1 : 0, to = f < F ? owner[f] : N;
    for (int32_t c = from; c <= to; ++c) s.own_start[c] = f;
    if (f < F) atomicAdd(&s.lo_fill[neighbour[f]], 1);
  }
  if (!team_barrier<B>(tm, sh)) return;
  // at most kMaxSlots internal faces per cell (the limit of the context path): it bounds the
  // per-cell list sort below and every row's work
  const int per = (c1 - c0 + B - 1) / B;  // each thread scans a contiguous run of the CTA's cells
  const int a0 = min(c1, c0 + tid * per), a1 = min(c1, a0 + per);
  int run = 0;
  for (int c = a0; c < a1; ++c) {
    const int n = s.lo_fill[c];
    if (n + s.own_start[c + 1] - s.own_start[c] > kMaxSlots) reject(s, kBadDegree, c);
    run += n;
  }
  int incl = run;  // block scan of the run totals
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  int before = 0, total = 0;
  for (int k = 0; k < B / 32; ++k) {
    if (k < warp) before += s_warp[k];
    total += s_warp[k];
  }
  if (tid == 0) s.cta_sum[tm.rank] = total;
  if (!team_barrier<B>(tm, sh)) return;
  if (ld_volatile_i32(s.reason) != 0) {
    if (tm.rank == 0 && tid == 0) s.stats->status = LFM_EINVAL;
    return;
  }
  if (warp == 0) {  // the faces of the lower ranks' cells
    int t = 0;
    for (int k = lane; k < tm.rank; k += 32) t += __ldcg(s.cta_sum + k);
    t = __reduce_add_sync(0xffffffffu, t);
    if (lane == 0) s_base = t;
  }
  __syncthreads();
  int base = s_base + before + incl - run;
  for (int c = a0; c < a1; ++c) {
    s.lo_start[c] = base;
    base += s.lo_fill[c];
    s.lo_fill[c] = 0;
  }
  if (tm.rank == 0 && tid == 0) s.lo_start[N] = F;
  if (!team_barrier<B>(tm, sh)) return;
  for (int f = f_first; f < F; f += f_step) {
    const int32_t n = neighbour[f];
    s.losort[s.lo_start[n] + atomicAdd(&s.lo_fill[n], 1)] = f;
  }
  if (!team_barrier<B>(tm, sh)) return;
  // ascending face order inside each cell's short list (at most kMaxSlots entries), so every
  // run sums in the same order; the same cells' share of the sum of x
  double v1[1] = {0.0};
  for (int c = c0 + tid; c < c1; c += B) {
    const int b = s.lo_start[c], e = s.lo_start[c + 1];
    for (int i = b + 1; i < e; ++i) {
      const int32_t v = s.losort[i];
      int j = i - 1;
      while (j >= b && s.losort[j] > v) {
        s.losort[j + 1] = s.losort[j];
        --j;
      }
      s.losort[j + 1] = v;
    }
    for (int i = b; i < e; ++i) s.lo_other[i] = owner[s.losort[i]];
    v1[0] += x[c];
  }

  // ---- initial residual and normFactor (a cell's lists are its own thread's) ---------------
  if (!team_allreduce<1, B>(tm, v1, sh, [&](int, double t, int l) {
        if (l == 0) sh.xref = t / (double)N;
      }))
    return;
  const double xRef = sh.xref;
  double u[3] = {0.0, 0.0, 0.0};
  for (int c = c0 + tid; c < c1; c += B) {
    const double ax = row(s, c, neighbour, diag, upper, x);
    double rs = diag[c];
    for (int i = s.lo_start[c]; i < s.lo_start[c + 1]; ++i) rs += upper[s.losort[i]];
    for (int f = s.own_start[c]; f < s.own_start[c + 1]; ++f) rs += upper[f];
    const double b = source[c];
    const double rc = b - ax;
    const double pA = rs * xRef;
    const double rd = 1.0 / diag[c];
    u[0] += fabs(ax - pA) + fabs(b - pA);
    u[1] += fabs(rc);
    const double wc = rd * rc;
    u[2] = fma(wc, rc, u[2]);
    s.rD[c] = rd;
    s.r[c] = rc;
    s.p[c] = wc;
  }
  if (!team_allreduce<3, B>(tm, u, sh, [&](int k, double t, int l) {
        if (l == 0) sh.out[k] = t;
      }))
    return;
  if (tid == 0) {
    sh.nf = sh.out[0] + 1e-20;
    sh.init_res = sh.res = sh.out[1] / sh.nf;
    sh.rho = sh.out[2];
    sh.conv = conv_test(sh.res, sh.init_res, tol, rel_tol) ? 1 : 0;
    sh.code = min_iter > 0 || !sh.conv ? kGo : kStop;
  }
  __syncthreads();
  int iters = 0;
  while (sh.code == kGo) {
    if (iters > 0) {
      const double beta = sh.beta;
      for (int c = c0 + tid; c < c1; c += B) s.p[c] = fma(beta, s.p[c], s.w[c]);
      if (!team_barrier<B>(tm, sh)) return;
    }
    double s1[1] = {0.0};
    for (int c = c0 + tid; c < c1; c += B) {
      const double qc = row(s, c, neighbour, diag, upper, s.p);
      s.q[c] = qc;
      s1[0] = fma(qc, s.p[c], s1[0]);
    }
    if (!team_allreduce<1, B>(tm, s1, sh, [&](int, double t, int l) {
          // two quotients as one instruction sequence on two lanes
          const double q = (l == 0 ? sh.rho : fabs(t)) / (l == 0 ? t : sh.nf);
          if (l == 0) sh.alpha = q;
          if (l == 1) sh.code = q < 1e-300 ? kSingular : kGo;
        }))
      return;
    if (sh.code != kGo) break;
    const double alpha = sh.alpha;
    double s2[2] = {0.0, 0.0};
    for (int c = c0 + tid; c < c1; c += B) {
      x[c] = fma(alpha, s.p[c], x[c]);
      const double rc = fma(-alpha, s.q[c], s.r[c]);
      const double wc = s.rD[c] * rc;
      s.r[c] = rc;
      s.w[c] = wc;
      s2[0] += fabs(rc);
      s2[1] = fma(wc, rc, s2[1]);
    }
    ++iters;
    if (!team_allreduce<2, B>(tm, s2, sh, [&](int k, double t, int l) {
          if (l != 0) return;
          if (k == 0) {
            const double res = t / sh.nf;
            const bool cv = conv_test(res, sh.init_res, tol, rel_tol);
            sh.res = res;
            sh.conv = cv ? 1 : 0;
            sh.code = !isfinite(res) ? kNonFinite : ((iters < max_iter && !cv) || iters < min_iter) ? kGo : kStop;
          } else {
            sh.beta = t / sh.rho;
            sh.rho = t;
          }
        }))
      return;
  }
  if (tm.rank == 0 && tid == 0) {
    lfm_step_stats st;
    st.iters = iters;
    st.converged = sh.conv;
    st.sweeps = iters > 0 ? 1 : 0;
    st.status = sh.code == kSingular ? LFM_ESINGULAR : sh.code == kNonFinite ? LFM_ENONFINITE : 0;
    st.init_res = sh.init_res;
    st.final_res = sh.res;
    st.norm_factor = sh.nf;
    *s.stats = st;
  }
}

// Device address of the scratch array, looked up once per device (with that device
// current) on the first call made on it.
constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
unsigned char* g_scratch_ptr[kMaxDevices] = {};
int g_max_ctas[kMaxDevices] = {};  // one CTA per SM at most, co-resident

int scratch_for_current_device(unsigned char** out, int* max_ctas) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return LFM_ECUDA;
  std::lock_guard<std::mutex> lk(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    int per_sm = 0, sms = 0;
    if (e != cudaSuccess || !p ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, static_pcg_kernel, kThreads, 0) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || per_sm < 1 || sms < 1)
      return LFM_ECUDA;
    g_max_ctas[dev] = sms < lfm::kTeamCap ? sms : lfm::kTeamCap;
    g_scratch_ptr[dev] = static_cast<unsigned char*>(p);
  }
  *max_ctas = g_max_ctas[dev];
  *out = g_scratch_ptr[dev];
  return LFM_OK;
}

}  // namespace

namespace {

// Whether the byte ranges [a, a + na) and [b, b + nb) overlap.
bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return na > 0 && nb > 0 && x < y + nb && y < x + na;
}

}  // namespace

extern "C" int lfm_pcg_solve_static(int32_t n_cells, int32_t n_faces, const int32_t* owner,
                                    const int32_t* neighbour, const double* diag, const double* upper,
                                    const double* source, double* x, const lfm_solver_opts* opts,
                                    lfm_step_stats* stats, void* cuda_stream) {
  using lfm::set_last_error;
  const char* me = "lfm_pcg_solve_static";
  if (n_cells <= 0 || n_faces < 0)
    return set_last_error(LFM_EINVAL, "%s: n_cells = %d, n_faces = %d (need n_cells > 0, n_faces >= 0)", me, n_cells,
                          n_faces);
  if (n_cells > kMaxCells || n_faces > kMaxFaces)
    return set_last_error(LFM_EINVAL, "%s: %d cells, %d faces exceed the fixed limits of %d cells and %d faces", me,
                          n_cells, n_faces, kMaxCells, kMaxFaces);
  if (!diag || !source || !x || !opts || (n_faces > 0 && (!owner || !neighbour || !upper)))
    return set_last_error(LFM_EINVAL, "%s: a required pointer is NULL", me);
  if (!(opts->tol >= 0) || !(opts->rel_tol >= 0) || opts->max_iter < 1 || opts->min_iter < 0 ||
      opts->min_iter > opts->max_iter || opts->precision != LFM_FP64)
    return set_last_error(LFM_EINVAL,
                          "%s: solver options (tol %g, rel_tol %g, max_iter %d, min_iter %d, precision %d) invalid; "
                          "precision must be LFM_FP64",
                          me, opts->tol, opts->rel_tol, opts->max_iter, opts->min_iter, opts->precision);
  const size_t xb = sizeof(double) * (size_t)n_cells;
  if (overlaps(x, xb, source, xb) || overlaps(x, xb, diag, xb) ||
      overlaps(x, xb, upper, sizeof(double) * (size_t)n_faces) ||
      overlaps(x, xb, owner, sizeof(int32_t) * (size_t)n_faces) ||
      overlaps(x, xb, neighbour, sizeof(int32_t) * (size_t)n_faces))
    return set_last_error(LFM_EINVAL, "%s: x overlaps an input array (the solve is not in place)", me);
  {
    // the call reads its record back and synchronises: it can never be part of a capture
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t ce = cudaStreamIsCapturing(static_cast<cudaStream_t>(cuda_stream), &cap);
    if (ce != cudaSuccess) {
      cudaGetLastError();
      return set_last_error(LFM_ECUDA, "%s: querying the stream: %s", me, cudaGetErrorString(ce));
    }
    if (cap != cudaStreamCaptureStatusNone)
      return set_last_error(LFM_ESTATE, "%s: the stream is being captured; this call synchronises and cannot be captured",
                            me);
  }
  unsigned char* scratch = nullptr;
  int max_ctas = 0;
  if (scratch_for_current_device(&scratch, &max_ctas) != LFM_OK)
    return set_last_error(LFM_ECUDA, "%s: device address of the fixed working array not available", me);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e;
  // the status, reason and barrier words must start at zero for every call
  if ((e = cudaMemsetAsync(scratch + kOffStats, 0, kScratchBytes - kOffStats, stream)) != cudaSuccess)
    return set_last_error(LFM_ECUDA, "%s: clearing the status words: %s", me, cudaGetErrorString(e));
  int ctas = (n_cells + kThreads - 1) / kThreads;
  if (ctas > max_ctas) ctas = max_ctas;
  double tol = opts->tol, rel_tol = opts->rel_tol;
  int32_t max_iter = opts->max_iter, min_iter = opts->min_iter;
  void* args[] = {&scratch, &n_cells, &n_faces, &owner, &neighbour, &diag,     &upper,
                  &source,  &x,       &tol,     &rel_tol, &max_iter, &min_iter};
  if ((e = cudaLaunchCooperativeKernel((const void*)static_pcg_kernel, dim3(ctas), dim3(kThreads), args, 0, stream)) !=
      cudaSuccess)
    return set_last_error(LFM_ECUDA, "%s: kernel launch: %s", me, cudaGetErrorString(e));
  // record, reason and barrier words lie together: one copy brings them back
  alignas(8) unsigned char back[kScratchBytes - kOffStats];
  if ((e = cudaMemcpyAsync(back, scratch + kOffStats, sizeof back, cudaMemcpyDeviceToHost, stream)) != cudaSuccess ||
      (e = cudaStreamSynchronize(stream)) != cudaSuccess)
    return set_last_error(LFM_ECUDA, "%s: %s", me, cudaGetErrorString(e));
  lfm_step_stats st;
  int32_t reason[2];
  int32_t waited;  // a barrier wait that ran out
  std::memcpy(&st, back, sizeof st);
  std::memcpy(reason, back + (kOffReason - kOffStats), sizeof reason);
  std::memcpy(&waited, back + (kOffSync - kOffStats) + offsetof(lfm::SyncWords, status), sizeof waited);
  if (waited != 0) st.status = waited;
  if (stats) *stats = st;
  switch (st.status) {
    case LFM_OK: return LFM_OK;
    case LFM_EINVAL:
      if (reason[0] == kBadFace)
        return set_last_error(LFM_EINVAL, "%s: face %d: owner/neighbour out of range or owner >= neighbour", me,
                              reason[1]);
      if (reason[0] == kBadOrder)
        return set_last_error(LFM_EINVAL, "%s: faces not sorted by owner at face %d", me, reason[1]);
      return set_last_error(LFM_EINVAL, "%s: cell %d has more than %d internal faces", me, reason[1], lfm::kMaxSlots);
    case LFM_ESINGULAR: return set_last_error(LFM_ESINGULAR, "%s: singular system (p.Ap / normFactor < 1e-300)", me);
    case LFM_ENONFINITE: return set_last_error(LFM_ENONFINITE, "%s: non-finite residual", me);
    case LFM_ETIMEOUT: return set_last_error(LFM_ETIMEOUT, "%s: a barrier wait ran out; x holds an unfinished iterate", me);
    default: return set_last_error(st.status, "%s: solver status %d", me, st.status);
  }
}
