// Device primitives: bounded team barriers with deterministic reductions.
//
// A "team" is a set of co-resident CTAs (a cooperative launch guarantees co-residency)
// working on one case. Each barrier may carry up to kMaxSums FP64 sums: every CTA reduces its
// threads' values in a fixed order (block_sums), publishes its partial sums and arrives on a
// counter that only grows; every CTA waits for the counter itself, then adds all CTAs' partial
// sums in rank order. The result depends only on the block and team size, never on arrival
// order, so repeated runs are bitwise identical.
//
// What bounds a barrier on GB300 (304 CTAs of 512 threads): the chain release - counter -
// acquire takes 1.6 us; the rest is FP64. A scheduler's FP64 unit takes about 64 clocks per
// warp instruction (half a lane per clock), dependent or not, so a sum costs what its longest
// chain of warp-wide adds on one scheduler does, and a value computed by every thread costs
// thousands of clocks: an FP64 division by all threads of 304 x 512 takes 2.8 us, by one warp
// 0.4. Hence (i) block_sums spreads each sum over warps of four schedulers with no lane idle
// until the last tree; (ii) the scalars that follow from the totals (alpha, beta, the scaled
// residual and the stopping decision) are formed by one lane of the warp that holds the total
// (`fin`) and handed to the CTA through shared memory.
//
// Every wait is bounded: a waiter that sees too few arrivals within the launch's time limit
// (or sees another CTA's error) records an error status and the caller leaves the kernel.
#pragma once

#include <cstdint>

#include "lfm_internal.h"

namespace lfm {

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ int ld_volatile_i32(const int32_t* p) {
  return *reinterpret_cast<const volatile int32_t*>(p);
}

// ---- checked builds ----------------------------------------------------------------------
// Compiled with -DLFM_CHECKED (the library variant liblapfoam_checked.so), every index a
// kernel reads from the mesh's addressing and then uses as an address (a slot's neighbour
// cell, a face's slot positions, a boundary face) is tested against its array's extent
// first. A bad index is replaced by an in-range one (the caller's fallback), and the first
// failing site is recorded in a word of this translation unit, which the host reads after
// the launch and reports as LFM_EINVAL. Nothing reads out of bounds and nothing traps: the
// team barriers keep working and the context stays usable. In the normal build the checks
// compile to nothing. check_inject (a test hook) makes one site report as failing without
// any bad index.
enum CheckSite {
  kChkSlotCell = 1,   // a slot's neighbour cell (FP64 / FP32 passes, set-up)
  kChkFaceSlot = 2,   // face <-> slot addressing: a face's slot positions, a slot's face
  kChkBFace = 3,      // boundary addressing: a cell's boundary faces, a boundary face's cell
  kChkSlotCellDf = 4  // a slot's neighbour cell (df64 passes)
};
#ifdef LFM_CHECKED
namespace {
__device__ int g_check_site;    // first failing site, 0 while none
__device__ int g_check_inject;  // test hook: this site reports as failing
}  // namespace
__device__ __forceinline__ int checked_index(int i, int n, int fallback, int site) {
  const bool bad = (unsigned)i >= (unsigned)n;
  if (bad || g_check_inject == site) atomicCAS(&g_check_site, 0, site);
  return bad ? fallback : i;
}
#define LFM_IDX(i, n, fallback, site) ::lfm::checked_index((int)(i), (int)(n), (fallback), (site))
#else
#define LFM_IDX(i, n, fallback, site) (i)
#endif

// Launch-wide team: CTAs of a cooperative launch, meeting through global memory.
struct Team {
  int size;
  int rank;
  SyncWords* sw;
  double* partials;
  uint64_t timeout_ns;
};

constexpr int kTeamCap = kMaxCtas / 2;  // partials: two buffers (barrier parity) of kMaxSums rows

// What the iteration decides after a pass (TeamShared::code).
enum StepCode { kGo = 0, kStop = 1, kSingular = 2, kNonFinite = 3 };

// Shared scratch of a CTA in a team, and the scalars of the solve it is in: written by one
// lane inside a barrier (or by thread 0 between two __syncthreads), read by all threads.
template <int B>
struct TeamShared {
  double red[B];            // block_sums
  double out[kMaxSums];     // team totals, where a barrier has no fin of its own
  double alpha, beta, rho;  // rho: w.r of the current residual
  double nf, init_res, res; // normFactor, the solve's first and latest scaled residual
  double nf0, init0;        // those of the step's first solve
  double xref;
  double inner_tol;         // mixed form: the inner solve's tolerance
  double seed[3];           // mixed form: the next step's normFactor sum, sum|r|, rho
  float2 alpha2, beta2, xref2;  // double-float copies (hi, lo)
  float alpha32, beta32;
  int code, conv;
  int iters;                // of a solve kept on chip
  int ok;                   // 0: a wait ran out or another CTA failed
  int par;                  // parity of the next barrier
  unsigned target;          // the counter's value after the last barrier passed
  unsigned long long phase[kPhases], phase_t;
};

// Thread 0 of a CTA, when the CTA joins a team (before its first arrival): every launch starts with
// the team's words cleared, and a team runs once per launch. A CTA that joins a team whose wait has
// already run out leaves at its first barrier.
template <int B>
__device__ __forceinline__ void team_join(const Team& tm, TeamShared<B>& sh) {
  sh.target = 0;
  sh.par = 0;
  sh.ok = ld_volatile_i32(&tm.sw->status) != LFM_ETIMEOUT;
}

// Spins until *count has reached target (modulo 2^32). False (with the error recorded) when
// the time limit runs out or another CTA has recorded an error. It polls with relaxed loads and
// acquires once at the end (what the arriving CTAs wrote before their arrival is visible to this
// thread afterwards): an acquire drops the SM's L1 lines, which a CTA of the team that is still
// in its gathers on the same SM would miss at every poll.
__device__ __forceinline__ bool wait_count(unsigned* count, unsigned target, int32_t* status, uint64_t timeout_ns) {
  uint64_t t0 = 0;
  unsigned spins = 0;
  while ((int)(ld_relaxed_u32(count) - target) < 0) {
    ++spins;
    if (spins > 64) __nanosleep(20);
    if ((spins & 31u) == 0) {
      if (ld_volatile_i32(status) != 0) return (int)(ld_acquire_u32(count) - target) >= 0;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > timeout_ns) {
        atomicCAS(status, 0, (int32_t)LFM_ETIMEOUT);
        return false;
      }
    }
  }
  ld_acquire_u32(count);
  return true;
}

// Arrival at a team barrier: a release add without a return value (it orders this CTA's phase
// and partial sum before it).
__device__ __forceinline__ void arrive_release(unsigned* count) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
}

// Fixed-order sums of NS values over the CTA. The values of one sum at a time go through
// shared memory to G warps, one per scheduler, whose lanes add B / (32 G) of them each; the
// lane sums go through shared memory once more to warp k (sum k), which adds G per lane and
// then its lanes (xor tree). Returns the total of sum k in every lane of warp k < NS. Chain of
// FP64 adds at 512 threads: 3 + 3 + 5 for each sum, the sums on different schedulers. (Each
// warp folding its own lanes first took 2 to 4 adds on each of a scheduler's four warps and
// sum, and one warp then added all sums: a barrier of 304 CTAs of 512 with 0 / 1 / 2 / 4 sums
// took 2.06 / 5.25 / 8.6 / 15.0 us and takes 1.56 / 4.41 / 4.88 / 7.87.) The order depends only
// on the block size.
template <int NS, int B>
__device__ __forceinline__ double block_sums(const double* v, TeamShared<B>& sh) {
  constexpr int nw = B / 32, kRows = NS <= 1 ? 1 : NS == 2 ? 2 : 4;
  constexpr int G = nw / kRows < 4 ? nw / kRows : 4;  // warps per sum
  constexpr int kPer = B / (32 * G);                  // values per lane
  constexpr int kStride = NS == 1 ? kPer * 32 : 32;   // lane sums: NS = 1 in the warp's own range
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double q[kPer];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    if (k > 0) __syncthreads();
    sh.red[tid] = v[k];
    __syncthreads();
    if (warp / G == k) {
      const double* from = sh.red + (warp % G) * (kPer * 32) + lane;
#pragma unroll
      for (int i = 0; i < kPer; ++i) q[i] = from[32 * i];
    }
  }
  if (NS > 1) __syncthreads();
  if (warp < NS * G) {
    double t = q[0];
#pragma unroll
    for (int i = 1; i < kPer; ++i) t += q[i];
    sh.red[warp * kStride + lane] = t;
  }
  __syncthreads();
  double t = 0.0;
  if (warp < NS) {
    const double* from = sh.red + warp * G * kStride + lane;
    t = from[0];
#pragma unroll
    for (int g = 1; g < G; ++g) t += from[g * kStride];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

// Team-wide barrier carrying NS sums. fin(k, total, lane) runs in all lanes of warp k < NS with
// the team total of sum k and may write scalars of sh, which every thread may read on return.
// False: a wait ran out or another CTA failed; the caller must leave the kernel.
// Protocol: warp k stores the CTA's partial of sum k and arrives; it waits until all CTAs have
// arrived for every sum and adds the partials in rank order (lane l takes ranks l, l + 32, ...,
// all loaded first; then a fixed xor tree). The partials are double-buffered by the barrier's
// parity: a CTA can overwrite one only two barriers later, when every CTA has arrived at the
// barrier between and so has read it. (With a last arriver that adds the partials, publishes
// the totals and releases a generation word, three more L2 round trips sit in the chain:
// 2.06 us without sums against 1.60.)
template <int NS, int B, class Fin>
__device__ bool team_allreduce(const Team& tm, const double* v, TeamShared<B>& sh, Fin&& fin) {
  constexpr int kArrivals = NS > 0 ? NS : 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double tot = 0.0;
  // every thread's global writes of the phase are ordered before the arrivals below by the
  // CTA synchronisation inside block_sums, or by this one
  if constexpr (NS > 0) {
    tot = block_sums<NS, B>(v, sh);
  } else {
    __syncthreads();
  }
  if (warp < kArrivals) {
    if (tm.size > 1) {
      double* pt = tm.partials + (size_t)(sh.par * kMaxSums + warp) * kTeamCap;
      if (lane == 0) {
        if constexpr (NS > 0) __stcg(pt + tm.rank, tot);
        arrive_release(&tm.sw->count);
        if (sh.ok && !wait_count(&tm.sw->count, sh.target + (unsigned)(kArrivals * tm.size), &tm.sw->status,
                                 tm.timeout_ns))
          sh.ok = 0;
      }
      __syncwarp();
      if constexpr (NS > 0) {
        constexpr int kBatch = 10;
        tot = 0.0;
        for (int r0 = 0; r0 < tm.size; r0 += 32 * kBatch) {
          double buf[kBatch];
#pragma unroll
          for (int i = 0; i < kBatch; ++i) {
            const int r = r0 + lane + 32 * i;
            buf[i] = r < tm.size ? __ldcg(pt + r) : 0.0;
          }
#pragma unroll
          for (int i = 0; i < kBatch; ++i)
            if (r0 + 32 * i < tm.size) tot += buf[i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (tm.size > o) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        tot = __shfl_sync(0xffffffffu, tot, 0);
      }
    }
    if constexpr (NS > 0) fin(warp, tot, lane);
  }
  __syncthreads();
  if (threadIdx.x == 0 && tm.size > 1) {  // read again only after the next barrier's first synchronisation
    sh.target += (unsigned)(kArrivals * tm.size);
    sh.par ^= 1;
  }
  return sh.ok != 0;
}

// Team-wide barrier without sums.
template <int B>
__device__ __forceinline__ bool team_barrier(const Team& tm, TeamShared<B>& sh) {
  return team_allreduce<0, B>(tm, nullptr, sh, [](int, double, int) {});
}

// Slot k's neighbour distance of a packed slot word (CaseDev::slot_code), from the table at
// shared-memory address dl. The lanes of a warp mostly hold the same word, and sixteen words
// sit in different banks, so the lookup never serialises. An ordinary shared load: the batched
// kernel rewrites the table for every job, and the compiler has to see that it is read.
__device__ __forceinline__ int code_delta(uint32_t dl, uint32_t word, int k) {
  const uint32_t at = (k == 0 ? word << 2 : word >> (4 * k - 2)) & 60u;
  return *static_cast<const int32_t*>(__cvta_shared_to_generic(dl + at));
}

// ---- bulk copies global -> shared, completed on an mbarrier ------------------------------
// One thread arms a stage's mbarrier with the byte count it expects and issues the bulk
// copies (cp.async.bulk: the copy engine moves the bytes, no thread registers hold them);
// every thread then waits on the barrier's phase. Source and destination must be 16-byte
// aligned and each size a multiple of 16 bytes.
extern __shared__ __align__(128) unsigned char lfm_dyn_smem[];

namespace {
// Test hook (set by the host for one launch): this CTA issues no copy for its first staged
// tile, so that its bounded wait runs out (-1: none).
__device__ int g_skip_copy_cta = -1;
}  // namespace

__device__ __forceinline__ unsigned dyn_smem_bytes() {
  unsigned v;
  asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
  return v;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// Makes the initialised barriers visible to the copy engine (the async proxy).
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Before bulk copies of data that ordinary stores wrote earlier in the launch (a row pass's
// diagonal): a barrier orders those stores for ordinary loads only, the copy engine reads
// global memory through another proxy.
__device__ __forceinline__ void bulk_reads_fence() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// L2 policy for data read once per pass (the matrix): evicted first, so that it does not
// displace the gathered vector.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(pol)
      : "memory");
}

// Waits for the barrier's phase with the given parity. False (with LFM_ETIMEOUT recorded,
// unless another error was) when the launch's time limit runs out or another CTA has
// recorded an error.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int32_t* status, uint64_t timeout_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (unsigned spins = 1;; ++spins) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spins & 15u) == 0) {
      if (ld_volatile_i32(status) != 0) return false;
      if (global_timer_ns() - t0 > timeout_ns) {
        atomicCAS(status, 0, (int32_t)LFM_ETIMEOUT);
        return false;
      }
    }
  }
}

// Waits for the barrier's phase without regard to the launch's status (bounded by the time
// limit): the drain of copies still in flight before a CTA that failed leaves.
__device__ __forceinline__ void mbar_drain(uint64_t* bar, unsigned parity, uint64_t timeout_ns) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > timeout_ns) return;
  }
}

// Runs body over the CTA's cells [c0, c1) in tiles of TC cells whose per-cell rows arrive in
// shared memory by bulk copies, NST stages of kStage bytes at the start of the dynamic shared
// memory (their mbarriers after them). issue(stage, t0, n, bar, pol), called by thread 0
// only, arms bar with the tile's byte count and issues its copies into stage; body(stage, t0,
// nt) processes tile [t0, t0 + nt) once its copies have landed. The copy of tile t + NST is
// issued as soon as every thread is done with tile t. False when a wait ran out or another CTA
// failed (status recorded): the CTA then lets its copies in flight land (bounded) before the
// caller leaves.
template <int TC, unsigned kStage, int NST = 2, typename Issue, typename Body>
__device__ __forceinline__ bool staged_tiles(int c0, int c1, const Team& tm, Issue&& issue, Body&& body) {
  unsigned char* sm = lfm_dyn_smem;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + NST * kStage);
  const int tid = threadIdx.x;
  const int ntiles = c1 > c0 ? (c1 - c0 + TC - 1) / TC : 0;
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) mbar_init(bar + s, 1);
    mbar_init_fence();
    bulk_reads_fence();  // once per pass: nothing staged is rewritten during it
    const uint64_t pol = l2_evict_first_policy();
    for (int t = 0; t < NST && t < ntiles; ++t) {
      const int t0 = c0 + t * TC;
      if (t == 0 && (int)blockIdx.x == g_skip_copy_cta) continue;
      issue(sm + t * kStage, t0, min(TC, c1 - t0), bar + t, pol);
    }
  }
  __syncthreads();
  int t = 0, s = 0;  // tile, its stage
  unsigned par = 0;  // parity of the stage's phase
  bool failed = false;
  for (; t < ntiles; ++t) {
    const bool got = mbar_wait(bar + s, par, &tm.sw->status, tm.timeout_ns);
    const int t0 = c0 + t * TC;
    if (got) body(static_cast<const unsigned char*>(sm + s * kStage), t0, min(TC, c1 - t0));
    if (__syncthreads_or(!got)) {  // every thread is done with stage s (or one wait failed)
      failed = true;
      break;
    }
    if (tid == 0 && t + NST < ntiles) {
      const int t2 = t0 + NST * TC;
      issue(sm + s * kStage, t2, min(TC, c1 - t2), bar + s, l2_evict_first_policy());
    }
    if (++s == NST) {
      s = 0;
      par ^= 1u;
    }
  }
  if (tid == 0) {
    if (failed)
      for (int u = t; u < ntiles && u < t + NST; ++u) mbar_drain(bar + u % NST, (u / NST) & 1, tm.timeout_ns);
    for (int u = 0; u < NST; ++u) mbar_inval(bar + u);
    if (!failed && tm.rank == 0) ++tm.sw->staged;  // read back by the host (a test's evidence)
  }
  __syncthreads();
  return !failed;
}

// Records an error status for the launch (first error wins).
__device__ __forceinline__ void set_status(SyncWords* sw, int32_t code) {
  atomicCAS(&sw->status, 0, code);
}

}  // namespace lfm
