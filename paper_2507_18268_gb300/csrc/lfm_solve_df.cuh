// lfm_solve_df.cuh -- the implicit laplacianFoam step in df64 (double-float) arithmetic,
// shared by the single-case kernel (lfm_step.cu) and the batched kernel (lfm_batch.cu).
//
// The same method as the FP64 step in lfm_solve.cuh (Eq. (1), the listing "laplacianFoam
// application": per step assemble fvm::ddt(T) - fvm::laplacian(DT, T) and solve it with the
// diagonal-preconditioned CG, convergence on OpenFOAM's normFactor-scaled L1 residual), with
// every per-cell operation done in df64 on the FP32 pipe (lfm_df64.cuh) and only per-CTA
// scalars (alpha, beta, the reduced sums) in FP64. Storage is 8 bytes per value as in FP64.
//
// Set-up (a0, when the mesh, DT or dt change): the face conductances g_f = DT_f |S_f|
// deltaCoeff_f, formed in FP64, are stored per slot as df64 (g2, the face's value at its
// slot in both of its cells' rows), and V/dt per cell (vdt2). Both are multiplied by the
// case's power-of-two scale s (df_scale), chosen so that V/dt is of order one: PCG is
// invariant under scaling A and b by a common factor, a power of two scales every FP64
// and df64 value exactly, and the scaled values keep far from FP32's underflow. Reported
// normFactors are divided by s.
//
// Per launch: the field T (FP64, x) is split into a triple-float (x2 = hi, mid; xlo = lo;
// see lfm_df64.cuh) by the first pass when x was written since the last df64 launch (flags),
// and its rounding is written back to x after the last step; otherwise the triple-float field
// carries over from the previous launch, so that launch boundaries do not round the field. Fluxes and
// ddt terms are differences of field values formed exactly from the three parts, and the
// per-iteration update adds the df64 correction to all three, so rounding at df64's 2^-48 is
// relative to corrections and differences, never to T itself. (A per-step rounding of T to
// 48 bits is a noise source that truncated-CG time stepping amplifies from step to step:
// on the 200^3 graded box it grew to 7e-10 relative over 100 steps.)
// Per step (phases separated by team barriers):
//   S  the last solve's correction added to the field; sum of x (for xRef); with correctors
//      also x at the start of the step
//   R  per row: diag = sum of the slot conductances (slot order) + boundary + V/dt, the
//      source, 1/diag (FP32 reciprocal + one df64 Newton step), the row sum; r = b - A x
//      (in flux form, see pass_rows_init_df), normFactor terms, sum|r|, w = rD r, rho; p = w
//   loop: P p = w + beta p; M q = A p, p.q; U e += alpha p, r -= alpha q, w = rD r, sum|r|, w.r
//   (e: the solve's correction to the field, df64)
// A row of A v is diag_c v_c - sum_k g_ck v_other(k): the off-diagonal coefficient of face f
// is -g_f in both rows (the matrix is symmetric), so the slot array of conductances is the
// matrix's off-diagonal part.
//
// Boundary faces (a few per cent of cells) are summed in FP64 and converted once per row;
// so are the optional volumetric sources. On general (non-orthogonal) geometry (kGeom) a
// phase G after S forms the Gauss gradient of the field and R adds the explicit correction.
// The mixed form's df64 outer passes are in lfm_solve_mixed_df.cuh.
#pragma once

#include <cuda_runtime.h>

#include "lfm_device.cuh"
#include "lfm_df64.cuh"
#include "lfm_internal.h"
#include "lfm_solve.cuh"

namespace lfm {
namespace {

__device__ __forceinline__ float2 pair_of(double v) {
  const df d = df_from_double(v);
  return make_float2(d.hi, d.lo);
}
__device__ __forceinline__ df df_of(float2 v) { return mkdf(v.x, v.y); }

// The team mean of the field as a pair (xRef), formed in the barrier that carries its sum.
template <int B>
__device__ __forceinline__ void fin_mean_df(TeamShared<B>& sh, const CaseDev& cs, double t, int lane) {
  if (lane == 0) sh.xref2 = pair_of(t / (double)cs.N);
}

// S: this thread's sum of x over [c0, c1) (per-thread df64 sum, converted once). `convert`:
// first pass of the launch, the triple-float field is split from the FP64 field x. `fold`:
// the previous solve's correction e (df64, see pass_update_df) is added to the field first.
// `save_old`: keep x as the step's starting field (the ddt source of the corrector passes).
template <int B>
__device__ __noinline__ double pass_sum_df(const CaseDev& cs, int c0, int c1, bool convert, bool fold,
                                           bool save_old) {
  float2* __restrict__ x2 = cs.x2;
  float* __restrict__ xl = cs.xlo;
  const float2* __restrict__ e2 = cs.e2;
  DfAcc acc;
  int c = c0 + (int)threadIdx.x;
  if (!convert && !save_old) {  // two cells per trip, loads first
    for (; c + B < c1; c += 2 * B) {
      tf a = ld_tf(x2, xl, c), b = ld_tf(x2, xl, c + B);
      if (fold) {
        const df ea = ld_df(e2 + c), eb = ld_df(e2 + c + B);
        a = tf_add_df(a, ea);
        b = tf_add_df(b, eb);
        st_tf(x2, xl, c, a);
        st_tf(x2, xl, c + B, b);
      }
      acc.add(tf_to_df(a));
      acc.add(tf_to_df(b));
    }
  }
  for (; c < c1; c += B) {
    tf v;
    if (convert) {
      v = tf_from_double(cs.x[c]);
      st_tf(x2, xl, c, v);
    } else {
      v = ld_tf(x2, xl, c);
      if (fold) {
        v = tf_add_df(v, ld_df(e2 + c));
        st_tf(x2, xl, c, v);
      }
    }
    if (save_old) st_tf(reinterpret_cast<float2*>(cs.x_old), cs.xolo, c, v);
    acc.add(tf_to_df(v));
  }
  return acc.value();
}

// After the first barrier of a launch that split the FP64 field: every CTA has read the flag,
// so the team's rank 0 marks the triple-float field current (it persists across launches:
// the FP64 field is only its rounding, rewritten at the end of every launch).
__device__ __forceinline__ void mark_split(const CaseDev& cs, const Team& tm, bool& convert) {
  if (convert && tm.rank == 0 && threadIdx.x == 0) *reinterpret_cast<volatile int32_t*>(cs.flags) = 1;
  convert = false;
}

// The FP64 field from the triple-float one (end of the launch; each CTA its own cells), with
// the last solve's correction added to the triple-float field first when it is not yet.
template <int B>
__device__ __noinline__ void pass_store_x(const CaseDev& cs, int c0, int c1, bool fold) {
  float2* __restrict__ x2 = cs.x2;
  float* __restrict__ xl = cs.xlo;
  double* __restrict__ x = cs.x;
  for (int c = c0 + (int)threadIdx.x; c < c1; c += B) {
    tf v = ld_tf(x2, xl, c);
    if (fold) {  // the triple-float field carries over to the next launch: keep it current
      v = tf_add_df(v, ld_df(cs.e2 + c));
      st_tf(x2, xl, c, v);
    }
    x[c] = tf_to_double(v);
  }
}

// Boundary conductance, source and flux g_b (T_b - x_c) of row c (fixedValue faces; zeroGradient
// adds nothing), in FP64 with the case scale, in ascending face order. The first two do not depend
// on the field and come as pairs from set-up; the flux is formed here, two FP64 operations per
// face beside the conversions (a third of a box's warps hold a boundary cell, and each spent some 25
// warp instructions of 64 clocks on the three sums).
__device__ __forceinline__ void row_boundary_df(const CaseDev& cs, int c, tf xc, df& gsum, df& ssum, df& flux,
                                                uint32_t word = 0xffffffffu) {
  gsum = mkdf(0.0f, 0.0f);
  ssum = mkdf(0.0f, 0.0f);
  flux = mkdf(0.0f, 0.0f);
  if (!(word >> 31)) return;  // the slot code says whether there are any (all ones when not coded)
  const int b0 = __ldg(cs.b_start + c), b1 = __ldg(cs.b_start + c + 1);
  if (b0 == b1) return;
  const float4 sums = __ldg(cs.bsum2 + b0);
  if (sums.x == 0.0f) return;  // no fixedValue face (or no conductance)
  gsum = mkdf(sums.x, sums.y);
  ssum = mkdf(sums.z, sums.w);
  const double x = tf_to_double(xc);
  double fl = 0.0;
  for (int k = b0; k < b1; ++k) {
    const double gb = __ldg(cs.bg + k) * cs.df_scale;  // a power of two: exact
    if (__double_as_longlong(gb) != 0) fl += gb * (__ldg(cs.bT + k) - x);
  }
  flux = df_from_double(fl);
}

// ---- general geometry ----------------------------------------------------------------
// G: the Gauss linear gradient of the field over [c0, c1) into grad2, in difference form
//   G_c = sum_k gE_k (T_k - T_c) + sum_fixedValue (bSf / V)(T_b - T_c) + gZ T_c
// (equal to the operator form gD T_c + gH + sum_k gE_k T_k; see CaseDev): a weighted sum of
// T values that nearly cancel would carry their rounding, ~2^-48 |T| / h, into the explicit
// correction; differences formed exactly from the triple-float field do not. The boundary
// terms (boundary cells only) are FP64; gZ T_c (gZ is zero up to the geometry's rounding) df64.
template <int B, int W>
__device__ __noinline__ void pass_grad_df(const CaseDev& cs, int c0, int c1) {
  const float2* __restrict__ x2 = cs.x2;
  const float* __restrict__ xl = cs.xlo;
  const size_t N = (size_t)cs.N;
  const int ns = nslots<W>(cs);
  const size_t WN = (size_t)ns * N;
  for (int c = c0 + (int)threadIdx.x; c < c1; c += B) {
    const tf xc = ld_tf(x2, xl, c);
    df g0 = mkdf(0.0f, 0.0f), g1 = g0, g2 = g0;
    int o[W > 0 ? kSlots<W> : 1];
    if constexpr (W > 0) neighbours<W, false>(cs.slot_other, cs.slot_code, cs.N, delta_table<W>(cs), c, o, kChkSlotCellDf);
#pragma unroll
    for (int k = 0; k < (W > 0 ? kSlots<W> : kMaxSlots); ++k) {
      if (W == 0 && k >= ns) break;
      const size_t at = (size_t)k * N + c;
      const int oc = W > 0 ? o[W > 0 ? k : 0] : LFM_IDX(__ldg(cs.slot_other + at), cs.N, c, kChkSlotCellDf);
      const df d = tf_diff(ld_tf(x2, xl, oc), xc);
      g0 = df_fma(ldg_df(cs.gE2 + at), d, g0);
      g1 = df_fma(ldg_df(cs.gE2 + WN + at), d, g1);
      g2 = df_fma(ldg_df(cs.gE2 + 2 * WN + at), d, g2);
    }
    const df xcd = tf_to_df(xc);
    g0 = df_fma(ldg_df(cs.gZ + c), xcd, g0);
    g1 = df_fma(ldg_df(cs.gZ + N + c), xcd, g1);
    g2 = df_fma(ldg_df(cs.gZ + 2 * N + c), xcd, g2);
    const int k0 = __ldg(cs.b_start + c), k1 = __ldg(cs.b_start + c + 1);
    if (k0 != k1) {  // boundary cells: the fixedValue faces' terms in FP64
      const double xd = tf_to_double(xc), rv = 1.0 / cs.V[c];
      double b0 = 0.0, b1 = 0.0, b2 = 0.0;
      for (int k = k0; k < k1; ++k) {
        const int bf = LFM_IDX(__ldg(cs.b_face + k), cs.NB, 0, kChkBFace);
        if (__ldg(cs.btype + bf) == LFM_FIXED_VALUE) {
          const double dT = (__ldg(cs.bval + bf) - xd) * rv;
          b0 = fma(cs.bSf[3 * (size_t)bf], dT, b0);
          b1 = fma(cs.bSf[3 * (size_t)bf + 1], dT, b1);
          b2 = fma(cs.bSf[3 * (size_t)bf + 2], dT, b2);
        }
      }
      g0 = df_add(g0, df_from_double(b0));
      g1 = df_add(g1, df_from_double(b1));
      g2 = df_add(g2, df_from_double(b2));
    }
    st_df(cs.grad2 + c, g0);
    st_df(cs.grad2 + N + c, g1);
    st_df(cs.grad2 + 2 * N + c, g2);
  }
}

// The explicit non-orthogonal correction of row c (scaled with the system): the sum over the
// cell's faces of the correction flux, through the weights cK, cL of the gradient.
template <int W>
__device__ __forceinline__ df op_corr_df(const CaseDev& cs, int c) {
  const size_t N = (size_t)cs.N;
  const int ns = nslots<W>(cs);
  const size_t WN = (size_t)ns * N;
  int oc[W > 0 ? kSlots<W> : 1];
  if constexpr (W > 0) neighbours<W, false>(cs.slot_other, cs.slot_code, cs.N, delta_table<W>(cs), c, oc, kChkSlotCellDf);
  const float2* __restrict__ G = cs.grad2;
  df v = df_mul(ldg_df(cs.cK2 + c), ld_df(G + c));
  v = df_fma(ldg_df(cs.cK2 + N + c), ld_df(G + N + c), v);
  v = df_fma(ldg_df(cs.cK2 + 2 * N + c), ld_df(G + 2 * N + c), v);
#pragma unroll
  for (int k = 0; k < (W > 0 ? kSlots<W> : kMaxSlots); ++k) {
    if (W == 0 && k >= ns) break;
    const size_t at = (size_t)k * N + c;
    const int o = W > 0 ? oc[W > 0 ? k : 0] : LFM_IDX(__ldg(cs.slot_other + at), cs.N, c, kChkSlotCellDf);
    v = df_fma(ldg_df(cs.cL2 + at), ld_df(G + o), v);
    v = df_fma(ldg_df(cs.cL2 + WN + at), ld_df(G + N + o), v);
    v = df_fma(ldg_df(cs.cL2 + 2 * WN + at), ld_df(G + 2 * N + o), v);
  }
  return v;
}

// sum_k g_k (x_other(k) - x_c) over the gathered neighbours of a row, in slot order. Neighbouring
// field values are nearly always within a factor of two, so the row takes the shorter exact
// difference unless one is not (a quarter of the instructions of the row passes, which issue
// 640 per row, are these differences).
template <int S>
__device__ __forceinline__ df flux_sum_df(const df (&g)[S], const tf (&xo)[S], tf xc) {
  const float lim = tf_near_limit(xc);
  bool near = true;
#pragma unroll
  for (int k = 0; k < S; ++k) near = near && tf_near(xo[k], xc, lim);
  df flux;
  if (near) {
    flux = df_mul(g[0], tf_diff_near(xo[0], xc));
#pragma unroll
    for (int k = 1; k < S; ++k) flux = df_fma(g[k], tf_diff_near(xo[k], xc), flux);
  } else {
    flux = df_mul(g[0], tf_diff(xo[0], xc));
#pragma unroll
    for (int k = 1; k < S; ++k) flux = df_fma(g[k], tf_diff(xo[k], xc), flux);
  }
  return flux;
}

// a - b for two values of one cell's field, by the shorter form where it is exact.
__device__ __forceinline__ df tf_diff_any(tf a, tf b) {
  return tf_near(a, b, tf_near_limit(b)) ? tf_diff_near(a, b) : tf_diff(a, b);
}

// L2 prefetch of what a row pass loads for row c before its gathers: the slot word or indices and
// conductances, the field value and V/dt. Issued one trip ahead (c + B), it shortens the
// dependent chain index -> neighbour value of the next row (row pass 0.32 -> 0.30 ms per
// step on the 200^3 graded box; one bulk prefetch of the tile per array and CTA instead was slower,
// 258 against 221 us for 8 M rows of the verification pass, none at all 235).
template <int W>
__device__ __forceinline__ void prefetch_row_df(const CaseDev& cs, int c) {
  const size_t N = (size_t)cs.N;
  const int ns = nslots<W>(cs);
  if (kCoded<W>) prefetch_l2(cs.slot_code + c);
  for (int k = 0; k < (W > 0 ? kSlots<W> : kMaxSlots); ++k) {
    if (W == 0 && k >= ns) break;
    if (!kCoded<W>) prefetch_l2(cs.slot_other + (size_t)k * N + c);
    prefetch_l2(cs.g2 + (size_t)k * N + c);
  }
  prefetch_l2(cs.x2 + c);
  prefetch_l2(cs.xlo + c);
  prefetch_l2(cs.vdt2 + c);
}

// R: rows of the matrix and, from the same loaded row, the initial residual, normFactor
// terms, sum|r| and rho; p = w. kSrc: correctors (ddt source from x_old) or volumetric
// sources present.
// The residual is evaluated in flux form,
//   r_c = sum_k g_k (x_other(k) - x_c) + sum_b g_b (T_b - x_c) + V/dt (x_old,c - x_c)
//         + V Su_c + V Sp_c x_c,
// which equals b - A x term by term. Formed as b - A x, r would be the small difference of
// two values of order V/dt T and carry their rounding error, ~2^-48 |b|, amplified by
// |b| / |r| (about 1e6 for a time step that changes T by one part in a million); the
// differences of nearby values here are almost exact, so r keeps the format's relative
// accuracy. A x for the normFactor terms is then b - r.
// kRows: the diagonal and its reciprocal are formed (the first pass of a launch); false: the
// reciprocal is read back, the diagonal is not needed.
template <int B, int W, bool kSrc, bool kRows>
__device__ __noinline__ Sums3 pass_rows_init_df(const CaseDev& cs, int c0, int c1, df xr) {
  const float2* __restrict__ x2 = cs.x2;
  const float* __restrict__ xl = cs.xlo;
  const float2* __restrict__ g2 = cs.g2;
  float2* __restrict__ r2 = reinterpret_cast<float2*>(cs.r);
  float2* __restrict__ p2 = reinterpret_cast<float2*>(cs.p);
  const size_t N = (size_t)cs.N;
  DfAcc a_nf, a_r, a_rho;
  for (int c = c0 + (int)threadIdx.x; c < c1; c += B) {
    if (c + B < c1) prefetch_row_df<W>(cs, c + B);
    const tf xc = ld_tf(x2, xl, c);
    df d, flux;
    uint32_t word = 0xffffffffu;
    if constexpr (W > 0) {
      constexpr int S = kSlots<W>;
      int o[S];
      df g[S];
      word = neighbours<W, false>(cs.slot_other, cs.slot_code, cs.N, delta_table<W>(cs), c, o, kChkSlotCellDf);
#pragma unroll
      for (int k = 0; k < S; ++k) g[k] = ldg_df(g2 + (size_t)k * N + c);
      tf xo_[S];
#pragma unroll
      for (int k = 0; k < S; ++k) xo_[k] = ld_tf(x2, xl, o[k]);
      if constexpr (kRows) {
        d = g[0];
#pragma unroll
        for (int k = 1; k < S; ++k) d = df_add(d, g[k]);  // padding slots hold 0
      }
      flux = flux_sum_df<S>(g, xo_, xc);
    } else {
      d = mkdf(0.0f, 0.0f);
      flux = mkdf(0.0f, 0.0f);
      for (int k = 0; k < cs.W; ++k) {
        const size_t at = (size_t)k * N + c;
        const df gk = ldg_df(g2 + at);
        if constexpr (kRows) d = df_add(d, gk);
        flux = df_fma(gk, tf_diff(ld_tf(x2, xl, LFM_IDX(__ldg(cs.slot_other + at), cs.N, c, kChkSlotCellDf)), xc), flux);
      }
    }
    df gb, sb, fb;
    row_boundary_df(cs, c, xc, gb, sb, fb, word);
    const df vdt = ldg_df(cs.vdt2 + c);
    const df xcd = tf_to_df(xc);
    const bool has_old = kSrc && cs.n_corr > 0;
    const tf xo = has_old ? ld_tf(reinterpret_cast<const float2*>(cs.x_old), cs.xolo, c) : xc;
    if constexpr (kRows) d = df_add(df_add(d, gb), vdt);
    df src = df_fma(vdt, has_old ? tf_to_df(xo) : xcd, sb);
    df sa = df_add(vdt, gb);
    df rc = df_add(flux, fb);
    if (has_old) rc = df_fma(vdt, tf_diff_any(xo, xc), rc);
    if (kSrc && (cs.vSp || cs.vSu)) {
      // the volumetric source V Su + V Sp T of the row's residual, in FP64 (proportional to T)
      const double sp = cs.vSp ? cs.vSp[c] * cs.df_scale : 0.0;
      const double su = cs.vSu ? cs.vSu[c] * cs.df_scale : 0.0;
      const df vsp = df_from_double(sp);
      if constexpr (kRows) d = df_sub(d, vsp);
      sa = df_sub(sa, vsp);
      src = df_add(src, df_from_double(su));
      rc = df_add(rc, df_from_double(fma(sp, tf_to_double(xc), su)));
    }
    if (kSrc && cs.Sf) {  // the explicit non-orthogonal correction joins the source
      const df corr = op_corr_df<W>(cs, c);
      src = df_add(src, corr);
      rc = df_add(rc, corr);
    }
    const df ax = df_sub(src, rc);
    const df rd = kRows ? df_rcp(d) : ld_df(cs.rD2 + c);
    const df sx = df_mul(sa, xr);
    a_nf.add(df_abs(df_sub(ax, sx)));
    a_nf.add(df_abs(df_sub(src, sx)));
    a_r.add(df_abs(rc));
    const df wc = df_mul(rd, rc);
    a_rho.add(df_mul(wc, rc));
    if constexpr (kRows) {
      st_df(cs.diag2 + c, d);
      st_df(cs.rD2 + c, rd);
    }
    st_df(r2 + c, rc);
    st_df(p2 + c, wc);
  }
  return Sums3{a_nf.value(), a_r.value(), a_rho.value()};
}

// Rows c and c2 of A v, all loads of both rows issued before any is used; the matrix arrays
// with evict-first (streaming) loads, so that they do not displace the gathered vector.
template <int W>
__device__ __forceinline__ void rows2_df(const CaseDev& cs, uint32_t dl, int c, int c2,
                                         const float2* __restrict__ v, df& y, df& y2, df& vc, df& vc2) {
  const size_t N = (size_t)cs.N;
  const float2* __restrict__ g2 = cs.g2;
  vc = ld_df(v + c);
  vc2 = ld_df(v + c2);
  const float2 dd1 = __ldcs(cs.diag2 + c), dd2 = __ldcs(cs.diag2 + c2);
  df acc = df_mul(df{dd1.x, dd1.y}, vc), acc2 = df_mul(df{dd2.x, dd2.y}, vc2);
  if constexpr (kCoded<W>) {
    constexpr int S = kSlots<W>;
    int o[S], o2[S];
    df g[S], h[S];
    neighbours<W, true>(cs.slot_other, cs.slot_code, cs.N, dl, c, o, kChkSlotCellDf);
    neighbours<W, true>(cs.slot_other, cs.slot_code, cs.N, dl, c2, o2, kChkSlotCellDf);
#pragma unroll
    for (int k = 0; k < S; ++k) {
      const float2 a = __ldcs(g2 + (size_t)k * N + c), b = __ldcs(g2 + (size_t)k * N + c2);
      g[k] = df{a.x, a.y};
      h[k] = df{b.x, b.y};
    }
    df xo[S], xo2[S];
#pragma unroll
    for (int k = 0; k < S; ++k) xo[k] = ld_df(v + o[k]);
#pragma unroll
    for (int k = 0; k < S; ++k) xo2[k] = ld_df(v + o2[k]);
#pragma unroll
    for (int k = 0; k < S; ++k) acc = df_fma(df_neg(g[k]), xo[k], acc);
#pragma unroll
    for (int k = 0; k < S; ++k) acc2 = df_fma(df_neg(h[k]), xo2[k], acc2);
  } else if constexpr (W > 0) {
    int o[W], o2[W];
    df g[W], h[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
      o[k] = LFM_IDX(__ldcs(cs.slot_other + (size_t)k * N + c), cs.N, c, kChkSlotCellDf);
      o2[k] = LFM_IDX(__ldcs(cs.slot_other + (size_t)k * N + c2), cs.N, c2, kChkSlotCellDf);
      const float2 a = __ldcs(g2 + (size_t)k * N + c), b = __ldcs(g2 + (size_t)k * N + c2);
      g[k] = df{a.x, a.y};
      h[k] = df{b.x, b.y};
    }
    df xo[W], xo2[W];
#pragma unroll
    for (int k = 0; k < W; ++k) xo[k] = ld_df(v + o[k]);
#pragma unroll
    for (int k = 0; k < W; ++k) xo2[k] = ld_df(v + o2[k]);
#pragma unroll
    for (int k = 0; k < W; ++k) acc = df_fma(df_neg(g[k]), xo[k], acc);
#pragma unroll
    for (int k = 0; k < W; ++k) acc2 = df_fma(df_neg(h[k]), xo2[k], acc2);
  } else {
    for (int k = 0; k < cs.W; ++k) {
      const size_t at = (size_t)k * N;
      acc = df_fma(df_neg(ldg_df(g2 + at + c)), ld_df(v + LFM_IDX(__ldg(cs.slot_other + at + c), cs.N, c, kChkSlotCellDf)), acc);
      acc2 = df_fma(df_neg(ldg_df(g2 + at + c2)), ld_df(v + LFM_IDX(__ldg(cs.slot_other + at + c2), cs.N, c2, kChkSlotCellDf)), acc2);
    }
  }
  y = acc;
  y2 = acc2;
}

template <int W>
__device__ __forceinline__ df row1_df(const CaseDev& cs, uint32_t dl, int c, const float2* __restrict__ v, df& vc) {
  const size_t N = (size_t)cs.N;
  vc = ld_df(v + c);
  df acc = df_mul(ld_df(cs.diag2 + c), vc);
  if constexpr (W > 0) {
    int o[kSlots<W>];
    neighbours<W, false>(cs.slot_other, cs.slot_code, cs.N, dl, c, o, kChkSlotCellDf);
#pragma unroll
    for (int k = 0; k < kSlots<W>; ++k)
      acc = df_fma(df_neg(ldg_df(cs.g2 + (size_t)k * N + c)), ld_df(v + o[k]), acc);
  } else {
    for (int k = 0; k < cs.W; ++k) {
      const size_t at = (size_t)k * N + c;
      acc = df_fma(df_neg(ldg_df(cs.g2 + at)), ld_df(v + LFM_IDX(__ldg(cs.slot_other + at), cs.N, c, kChkSlotCellDf)), acc);
    }
  }
  return acc;
}

// P: p = w + beta p.
template <int B>
__device__ __forceinline__ void pass_direction_df(int c0, int c1, df beta, float2* __restrict__ p,
                                                  const float2* __restrict__ w) {
  int c = c0 + (int)threadIdx.x;
  for (; c + B < c1; c += 2 * B) {
    pf_next<B>(p, c, c1);
    pf_next<B>(w, c, c1);
    const df p1 = ld_df(p + c), p2 = ld_df(p + c + B), w1 = ld_df(w + c), w2 = ld_df(w + c + B);
    st_df(p + c, df_fma(beta, p1, w1));
    st_df(p + c + B, df_fma(beta, p2, w2));
  }
  if (c < c1) st_df(p + c, df_fma(beta, ld_df(p + c), ld_df(w + c)));
}

// P from CaseDev::late_cells / 2 cells on: e += alpha p, the correction's update with the last
// direction, and p = w + beta p; backwards, as pass_direction_x (lfm_solve.cuh). It starts with
// e = alpha p (first). Per iteration of 8 M cells, P and U with the update in U: 31 + 78 us, here
// 47 + 50; the call 10.89 -> 10.57 ms.
template <int B>
__device__ __forceinline__ void pass_direction_x_df(int c0, int c1, df alpha, df beta, float2* __restrict__ e, bool first,
                                                  float2* __restrict__ p, const float2* __restrict__ w) {
  int c = c0 + (int)threadIdx.x;
  if (c >= c1) return;
  c += (c1 - 1 - c) / B * B;  // the thread's last row
  auto step_e = [&](int i, df pi) { st_df(e + i, first ? df_mul(alpha, pi) : df_fma(alpha, pi, ld_df(e + i))); };
  for (; c >= c0 + B; c -= 2 * B) {
    const int d = c - B;
    pf_back<B>(p, c, c0);
    pf_back<B>(w, c, c0);
    if (!first) pf_back<B>(e, c, c0);
    const df p1 = ld_df(p + c), p2 = ld_df(p + d), w1 = ld_df(w + c), w2 = ld_df(w + d);
    if (first) {
      st_df(e + c, df_mul(alpha, p1));
      st_df(e + d, df_mul(alpha, p2));
    } else {
      const df e1 = ld_df(e + c), e2 = ld_df(e + d);
      st_df(e + c, df_fma(alpha, p1, e1));
      st_df(e + d, df_fma(alpha, p2, e2));
    }
    st_df(p + c, df_fma(beta, p1, w1));
    st_df(p + d, df_fma(beta, p2, w2));
  }
  if (c >= c0) {
    const df pc = ld_df(p + c);
    step_e(c, pc);
    st_df(p + c, df_fma(beta, pc, ld_df(w + c)));
  }
}

// The correction's last update, after the iteration that ended the solve.
template <int B>
__device__ __forceinline__ void pass_solution_df(int c0, int c1, df alpha, float2* __restrict__ e, bool first,
                                                 const float2* __restrict__ p) {
  int c = c0 + (int)threadIdx.x;
  for (; c + B < c1; c += 2 * B) {
    pf_next<B>(p, c, c1);
    if (!first) pf_next<B>(e, c, c1);
    const df p1 = ld_df(p + c), p2 = ld_df(p + c + B);
    if (first) {
      st_df(e + c, df_mul(alpha, p1));
      st_df(e + c + B, df_mul(alpha, p2));
    } else {
      const df e1 = ld_df(e + c), e2 = ld_df(e + c + B);
      st_df(e + c, df_fma(alpha, p1, e1));
      st_df(e + c + B, df_fma(alpha, p2, e2));
    }
  }
  if (c < c1) {
    const df pc = ld_df(p + c);
    st_df(e + c, first ? df_mul(alpha, pc) : df_fma(alpha, pc, ld_df(e + c)));
  }
}

// M: q = A p; returns this thread's share of p.q.
template <int B, int W>
__device__ __forceinline__ double pass_amul_dot_df(const CaseDev& cs, uint32_t dl, int c0, int c1, const float2* __restrict__ p,
                                                   float2* __restrict__ q) {
  DfAcc s;
  int c = c0 + (int)threadIdx.x;
  for (; c + B < c1; c += 2 * B) {
    df y1, y2, pc1, pc2;
    rows2_df<W>(cs, dl, c, c + B, p, y1, y2, pc1, pc2);
    st_df(q + c, y1);
    st_df(q + c + B, y2);
    s.add(df_mul(y1, pc1));
    s.add(df_mul(y2, pc2));
  }
  if (c < c1) {
    df pc;
    const df y = row1_df<W>(cs, dl, c, p, pc);
    st_df(q + c, y);
    s.add(df_mul(y, pc));
  }
  return s.value();
}

// M with the matrix rows streamed into shared memory by bulk copies, as the FP32 A p
// (pass_amul_dot_f32_bulk, lfm_solve.cuh): for packed meshes, one row per thread and tile (60
// bytes per cell), three stages. The same cells per thread in the same order and the same
// operations as the register form: equal results bit for bit. Needs N a multiple of 4 and the
// dynamic shared memory of stage_bytes_df; ok = false when a wait ran out (status recorded).
constexpr int kDfStages = 3;
template <int W>
__host__ __device__ constexpr unsigned stage_row_df() {  // bytes per cell: the code word, conductances, diagonal
  return 4u + 8u * kSlots<W> + 8u;
}
template <int B, int W>
__host__ __device__ constexpr unsigned stage_bytes_df() {
  return kCoded<W> ? kDfStages * (B * stage_row_df<W>()) + 8u * kDfStages : 0u;
}

template <int B, int W>
__device__ __noinline__ double pass_amul_dot_df_bulk(const CaseDev& cs, int c0, int c1, const float2* __restrict__ p,
                                                     float2* __restrict__ q, const Team& tm, bool& ok) {
  constexpr int S = kSlots<W>;
  constexpr unsigned kStage = B * stage_row_df<W>();
  const size_t N = (size_t)cs.N;
  const uint32_t dl = delta_table<W>(cs);
  const int tid = threadIdx.x;
  DfAcc acc;
  auto issue = [&](unsigned char* st, int t0, int n, uint64_t* bar, uint64_t pol) {
    mbar_arrive_expect_tx(bar, (unsigned)n * stage_row_df<W>());
#pragma unroll
    for (int k = 0; k < S; ++k) bulk_g2s(st + 8u * B * k, cs.g2 + (size_t)k * N + t0, 8u * n, bar, pol);
    bulk_g2s(st + 8u * B * S, cs.diag2 + t0, 8u * n, bar, pol);
    bulk_g2s(st + 8u * B * (S + 1), cs.slot_code + t0, 4u * n, bar, pol);
  };
  auto body = [&](const unsigned char* st, int t0, int nt) {
    if (tid >= nt) return;
    const float2* sg = reinterpret_cast<const float2*>(st);
    const uint32_t word = reinterpret_cast<const uint32_t*>(st + 8u * B * (S + 1))[tid];
    const int c = t0 + tid;
    df x[S];
#pragma unroll
    for (int k = 0; k < S; ++k) x[k] = ld_df(p + LFM_IDX(c + code_delta(dl, word, k), cs.N, c, kChkSlotCellDf));
    const df pc = ld_df(p + c);
    df y = df_mul(ld_df(sg + B * S + tid), pc);
#pragma unroll
    for (int k = 0; k < S; ++k) y = df_fma(df_neg(ld_df(sg + B * k + tid)), x[k], y);
    st_df(q + c, y);
    acc.add(df_mul(y, pc));
  };
  ok = staged_tiles<B, kStage, kDfStages>(c0, c1, tm, issue, body);
  return acc.value();
}

template <int B, int W>
__device__ __forceinline__ double amul_dot_df(const CaseDev& cs, const CaseDev& cref, int c0, int c1,
                                              const float2* __restrict__ p, float2* __restrict__ q, const Team& tm,
                                              bool& ok) {
  ok = true;
  if constexpr (kCoded<W>) {
    if ((cs.N & 3) == 0 && dyn_smem_bytes() >= stage_bytes_df<B, W>())
      return pass_amul_dot_df_bulk<B, W>(cref, c0, c1, p, q, tm, ok);
  }
  return pass_amul_dot_df<B, W>(cs, delta_table<W>(cref), c0, c1, p, q);
}

// U: e += alpha p (first iteration of a solve: e = alpha p), r -= alpha q, w = rD r; returns
// this thread's sum|r| and w.r. e, the solve's correction to the field, is added to the
// triple-float field once per solve (pass_sum_df, pass_store_x), so an iteration moves 8
// bytes of field state per cell instead of reading and writing the field's 12.
template <int B>
__device__ __forceinline__ double2 pass_update_df(int c0, int c1, df alpha, float2* __restrict__ e, bool first,
                                                  float2* __restrict__ r, float2* __restrict__ w,
                                                  const float2* __restrict__ p, const float2* __restrict__ q,
                                                  const float2* __restrict__ rD) {
  DfAcc sa, sr;
  const df nalpha = df_neg(alpha);
  int c = c0 + (int)threadIdx.x;
  for (; c + B < c1; c += 2 * B) {
    const int k = c + B;
    const df pa = ld_df(p + c), pb = ld_df(p + k), qa = ld_df(q + c), qb = ld_df(q + k);
    const df ra = ld_df(r + c), rb = ld_df(r + k);
    const df da = ld_df(rD + c), db = ld_df(rD + k);
    const df rna = df_fma(nalpha, qa, ra), rnb = df_fma(nalpha, qb, rb);
    const df wa = df_mul(da, rna), wb = df_mul(db, rnb);
    if (first) {
      st_df(e + c, df_mul(alpha, pa));
      st_df(e + k, df_mul(alpha, pb));
    } else {
      const df ea = ld_df(e + c), eb = ld_df(e + k);
      st_df(e + c, df_fma(alpha, pa, ea));
      st_df(e + k, df_fma(alpha, pb, eb));
    }
    st_df(r + c, rna);
    st_df(r + k, rnb);
    st_df(w + c, wa);
    st_df(w + k, wb);
    sa.add(df_abs(rna));
    sa.add(df_abs(rnb));
    sr.add(df_mul(wa, rna));
    sr.add(df_mul(wb, rnb));
  }
  if (c < c1) {
    const df rn = df_fma(nalpha, ld_df(q + c), ld_df(r + c));
    const df wn = df_mul(ld_df(rD + c), rn);
    const df pc = ld_df(p + c);
    st_df(e + c, first ? df_mul(alpha, pc) : df_fma(alpha, pc, ld_df(e + c)));
    st_df(r + c, rn);
    st_df(w + c, wn);
    sa.add(df_abs(rn));
    sr.add(df_mul(wn, rn));
  }
  return make_double2(sa.value(), sr.value());
}

// U: r -= alpha q, w = rD r; returns this thread's sum|r| and w.r. (e's update is left to the next
// direction pass or, after the last iteration, to pass_solution_df.)
template <int B>
__device__ __forceinline__ double2 pass_update_late_df(int c0, int c1, df alpha, float2* __restrict__ r,
                                                  float2* __restrict__ w, const float2* __restrict__ q,
                                                  const float2* __restrict__ rD) {
  DfAcc sa, sr;
  const df nalpha = df_neg(alpha);
  int c = c0 + (int)threadIdx.x;
  for (; c + B < c1; c += 2 * B) {
    const int k = c + B;
    const df qa = ld_df(q + c), qb = ld_df(q + k);
    const df ra = ld_df(r + c), rb = ld_df(r + k);
    const df da = ld_df(rD + c), db = ld_df(rD + k);
    const df rna = df_fma(nalpha, qa, ra), rnb = df_fma(nalpha, qb, rb);
    const df wa = df_mul(da, rna), wb = df_mul(db, rnb);
    st_df(r + c, rna);
    st_df(r + k, rnb);
    st_df(w + c, wa);
    st_df(w + k, wb);
    sa.add(df_abs(rna));
    sa.add(df_abs(rnb));
    sr.add(df_mul(wa, rna));
    sr.add(df_mul(wb, rnb));
  }
  if (c < c1) {
    const df rn = df_fma(nalpha, ld_df(q + c), ld_df(r + c));
    const df wn = df_mul(ld_df(rD + c), rn);
    st_df(r + c, rn);
    st_df(w + c, wn);
    sa.add(df_abs(rn));
    sr.add(df_mul(wn, rn));
  }
  return make_double2(sa.value(), sr.value());
}

// The df64 solve kept on chip (see cg_on_chip). The conductances are stored, the off-diagonals
// are their negatives; e starts at zero (e = alpha p + 0 equals the streamed form's e = alpha p).
struct ChipDf {
  using V = df;
  static constexpr bool kSolInU = false;  // e is read by the row's own thread only
  df *p, *q, *w, *sol;
  const df *r, *rD, *coef, *diag;
  struct Sum {
    DfAcc a;
    __device__ __forceinline__ void dot(df x, df y) { a.add(df_mul(x, y)); }
    __device__ __forceinline__ void abs(df x) { a.add(df_abs(x)); }
    __device__ __forceinline__ double value() const { return a.value(); }
  };
  static __device__ __forceinline__ df ld(const df* a, int i) { return ld_df(reinterpret_cast<const float2*>(a) + i); }
  static __device__ __forceinline__ void st(df* a, int i, df v) { st_df(reinterpret_cast<float2*>(a) + i, v); }
  static __device__ __forceinline__ df mul(df a, df b) { return df_mul(a, b); }
  static __device__ __forceinline__ df fma(df a, df b, df c) { return df_fma(a, b, c); }
  static __device__ __forceinline__ df slot(df g, df x, df y) { return df_fma(df_neg(g), x, y); }
  static __device__ __forceinline__ df neg(df a) { return df_neg(a); }
  __device__ __forceinline__ df sol0(int) const { return mkdf(0.0f, 0.0f); }
  template <class Sh>
  static __device__ __forceinline__ df alpha(const Sh& sh) { return df_of(sh.alpha2); }
  template <class Sh>
  static __device__ __forceinline__ df beta(const Sh& sh) { return df_of(sh.beta2); }
};
static_assert(sizeof(df) == sizeof(float2), "df arrays are stored as float2");

// The steps of one launch. Returns false when a barrier failed (the caller leaves).
// `pending` tracks whether e holds a correction not yet added to the field (the same in every
// CTA: it follows the team-wide iteration counts).
template <int B, int W, bool kGeom, int R>
__device__ bool steps_df64(const CaseDev& cs, const CaseDev& cref, const Team& tm, int n_steps, TeamShared<B>& sh,
                           int c0, int c1, bool& pending) {
  const int tid = threadIdx.x;
  float2* __restrict__ e = cs.e2;
  float2* __restrict__ r = reinterpret_cast<float2*>(cs.r);
  float2* __restrict__ w = reinterpret_cast<float2*>(cs.w);
  float2* __restrict__ p = reinterpret_cast<float2*>(cs.p);
  float2* __restrict__ q = reinterpret_cast<float2*>(cs.q);
  const float2* __restrict__ rD = cs.rD2;

  PhaseClock<B> clk(cs, tm, sh);
  const bool src_mode = cs.n_corr > 0 || cs.vSu != nullptr || cs.vSp != nullptr || (kGeom && cs.Sf != nullptr);
  bool convert = ld_volatile_i32(cs.flags) == 0;  // read by every CTA before the first barrier
  [[maybe_unused]] bool loaded = false;
  for (int step = 0; step < n_steps; ++step) {
    int iters_tot = 0, solves = 0, status = 0;
    for (int pass = 0; pass <= cs.n_corr; ++pass) {
      // ---- S: sum of x (first pass of the launch: split the FP64 field; otherwise the last
      //      solve's correction is added first) ---------------------------------------------
      const double v[1] = {pass_sum_df<B>(cref, c0, c1, convert, pending, pass == 0 && cs.n_corr > 0)};
      pending = false;
      if (!team_allreduce<1, B>(tm, v, sh, [&](int, double t, int lane) { fin_mean_df(sh, cs, t, lane); })) return false;
      mark_split(cs, tm, convert);
      if constexpr (kGeom) {
        if (cs.Sf) {  // ---- G: the gradient of the (folded) field, for the correction --------
          pass_grad_df<B, W>(cref, c0, c1);
          if (!team_barrier<B>(tm, sh)) return false;
        }
      }
      clk.lap(kPhAssembly);
      // ---- R: rows, initial residual, normFactor, first direction ----------------------
      const bool rows = step == 0 && pass == 0;  // the matrix is assembled in the launch's first pass
      const df xr = df_of(sh.xref2);
      const Sums3 ui = src_mode ? (rows ? pass_rows_init_df<B, W, true, true>(cref, c0, c1, xr)
                                        : pass_rows_init_df<B, W, true, false>(cref, c0, c1, xr))
                                : (rows ? pass_rows_init_df<B, W, false, true>(cref, c0, c1, xr)
                                        : pass_rows_init_df<B, W, false, false>(cref, c0, c1, xr));
      const double u[3] = {ui.a, ui.b, ui.c};
      if (!team_allreduce<3, B>(tm, u, sh, [&](int k, double t, int lane) {
            if (lane == 0) sh.out[k] = t;
          }))
        return false;
      clk.lap(kPhInit);
      if (tid == 0) {
        sh.nf = sh.out[0] + kSmall * cs.df_scale;
        sh.init_res = sh.res = sh.out[1] / sh.nf;
        sh.rho = sh.out[2];
        sh.conv = converged(sh.res, sh.init_res, cs.tol, cs.rel_tol) ? 1 : 0;
        sh.code = cs.min_iter > 0 || !sh.conv ? kGo : kStop;
        sh.iters = 0;
        if (pass == 0) {
          sh.nf0 = sh.nf * (1.0 / cs.df_scale);  // a power of two: exact
          sh.init0 = sh.init_res;
        }
      }
      __syncthreads();
      int iters = 0;
      if constexpr (R > 0) {
        auto df_at = [](const void* a) { return reinterpret_cast<df*>(const_cast<void*>(a)); };
        const ChipDf f{df_at(p), df_at(q), df_at(w), df_at(e), df_at(r), df_at(rD), df_at(cs.g2), df_at(cs.diag2)};
        if (sh.code == kGo) {
          pending = true;  // unless the first product ends the solve: e is then zero, the same field
          if (!cg_on_chip<ChipDf, B, W, R>(
                  f, cs, cref, tm, sh, clk, c0, c1, loaded,
                  [&](double t, int lane) {
                    fin_sigma(sh, t, lane);
                    if (lane == 0) sh.alpha2 = pair_of(sh.alpha);
                  },
                  [&](int k, double t, int lane, int done) {
                    fin_update(sh, k, t, lane, cs.tol, cs.rel_tol, done, cs.max_iter, cs.min_iter);
                    if (k == 0 && lane == 0) sh.iters = done;
                    if (k == 1 && lane == 0) sh.beta2 = pair_of(sh.beta);
                  })) {
            pending = false;  // the solution was not written
            return false;
          }
        }
        iters = sh.iters;
      }
      // e is updated in P (not compiled into the kernels that serve general geometry, the batched ones
      // among them: the second form's code made batches 2 to 3 % slower)
      const bool late = R == 0 && !kGeom && cs.N >= cs.late_cells / 2;
      bool due = false;  // the last iteration's e += alpha p is still to be done
      while (R == 0 && sh.code == kGo) {
        if (iters > 0) {
          if (late)
            pass_direction_x_df<B>(c0, c1, df_of(sh.alpha2), df_of(sh.beta2), e, iters == 1, p, w);
          else
            pass_direction_df<B>(c0, c1, df_of(sh.beta2), p, w);
          due = false;
          if (!team_barrier<B>(tm, sh)) return false;
          clk.lap(kPhP);
        }
        bool m_ok;
        const double s1[1] = {amul_dot_df<B, W>(cs, cref, c0, c1, p, q, tm, m_ok)};
        if (!m_ok) return false;
        if (!team_allreduce<1, B>(tm, s1, sh, [&](int, double t, int lane) {
              fin_sigma(sh, t, lane);
              if (lane == 0) sh.alpha2 = pair_of(sh.alpha);
            }))
          return false;
        clk.lap(kPhM);
        if (sh.code != kGo) break;
        const double2 su = late ? pass_update_late_df<B>(c0, c1, df_of(sh.alpha2), r, w, q, rD)
                                : pass_update_df<B>(c0, c1, df_of(sh.alpha2), e, iters == 0, r, w, p, q, rD);
        due = late;
        pending = pending || !late;
        const double s2[2] = {su.x, su.y};
        ++iters;
        if (!team_allreduce<2, B>(tm, s2, sh, [&](int k, double t, int lane) {
              fin_update(sh, k, t, lane, cs.tol, cs.rel_tol, iters, cs.max_iter, cs.min_iter);
              if (k == 1 && lane == 0) sh.beta2 = pair_of(sh.beta);
            }))
          return false;
        clk.lap(kPhU);
      }
      if (late && iters > 0 && tm.rank == 0 && tid == 0) ++tm.sw->late;
      if (due) pass_solution_df<B>(c0, c1, df_of(sh.alpha2), e, iters == 1, p);
      if (late && iters > 0) pending = true;
      if (sh.code == kSingular) status = LFM_ESINGULAR;
      if (sh.code == kNonFinite) status = LFM_ENONFINITE;
      iters_tot += iters;
      solves += iters > 0 ? 1 : 0;
      if (status != 0) break;
    }
    write_stats(cs, tm, step, iters_tot, sh.conv, solves, status, sh.init0, sh.res, sh.nf0);
    clk.flush();
    if (status != 0) {
      if (tm.rank == 0 && tid == 0) set_status(cs.sync, status);
      return true;
    }
  }
  return true;
}

// kGeom: the kernel serves general geometry (the gradient phase is compiled in). R: rows per thread
// of a solve kept on chip (0: streamed).
template <int B, int W, bool kGeom = false, int R = 0>
__device__ void run_steps_df64(const CaseDev& cs, const CaseDev& cref, const Team& tm, int n_steps, TeamShared<B>& sh) {
  if (n_steps <= 0) return;
  int c0, c1;
  cta_range(cs.N, tm.size, tm.rank, c0, c1);
  bool pending = false;
  steps_df64<B, W, kGeom, R>(cs, cref, tm, n_steps, sh, c0, c1, pending);
  // the field and the correction of the CTA's own cells are written by this CTA only, so the
  // FP64 field can be written back without another barrier, also after an early exit.
  pass_store_x<B>(cref, c0, c1, pending);
}

}  // namespace
}  // namespace lfm
