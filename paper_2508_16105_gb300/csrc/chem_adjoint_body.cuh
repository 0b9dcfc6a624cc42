// Discrete adjoint of the per-cell chemistry step (sm_103a, FP64): device code,
// templated on the reaction sequence (generic or specialised to a mechanism).
//
// Differentiates the map (T0, Y0, ln A_r, E_r) -> (T, Y)(dt) along each cell's
// frozen sequence of accepted RODAS3 steps (the step sizes are held fixed; the
// rejected attempts and the controller contribute nothing).  Three kernels:
//
//  1. record:  the forward integration again, writing the start state y_n and
//              the size h_n of every accepted step into a pool at per-cell
//              offsets (an exclusive scan of the forward pass's step counts)
//              and, when the caller's workspace holds them, the step's stage
//              checkpoint: the LU factors of M and the stage vectors u_1..u_4;
//  2. reverse: a persistent queue over cells; each lane walks its cell's steps
//              backwards.  Per step it reads the stage checkpoint or recomputes
//              the stages (J(y_n), the LU of M = I/(gamma h) - J, u_1..u_4),
//              then propagates the cotangent:
//                  w_i = M^-T ubar_i                       (transposed LU solves)
//                  ybar += J(Y_i)^T w_i,  ubar_j += a_ij J(Y_i)^T w_i + c_ij/h w_i
//                  ybar += grad_y (w_i^T J(y) u_i),  thbar += grad_th (w_i^T J u_i)
//              J^T w is contracted on the fly (jtw_value: no matrix is formed), and
//              the second-derivative terms grad(w^T J u) = d/de [J(y + e u)^T w] of all
//              four stages come from one evaluation of that contraction with its
//              derivatives (hvp_sum; the precompiled kernels: one dual-number
//              evaluation per stage, jtw);
//  3. reduce:  per-cell parameter gradients summed over cells in a fixed order
//              (bitwise reproducible; no floating-point atomics).
//
// Parameters: ln A_r (of k_inf for falloff reactions) and E_r in J/mol.
#pragma once
#if !defined(__CUDACC_RTC__)  /* run-time compilation: types from the preamble */
#include <cuda_runtime.h>
#include <stdint.h>
#endif

#include "chem_device.cuh"
#include "chem_launch.h"
#include "dual_math.cuh"

namespace rde {

constexpr unsigned kFullA = 0xffffffffu;
constexpr int kThreadsA = kLaneThreads;

// lane-slot view of an array of dual numbers (two slots each)
struct DualSlots {
  Lane L;
  int base;
  __device__ __forceinline__ Dual get(int i) const { return mk(L[base + 2 * i], L[base + 2 * i + 1]); }
  __device__ __forceinline__ void set(int i, Dual v) const {
    L[base + 2 * i] = v.v;
    L[base + 2 * i + 1] = v.d;
  }
  __device__ __forceinline__ void add(int i, Dual v) const {
    L[base + 2 * i] += v.v;
    L[base + 2 * i + 1] += v.d;
  }
};

// Slot map of the reverse kernel.  The forward slots keep the forward kernel's
// names (so the f evaluation, assemble_matrix, lu_factor and lu_solve serve both).  jtw_value
// uses C, G, HRT, CPR, WDOT (for w_k W_k), WD and HD beside the LU.  In the second-derivative
// phase, when the LU is no longer needed, 18 K slots from 0 hold hvp_sum's arrays (or jtw's
// nine dual ones).
template <int K>
struct AdjSlots {
  static constexpr int N = K + 1;
  static constexpr int MX = 0;
  static constexpr int C = MX + N * N;
  static constexpr int G = C + K;
  static constexpr int HRT = G + K;
  static constexpr int CPR = HRT + K;
  static constexpr int WDOT = CPR + K;
  static constexpr int WT = WDOT + K;
  static constexpr int WD = WT + K;
  static constexpr int HD = WD + K;
  static constexpr int DC = HD + K;
  static constexpr int ARG = (DC + K > 18 * K) ? DC + K : 18 * K;   // room for the dual arrays
  static constexpr int VEC = ARG + N;
  static constexpr int TOTAL = VEC + N;
  static constexpr size_t bytes(int threads) { return sizeof(double) * TOTAL * threads; }
};

// ---------------------------------------------------------------------------
// Transposed solve with the factors of lu_factor
// ---------------------------------------------------------------------------
// M^T x = b in place in VEC: P M = L U, so M^T = U^T L^T P; solve U^T z = b, L^T v = z,
// then undo the row interchanges (`piv`, lu_factor's swaps) in reverse order.  The right-
// hand side stays in registers; a finished component updates the others along its row of
// the factors, so the multiply-adds of a row are independent of one another.  The factors
// are those of the live unknowns (INERT); the inert species' rows of M are e_k / (gamma h)
// and their columns are kept as assembled, so w_k = gamma h (b_k - sum_live M_ik w_i).
// Compiled once (four calls a step).
template <int K, unsigned INERT>
__device__ __noinline__ void lu_solve_t(const Lane L, unsigned long long piv, double gh) {
  using S = AdjSlots<K>;
  constexpr int N = S::N;
  double x[N];
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (live<INERT>(i)) x[i] = L[S::VEC + i];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if (!live<INERT>(j)) continue;
    x[j] *= L[S::MX + j * N + j];
#pragma unroll
    for (int i = j + 1; i < N; ++i)
      if (live<INERT>(i)) x[i] = fma(-L[S::MX + j * N + i], x[j], x[i]);
  }
#pragma unroll
  for (int j = N - 1; j > 0; --j) {
    if (!live<INERT>(j)) continue;
#pragma unroll
    for (int i = 0; i < j; ++i)
      if (live<INERT>(i)) x[i] = fma(-L[S::MX + j * N + i], x[j], x[i]);
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (live<INERT>(i)) L[S::VEC + i] = x[i];
#pragma unroll 1
  for (int k = N - 1; k >= 0; --k) {
    const int p = (int)((piv >> (4 * k)) & 15ull);
    if (p != k) {
      const double t = L[S::VEC + k];
      L[S::VEC + k] = L[S::VEC + p];
      L[S::VEC + p] = t;
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (live<INERT>(k)) continue;
    double acc = L[S::VEC + k];
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (live<INERT>(i)) acc = fma(-L[S::MX + i * N + k], L[S::VEC + i], acc);
    L[S::VEC + k] = acc * gh;
  }
}

// ---------------------------------------------------------------------------
// J^T w without forming J, and the parameter cotangents, at state y (of type S)
// ---------------------------------------------------------------------------

// The derivative part of g = J(y)^T w along the dual numbers' direction (the precompiled
// kernels' second-derivative term of one stage), with that of the parameter cotangents
// w^T df/d(ln A_r) and w^T df/dE_r added to the lane's global accumulators
// thA[r * stride], thE[r * stride].  y: N dual values; w: N primal values.  Uses nine dual
// arrays of K from slot `base`.
template <int K, class RX>
__device__ void jtw(const MechView& m, Lane L, int base, double invp, const Dual* y, const double* w, double* g,
                    double* thA, double* thE, long long stride) {
  using S = Dual;
  const DualSlots Cc{L, base}, Gg{L, base + 2 * K}, Hh{L, base + 4 * K}, Cp{L, base + 6 * K}, Wd{L, base + 8 * K},
      Wt{L, base + 10 * K}, WDv{L, base + 12 * K}, HDv{L, base + 14 * K}, DCv{L, base + 16 * K};
  const SpecPacked* sp = m.sp;
  const S T = y[K];
  const S invT = 1.0 / T;
  const S lnT = slog(m, T);
  S sumYW = cst<S>(0.0);
#pragma unroll
  for (int k = 0; k < K; ++k) sumYW += y[k] * sp[k].Winv;
  const S RT = kRu * T;
  const S invrho = RT * sumYW * invp;
  const S rho = 1.0 / invrho;
  S Msum = cst<S>(0.0), cpm = cst<S>(0.0), dcpm = cst<S>(0.0);
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const S yw = y[k] * sp[k].Winv;
    const S c = yw * rho;
    Cc.set(k, c);
    Msum += c;
    const int r = (val(T) >= sp[k].Tmid) ? 1 : 0;
    const double* a = sp[k].cp[r];
    const S cp = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
    const double* hh = sp[k].h[r];
    const S h = hh[0] + T * (hh[1] + T * (hh[2] + T * (hh[3] + T * hh[4]))) + hh[5] * invT;
    const double* gg = sp[k].g[r];
    const S gv = gg[0] + gg[1] * lnT + T * (gg[2] + T * (gg[3] + T * (gg[4] + T * gg[5]))) + gg[6] * invT;
    const double* dc = sp[k].dcp[r];
    dcpm += yw * (dc[0] + T * (dc[1] + T * (dc[2] + T * dc[3])));
    cpm += yw * cp;
    Gg.set(k, gv);
    Hh.set(k, h);
    Cp.set(k, cp);
    Wd.set(k, cst<S>(0.0));
    Wt.set(k, cst<S>(0.0));
    WDv.set(k, cst<S>(0.0));
    HDv.set(k, cst<S>(0.0));
    DCv.set(k, cst<S>(0.0));
  }
  const S cpm_J = kRu * cpm;
  const S lnPRT = kLnPstdOverRu - lnT;
  const S fac_T = (w[K] * RT) / cpm_J;   // weight of the temperature row in w^T df/dq
  RX::each(m, [&](const auto& x, int r) {
    const S lnk = x.lnA() + x.b() * lnT - x.EaR() * invT;
    S M = cst<S>(1.0);
    if (x.type() != RX_ELEM) {
      M = Msum;
      for (int e = x.eff_begin(); e < x.eff_end(); ++e) M += x.eff_am1(m, e) * Cc.get(x.eff_k(m, e));
    }
    const bool fo = (x.type() == RX_LINDEMANN || x.type() == RX_TROE);
    S kf, dlnkf, dkf_dM = cst<S>(0.0), phi = cst<S>(1.0);
    if (fo) {
      kf = falloff_s<S>(m, x, T, lnT, invT, M, sexp(m, lnk), dlnkf, dkf_dM, phi);
    } else {
      kf = sexp(m, lnk);
      dlnkf = (x.b() + x.EaR() * invT) * invT;
    }
    S kr = cst<S>(0.0), dlnKc = cst<S>(0.0);
    if (x.rev()) {
      S lnKc = x.dnu() * lnPRT;
      S dh = cst<S>(0.0);
      for (int q = 0; q < x.nf(); ++q) {
        lnKc += x.fod(q) * Gg.get(x.fi(q));
        dh -= x.fod(q) * Hh.get(x.fi(q));
      }
      for (int q = 0; q < x.nb(); ++q) {
        lnKc -= x.bod(q) * Gg.get(x.bi(q));
        dh += x.bod(q) * Hh.get(x.bi(q));
      }
      kr = fo ? kf * sexp(m, -lnKc) : sexp(m, lnk - lnKc);
      dlnKc = (dh - x.dnu()) * invT;
    }
    S cf[kMaxSide], cb[kMaxSide], pf[kMaxSide], pb[kMaxSide];
#pragma unroll
    for (int q = 0; q < kMaxSide; ++q) {
      cf[q] = (q < x.nf()) ? Cc.get(x.fi(q)) : cst<S>(1.0);
      cb[q] = (q < x.nb()) ? Cc.get(x.bi(q)) : cst<S>(1.0);
      pf[q] = (q < x.nf()) ? ipow_s(cf[q], x.fo(q)) : cst<S>(1.0);
      pb[q] = (q < x.nb()) ? ipow_s(cb[q], x.bo(q)) : cst<S>(1.0);
    }
    S Pf = pf[0], Pb = pb[0];
    if (x.nf() > 1) Pf = Pf * pf[1];
    if (x.nf() > 2) Pf = Pf * pf[2];
    if (x.nb() > 1) Pb = Pb * pb[1];
    if (x.nb() > 2) Pb = Pb * pb[2];
    const S q0 = kf * Pf - kr * Pb;
    const bool tb = (x.type() == RX_THREEBODY);
    const S mf = tb ? M : cst<S>(1.0);
    const S q = mf * q0;
    const S dqdT = mf * (kf * dlnkf * Pf - kr * (dlnkf - dlnKc) * Pb);
    // contraction weights of this reaction: s1 = sum_p wt_p nu_p, s2 = sum_p (H/RT)_p nu_p
    double s1 = 0.0;
    S s2 = cst<S>(0.0);
    for (int pp = 0; pp < x.np(); ++pp) {
      const int k = x.pi(pp);
      s1 += w[k] * sp[k].W * x.pnu(pp);
      s2 += x.pnu(pp) * Hh.get(k);
    }
    // gradient of q w.r.t. the concentrations of each side's species, and grad q . c
    S gf[kMaxSide], gb[kMaxSide];
    const S mkf = mf * kf, mkr = mf * kr;
    S gc = cst<S>(0.0);
#pragma unroll
    for (int s = 0; s < kMaxSide; ++s) {
      const S df = (x.fo(s) == 1) ? cst<S>(1.0) : (x.fo(s) == 2 ? 2.0 * cf[s] : 3.0 * (cf[s] * cf[s]));
      const S db = (x.bo(s) == 1) ? cst<S>(1.0) : (x.bo(s) == 2 ? 2.0 * cb[s] : 3.0 * (cb[s] * cb[s]));
      S of = cst<S>(1.0), ob = cst<S>(1.0);
#pragma unroll
      for (int t = 0; t < kMaxSide; ++t) {
        if (t != s && t < x.nf()) of = of * pf[t];
        if (t != s && t < x.nb()) ob = ob * pb[t];
      }
      gf[s] = mkf * df * of;
      gb[s] = -(mkr * db * ob);
      if (s < x.nf()) gc += gf[s] * cf[s];
      if (s < x.nb()) gc += gb[s] * cb[s];
    }
    S allc = cst<S>(0.0);
    if (tb) allc = q0;
    else if (fo) allc = (val(kf) != 0.0) ? dkf_dM * (q0 / kf) : cst<S>(0.0);
    if (x.type() != RX_ELEM) gc += allc * M;
    for (int pp = 0; pp < x.np(); ++pp) {
      const int k = x.pi(pp);
      const double nu = x.pnu(pp);
      Wd.add(k, nu * q);
      Wt.add(k, nu * dqdT);
      DCv.add(k, nu * gc);
    }
    for (int s = 0; s < x.nf(); ++s) {
      WDv.add(x.fi(s), s1 * gf[s]);
      HDv.add(x.fi(s), s2 * gf[s]);
    }
    for (int s = 0; s < x.nb(); ++s) {
      WDv.add(x.bi(s), s1 * gb[s]);
      HDv.add(x.bi(s), s2 * gb[s]);
    }
    if (x.type() != RX_ELEM) {
      const S a1 = s1 * allc, a2 = s2 * allc;
#pragma unroll 1
      for (int j = 0; j < K; ++j) {
        WDv.add(j, a1);
        HDv.add(j, a2);
      }
      for (int e = x.eff_begin(); e < x.eff_end(); ++e) {
        WDv.add(x.eff_k(m, e), a1 * x.eff_am1(m, e));
        HDv.add(x.eff_k(m, e), a2 * x.eff_am1(m, e));
      }
    }
    // w^T df/dq_r = (s1 - w_T R T s2 / c_p) / rho;  d q / d ln A = phi q;  d q / d E = -phi q / (R T)
    const S sr = (s1 - fac_T * s2) * invrho;
    const S tA = sr * phi * q;
    const S tE = -(tA / RT);
    thA[r * stride] += der(tA);
    thE[r * stride] += der(tE);
  });
  // f_T and the assembly of J^T w
  S sum_hw = cst<S>(0.0), wfe = cst<S>(0.0), wfT = cst<S>(0.0), HDc = cst<S>(0.0), Cw = cst<S>(0.0),
    HwT = cst<S>(0.0);
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const S wd = Wd.get(k), dc = DCv.get(k), h = Hh.get(k), wt = Wt.get(k);
    const double wtk = w[k] * sp[k].W;
    sum_hw += h * wd;
    wfe += wtk * (wd - dc);
    wfT += wtk * (wt + (wd - dc) * invT);
    HDc += h * dc;
    Cw += Cp.get(k) * wd;
    HwT += h * (wt - dc * invT);
  }
  const S fT = -(RT * sum_hw * invrho) / cpm_J;
  const S Wbar = 1.0 / sumYW;
  const S beta = Wbar * invrho * wfe;
  const S inv_cp = 1.0 / cpm_J;
  const S coef = -(RT * inv_cp);
  const S wHDc = Wbar * invrho * HDc;
  const S fcp = fT * inv_cp;
#pragma unroll 1
  for (int i = 0; i < K; ++i) {
    const S gi = sp[i].Winv * (WDv.get(i) + beta +
                               w[K] * (coef * (HDv.get(i) - wHDc) - fcp * (kRu * Cp.get(i) - cpm_J * Wbar)));
    g[i] = der(gi);
  }
  const S JTT = -((kRu * Cw + RT * HwT) * invrho * inv_cp) + fT * invT - fT * (kRu * dcpm) * inv_cp;
  const S gT = invrho * wfT + w[K] * JTT;
  g[K] = der(gT);
}

// ---------------------------------------------------------------------------
// The same J^T w for a double state, contracted reaction by reaction
// ---------------------------------------------------------------------------
// Every term of the final assembly is linear in the reactions' rates q, their T dq/dT and
// their concentration gradients, so the species sums (sum_k w_k W_k omega_k and its kin)
// are taken per reaction with the reaction's own weights s1 = sum_k w_k W_k nu_k,
// s2 = sum_k (H/RT)_k nu_k, sc = sum_k (Cp/R)_k nu_k: no per-species production arrays.
// The rates come from the forward step's rate_pair, and grad q . c from Euler's theorem
// (2 q for a bimolecular reaction both ways).  About 1,100 FP64 operations at 9 species
// and 21 reactions, 1,900 with per-species arrays and FP64 exponentials' arguments.

// state-dependent quantities of one evaluation point, with C, G (fixed point), HRT, CPR of
// the slot map S filled; dcp receives d(Cp/R)/dT of species k
template <int K, class S, class RX, class F>
__device__ __forceinline__ RhsCtx adj_species(const MechView& m, Lane L, const double* y, double invp, F&& dcp_of) {
  RhsCtx cx;
  const SpecPacked* sp = m.sp;
  const double T = y[K];
  cx.T = T;
  cx.invT = recip(T);
  cx.lnT = log_tab(T, m.logtab);
  double sumYW = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double yw = y[k] * sp[k].Winv;
    L[S::C + k] = yw;
    sumYW += yw;
  }
  cx.RT = kRu * T;
  cx.invrho = cx.RT * sumYW * invp;
  cx.rho = recip(cx.invrho);
  cx.sumYW = sumYW;
  cx.Msum = 0.0;
  cx.cpm = cx.dcpm = 0.0;
  cx.fix = false;
  cx.zlnT = cx.zinvT = 0;
  cx.zs = 0;
  cx.poison = false;
  if constexpr (RX::kFix) cx.fix = T >= m.hdr->Tfix && T < 8192.0;
  uint64_t t = 0;
  if (cx.fix) {
    t = to_fix(T, 50);
    cx.zlnT = to_fix(cx.lnT, 59);
    cx.zinvT = to_fix(cx.invT, 70);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double yw = L[S::C + k], c = yw * cx.rho;
    L[S::C + k] = c;
    cx.Msum += c;
    double cp, h, g, dcp;
    if (cx.fix) {
      if constexpr (RX::kFix) {
        int64_t z;
        thermo_fix<true, RX>(sp[k], k, T, t, cx, cp, h, z, dcp);
        g = park_fix(z);
      }
    } else {
      thermo_fp64<true>(sp[k], T, cx.lnT, cx.invT, cp, h, g, dcp);
      cx.zs = max(cx.zs, fix_shift(g));
    }
    L[S::G + k] = g;
    L[S::HRT + k] = h;
    L[S::CPR + k] = cp;
    cx.cpm = fma(yw, cp, cx.cpm);
    cx.dcpm = fma(yw, dcp, cx.dcpm);
    dcp_of(k, dcp, yw);
  }
  cx.lnPRT = kLnPstdOverRu - cx.lnT;
  if (!cx.fix) cx.zs = max(cx.zs, fix_shift(cx.lnPRT));
  cx.zPRT = log2_fix(cx.lnPRT, cx.zs) + kParkBias;
  if (!cx.fix) {
#pragma unroll
    for (int k = 0; k < K; ++k) L[S::G + k] = park_fix(log2_fix(L[S::G + k], cx.zs));
  }
  return cx;
}

// g = J(y)^T w, and w^T df/d(ln A_r), w^T df/dE_r added to thA, thE.  Compiled once (not inlined): three calls a step.
template <int K, class RX>
__device__ __noinline__ void jtw_value(const MechView m, const Lane L, double invp, const double* y, const double* w,
                                       double* g, double* thA, double* thE, long long stride) {
  using S = AdjSlots<K>;
  constexpr int WW = S::WDOT;   // w_k W_k
  const SpecPacked* sp = m.sp;
  const RhsCtx cx = adj_species<K, S, RX>(m, L, y, invp, [](int, double, double) {});
  const double T = cx.T, invT = cx.invT, invrho = cx.invrho, wT = w[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    L[WW + k] = w[k] * sp[k].W;
    L[S::WD + k] = 0.0;
    L[S::HD + k] = 0.0;
  }
  const double cpm_J = kRu * cx.cpm, inv_cp = recip(cpm_J);
  const double facT = wT * cx.RT * inv_cp;   // weight of the temperature row in w^T df/dq
  const double invRT = recip(cx.RT);
  double Vhw = 0.0, Vhg = 0.0, Vcw = 0.0, Vht = 0.0, Ve = 0.0, Vt = 0.0, WDall = 0.0, HDall = 0.0;
  RX::each(m, [&](const auto& x, int r) {
    double M = 1.0;
    if (x.type() != RX_ELEM) M = x.template third_body<S>(m, L, cx.Msum);
    const bool fo = (x.type() == RX_LINDEMANN || x.type() == RX_TROE);
    const bool tb = (x.type() == RX_THREEBODY);
    double kf, kb = 0.0, beta, dkf_dM = 0.0, phi = 1.0;   // beta = T dlnk_f/dT
    if (cx.fix) rate_pair<S, true>(m, L, cx, x, fo, kf, kb);
    else rate_pair<S, false>(m, L, cx, x, fo, kf, kb);
    if (fo) {
      double dlnkf;
      kf = falloff_s<double>(m, x, T, cx.lnT, invT, M, kf, dlnkf, dkf_dM, phi);
      beta = dlnkf * T;
    } else {
      beta = fma(x.EaR(), invT, x.b());
    }
    double s1 = 0.0, s2 = 0.0, sc = 0.0;
    for (int pp = 0; pp < x.np(); ++pp) {
      const int k = x.pi(pp);
      s1 = fma(x.pnu(pp), L[WW + k], s1);
      s2 = fma(x.pnu(pp), L[S::HRT + k], s2);
      sc = fma(x.pnu(pp), L[S::CPR + k], sc);
    }
    double cf[kMaxSide], cb[kMaxSide], pf[kMaxSide], pb[kMaxSide];
#pragma unroll
    for (int q = 0; q < kMaxSide; ++q) {
      cf[q] = (q < x.nf()) ? L[S::C + x.fi(q)] : 1.0;
      cb[q] = (q < x.nb()) ? L[S::C + x.bi(q)] : 1.0;
      pf[q] = (q < x.nf()) ? ipow(cf[q], x.fo(q)) : 1.0;
      pb[q] = (q < x.nb()) ? ipow(cb[q], x.bo(q)) : 1.0;
    }
    double Pf = pf[0], Pb = pb[0];
    if (x.nf() > 1) Pf *= pf[1];
    if (x.nf() > 2) Pf *= pf[2];
    if (x.nb() > 1) Pb *= pb[1];
    if (x.nb() > 2) Pb *= pb[2];
    const double kr = !x.rev() ? 0.0 : (fo ? kf * kb : kb);
    const double rb = x.rev() ? kr * Pb : 0.0;
    const double q0 = x.rev() ? fma(kf, Pf, -rb) : kf * Pf;
    double q = q0, tq = q0 * beta;
    if (x.rev()) tq = fma(rb, s2 - x.dnu(), tq);
    const double mkf = tb ? M * kf : kf, mkr = tb ? M * kr : kr;
    if (tb) {
      q *= M;
      tq *= M;
    }
#pragma unroll
    for (int s = 0; s < kMaxSide; ++s) {
      double vf = mkf, vb = -mkr;
      if (s < x.nf() && x.fo(s) == 2) vf *= 2.0 * cf[s];
      if (s < x.nf() && x.fo(s) == 3) vf *= 3.0 * (cf[s] * cf[s]);
      if (s < x.nb() && x.bo(s) == 2) vb *= 2.0 * cb[s];
      if (s < x.nb() && x.bo(s) == 3) vb *= 3.0 * (cb[s] * cb[s]);
#pragma unroll
      for (int t = 0; t < kMaxSide; ++t) {
        if (t != s && s < x.nf() && t < x.nf()) vf *= pf[t];
        if (t != s && s < x.nb() && t < x.nb()) vb *= pb[t];
      }
      if (s < x.nf()) {
        L[S::WD + x.fi(s)] = fma(s1, vf, L[S::WD + x.fi(s)]);
        L[S::HD + x.fi(s)] = fma(s2, vf, L[S::HD + x.fi(s)]);
      }
      if (x.rev() && s < x.nb()) {
        L[S::WD + x.bi(s)] = fma(s1, vb, L[S::WD + x.bi(s)]);
        L[S::HD + x.bi(s)] = fma(s2, vb, L[S::HD + x.bi(s)]);
      }
    }
    double allc = 0.0;
    if (tb) allc = q0;
    else if (fo) allc = (kf != 0.0) ? dkf_dM * (q0 / kf) : 0.0;
    int of = 0, ob = 0;
    for (int s = 0; s < x.nf(); ++s) of += x.fo(s);
    for (int s = 0; s < x.nb(); ++s) ob += x.bo(s);
    double dG = 0.0;   // grad q . c - 2 q
    if (of != 2) dG = (double)(of - 2) * (kf * Pf);
    if (x.rev() && ob != 2) dG = fma((double)(2 - ob), rb, dG);
    if (tb) dG = fma(M, dG, q);
    if (fo) dG = fma(allc, M, dG);
    if (of != 2 || (x.rev() && ob != 2) || x.type() != RX_ELEM) {
      Ve = fma(-s1, q + dG, Ve);
      Vhg = fma(s2, dG, Vhg);
    } else {
      Ve = fma(-s1, q, Ve);
    }
    Vhw = fma(s2, q, Vhw);
    Vcw = fma(sc, q, Vcw);
    Vht = fma(s2, tq, Vht);
    Vt = fma(s1, tq, Vt);
    if (x.type() != RX_ELEM) {
      const double a1 = s1 * allc, a2 = s2 * allc;
      WDall += a1;
      HDall += a2;
      for (int e = x.eff_begin(); e < x.eff_end(); ++e) {
        const int k = x.eff_k(m, e);
        L[S::WD + k] = fma(a1, x.eff_am1(m, e), L[S::WD + k]);
        L[S::HD + k] = fma(a2, x.eff_am1(m, e), L[S::HD + k]);
      }
    }
    // w^T df/dq_r = (s1 - w_T R T s2 / c_p) / rho;  d q / d ln A = phi q;  d q / d E = -phi q / (R T)
    double tA = fma(-facT, s2, s1) * (invrho * q);
    if (fo) tA *= phi;
    thA[r * stride] += tA;
    thE[r * stride] -= tA * invRT;
  });
  const double Wbar = cx.rho * cx.RT * invp;
  const double HDc = fma(2.0, Vhw, Vhg);
  const double fT = -(cx.RT * Vhw * invrho) * inv_cp;
  const double wr = Wbar * invrho;
  const double beta = wr * Ve;
  const double coef = -(cx.RT * inv_cp), fcp = fT * inv_cp;
  const double c0 = WDall + beta + wT * fma(coef, HDall - wr * HDc, fT * Wbar), c1 = wT * coef, c2 = wT * fcp * kRu;
#pragma unroll
  for (int i = 0; i < K; ++i)
    g[i] = sp[i].Winv * (L[S::WD + i] + fma(c1, L[S::HD + i], fma(-c2, L[S::CPR + i], c0)));
  const double JTT = -((kRu * Vcw + cx.RT * ((Vht - HDc) * invT)) * invrho * inv_cp) + fT * invT -
                     fcp * (kRu * cx.dcpm);
  g[K] = invrho * ((Vt + Ve) * invT) + wT * JTT;
}

// ---------------------------------------------------------------------------
// Second-derivative terms of several stages in one evaluation
// ---------------------------------------------------------------------------
// A value with ND derivative parts (directions).  The stage terms
//     ybar += sum_i grad_y (w_i^T J(y) u_i)
// share the point y, so one evaluation can carry ND directions u_i: the primal
// part (rates, exponentials, thermo) is computed once instead of once per
// direction.  The species accumulators of jtw keep only their primal parts,
// which do not depend on w; their derivative parts are contracted with the
// weights of the final assembly as they are added, into per-direction scalars
// and two direction-summed species arrays.
template <int ND>
struct DualN {
  double v;
  double d[ND];
};
template <int ND>
__device__ __forceinline__ DualN<ND> dn_const(double v) {
  DualN<ND> r;
  r.v = v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = 0.0;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator+(const DualN<ND>& a, const DualN<ND>& b) {
  DualN<ND> r;
  r.v = a.v + b.v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = a.d[i] + b.d[i];
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator-(const DualN<ND>& a, const DualN<ND>& b) {
  DualN<ND> r;
  r.v = a.v - b.v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = a.d[i] - b.d[i];
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator-(const DualN<ND>& a) {
  DualN<ND> r;
  r.v = -a.v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = -a.d[i];
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator+(const DualN<ND>& a, double b) {
  DualN<ND> r = a;
  r.v = a.v + b;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator+(double a, const DualN<ND>& b) { return b + a; }
template <int ND>
__device__ __forceinline__ DualN<ND> operator-(const DualN<ND>& a, double b) {
  DualN<ND> r = a;
  r.v = a.v - b;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator-(double a, const DualN<ND>& b) {
  DualN<ND> r;
  r.v = a - b.v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = -b.d[i];
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator*(const DualN<ND>& a, const DualN<ND>& b) {
  DualN<ND> r;
  r.v = a.v * b.v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = fma(a.v, b.d[i], a.d[i] * b.v);
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator*(double a, const DualN<ND>& b) {
  DualN<ND> r;
  r.v = a * b.v;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = a * b.d[i];
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator*(const DualN<ND>& a, double b) { return b * a; }
template <int ND>
__device__ __forceinline__ DualN<ND> operator/(const DualN<ND>& a, const DualN<ND>& b) {
  const double inv = recip(b.v);
  DualN<ND> r;
  r.v = a.v * inv;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = (a.d[i] - r.v * b.d[i]) * inv;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator/(double a, const DualN<ND>& b) {
  const double inv = recip(b.v);
  DualN<ND> r;
  r.v = a * inv;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = -(r.v * b.d[i]) * inv;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> operator/(const DualN<ND>& a, double b) {
  DualN<ND> r;
  r.v = a.v / b;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = a.d[i] / b;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND>& operator+=(DualN<ND>& a, const DualN<ND>& b) { a = a + b; return a; }
template <int ND>
__device__ __forceinline__ DualN<ND>& operator-=(DualN<ND>& a, const DualN<ND>& b) { a = a - b; return a; }
template <int ND>
__device__ __forceinline__ DualN<ND>& operator*=(DualN<ND>& a, const DualN<ND>& b) { a = a * b; return a; }
template <int ND>
__device__ __forceinline__ double val(const DualN<ND>& x) { return x.v; }
template <> __device__ __forceinline__ DualN<2> cst<DualN<2>>(double v) { return dn_const<2>(v); }
template <> __device__ __forceinline__ DualN<4> cst<DualN<4>>(double v) { return dn_const<4>(v); }
template <int ND>
__device__ __forceinline__ DualN<ND> sexp(const MechView& m, const DualN<ND>& x) {
  const double e = exp_tab(x.v, m.exptab);
  DualN<ND> r;
  r.v = e;
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = e * x.d[i];
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> slog(const MechView& m, const DualN<ND>& x) {
  DualN<ND> r;
  r.v = log_tab(x.v, m.logtab);
#pragma unroll
  for (int i = 0; i < ND; ++i) r.d[i] = x.d[i] / x.v;
  return r;
}
template <int ND>
__device__ __forceinline__ DualN<ND> smax300(const DualN<ND>& x) { return x.v > 1e-300 ? x : dn_const<ND>(1e-300); }
// direction i of x as a single dual number
template <int ND>
__device__ __forceinline__ Dual view(const DualN<ND>& x, int i) { return mk(x.v, x.d[i]); }

// Slots of hvp_sum (arrays of K from 0): concentrations and their ND derivative parts;
// G/RT (fixed point), H/RT, Cp/R and T times the derivatives of the last two; w_k W_k of
// the ND stages; the direction-summed derivative parts of sum w D and of w_T sum H D with
// the primal sum H D; sum_i w_T,i dc/du_i.
template <int K, int ND>
struct HvpSlots {
  static constexpr int C = 0, CD = C + K, G = CD + ND * K, HRT = G + K, CPR = HRT + K, TH = CPR + K, TP = TH + K,
                       WW = TP + K, WDS = WW + ND * K, HDP = WDS + K, HDS = HDP + K, CWK = HDS + K, TOTAL = CWK + K;
};

// g += sum_{i < ND} d/de [J(y + e u_i)^T w_i] and the parameter terms
// d/de [w_i^T df/d(ln A_r)], d/de [w_i^T df/dE_r] added to thA / thE.  y: N primal
// values; u_i, w_i: stages st0 .. st0 + ND - 1 of the lane's U and W (element e
// of stage s at [(s N + e) nl]).  Each direction's terms equal those of one
// dual-number evaluation of jtw, up to rounding order.
//
// FP64 operations bound it (64 pipe cycles a warp instruction), so the derivative parts
// are written out instead of carried as dual numbers: a temperature-only quantity X has the
// one derivative T dX/dT and enters direction i through tau_i = u_iT / T; species sums are
// contracted per reaction with its weights s1_i = sum_k w_ik W_k nu_k, s2 = sum_k (H/RT)_k
// nu_k (as in jtw_value); and grad q . c is 2 q plus a term of the reactions that are not
// bimolecular both ways.  About 240 operations a reaction with four directions, against
// 1,000 with dual numbers throughout; falloff reactions keep dual numbers.  With jtw_value
// and the barrier an iteration, the calibration step of 3,000 front-heavy cells took 166 ms
// instead of 249.
template <int K, int ND, class RX>
__device__ __noinline__ void hvp_sum(const MechView m, const Lane L, double invp, const double* y, const double* U,
                                     const double* W, int st0, long long nl, double* g, double* thA, double* thE,
                                     long long stride) {
  constexpr int N = K + 1;
  using D = DualN<ND>;
  using HS = HvpSlots<K, ND>;
  static_assert(HS::TOTAL <= 18 * K, "hvp_sum slots exceed the reverse kernel's dual area");
  const SpecPacked* sp = m.sp;
  auto u_at = [&](int i, int e) { return U[((long long)(st0 + i) * N + e) * nl]; };
  auto w_at = [&](int i, int e) { return W[((long long)(st0 + i) * N + e) * nl]; };
  double ddcpm = 0.0;   // T d(sum yw dCp/dT)/dT at fixed composition
  const RhsCtx cx = adj_species<K, HS, RX>(m, L, y, invp, [&](int k, double dcp, double yw) {
    L[HS::TP + k] = y[K] * dcp;
    const double* dc = sp[k].dcp[(y[K] >= sp[k].Tmid) ? 1 : 0];
    ddcpm = fma(yw, y[K] * fma(y[K], fma(y[K], 3.0 * dc[3], 2.0 * dc[2]), dc[1]), ddcpm);
  });
  const double T = cx.T, invT = cx.invT, invrho = cx.invrho, rho = cx.rho;
  const double Wbar = rho * cx.RT * invp;
  double tau[ND], wK[ND], rl[ND];   // u_T / T, w_T, d ln(1/rho)
  double cpd[ND], dcpd[ND];         // derivative parts of sum yw Cp/R and sum yw d(Cp/R)/dT
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    tau[i] = u_at(i, K) * invT;
    wK[i] = w_at(i, K);
    rl[i] = cpd[i] = dcpd[i] = 0.0;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      const double ywd = u_at(i, k) * sp[k].Winv;
      L[HS::CD + i * K + k] = ywd;
      rl[i] += ywd;
    }
  }
#pragma unroll
  for (int i = 0; i < ND; ++i) rl[i] = fma(rl[i], Wbar, tau[i]);
  double wkt = 0.0;   // sum_i w_T,i tau_i
#pragma unroll
  for (int i = 0; i < ND; ++i) wkt = fma(wK[i], tau[i], wkt);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double c = L[HS::C + k], cp = L[HS::CPR + k], tp = L[HS::TP + k];
    double cw = 0.0;
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      const double ywd = L[HS::CD + i * K + k];
      cpd[i] = fma(ywd, cp, cpd[i]);
      dcpd[i] = fma(ywd, tp, dcpd[i]);
      const double cd = fma(ywd, rho, -(c * rl[i]));
      L[HS::CD + i * K + k] = cd;
      cw = fma(wK[i], cd, cw);
      L[HS::WW + i * K + k] = w_at(i, k) * sp[k].W;
    }
    L[HS::CWK + k] = cw;
    L[HS::TH + k] = cp - L[HS::HRT + k];
    L[HS::WDS + k] = 0.0;
    L[HS::HDP + k] = 0.0;
    L[HS::HDS + k] = 0.0;
  }
  const double cpm_J = kRu * cx.cpm, inv_cp = recip(cpm_J), invRT = recip(cx.RT);
  // c_p's derivative parts; the weight w_T R T / c_p of the temperature row in w^T df/dq and
  // the sums over i of its derivative and of its value times tau_i
  double facT[ND], SF1 = 0.0, SF2 = 0.0;
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    cpd[i] = kRu * fma(cx.dcpm * T, tau[i], cpd[i]);
    dcpd[i] = kRu * fma(ddcpm, tau[i], dcpd[i] * invT);   // of sum yw d(Cp)/dT
    facT[i] = wK[i] * (cx.RT * inv_cp);
    SF1 += facT[i] * (tau[i] - cpd[i] * inv_cp);
    SF2 = fma(facT[i], tau[i], SF2);
  }
  // contracted sums: derivative parts by direction (SHW: s2 q, SCW: sc q, SE: s1 (q - grad q.c)
  // with its sign reversed, ST: s1 T dq/dT, SHT: s2 T dq/dT, SHG: s2 (grad q.c - 2 q)) and
  // primal values, V?t with the temperature derivative of the weight
  double SHW[ND], SCW[ND], SE[ND], ST[ND], SHT[ND], SHG[ND], Ve[ND], Vt[ND];
#pragma unroll
  for (int i = 0; i < ND; ++i) SHW[i] = SCW[i] = SE[i] = ST[i] = SHT[i] = SHG[i] = Ve[i] = Vt[i] = 0.0;
  double Vhw = 0.0, Vhg = 0.0, Vcw = 0.0, Vht = 0.0, Vhwt = 0.0, Vhgt = 0.0, Vcwt = 0.0, Vhtt = 0.0;
  double WDS_all = 0.0, HDP_all = 0.0, HDS_all = 0.0;   // terms of every species
  auto cget = [&](int k) {
    D r;
    r.v = L[HS::C + k];
#pragma unroll
    for (int i = 0; i < ND; ++i) r.d[i] = L[HS::CD + i * K + k];
    return r;
  };
  RX::each(m, [&](const auto& x, int r) {
    const bool fo = (x.type() == RX_LINDEMANN || x.type() == RX_TROE);
    const bool tb = (x.type() == RX_THREEBODY);
    double kf, kb = 0.0;
    if (cx.fix) rate_pair<HS, true>(m, L, cx, x, fo, kf, kb);
    else rate_pair<HS, false>(m, L, cx, x, fo, kf, kb);
    // reaction weights; t?: T times their temperature derivatives
    double s1[ND], s2 = 0.0, s2t = 0.0, sc = 0.0, sct = 0.0;
#pragma unroll
    for (int i = 0; i < ND; ++i) s1[i] = 0.0;
    for (int pp = 0; pp < x.np(); ++pp) {
      const int k = x.pi(pp);
      const double nu = x.pnu(pp);
      s2 = fma(nu, L[HS::HRT + k], s2);
      s2t = fma(nu, L[HS::TH + k], s2t);
      sc = fma(nu, L[HS::CPR + k], sc);
      sct = fma(nu, L[HS::TP + k], sct);
#pragma unroll
      for (int i = 0; i < ND; ++i) s1[i] = fma(nu, L[HS::WW + i * K + k], s1[i]);
    }
    const double s2w = s2t * wkt;
    // third-body concentration
    D M = cst<D>(1.0);
    if (x.type() != RX_ELEM) {
      M.v = cx.Msum;
#pragma unroll
      for (int i = 0; i < ND; ++i) M.d[i] = -(cx.Msum * tau[i]);   // sum_k c_k = p / (R_u T)
      for (int e = x.eff_begin(); e < x.eff_end(); ++e) M += x.eff_am1(m, e) * cget(x.eff_k(m, e));
    }
    // concentration products of both sides
    D pf[kMaxSide], pb[kMaxSide];
#pragma unroll
    for (int q = 0; q < kMaxSide; ++q) {
      if (q < x.nf()) pf[q] = ipow_s(cget(x.fi(q)), x.fo(q));
      if (q < x.nb()) pb[q] = ipow_s(cget(x.bi(q)), x.bo(q));
    }
    D Pf = pf[0], Pb = pb[0];
    if (x.nf() > 1) Pf = Pf * pf[1];
    if (x.nf() > 2) Pf = Pf * pf[2];
    if (x.nb() > 1) Pb = Pb * pb[1];
    if (x.nb() > 2) Pb = Pb * pb[2];
    int of = 0, ob = 0;
    for (int s = 0; s < x.nf(); ++s) of += x.fo(s);
    for (int s = 0; s < x.nb(); ++s) ob += x.bo(s);
    const bool euler = of != 2 || (x.rev() && ob != 2) || x.type() != RX_ELEM;   // grad q . c is not 2 q
    // side-by-side rates: fk = k P of each side with k's T-derivative beta = T dln k/dT
    double q, tq, dG = 0.0, qd[ND], tqd[ND], dGd[ND], phiq_v = 0.0, phiq_d[ND];
    D allc = cst<D>(0.0);
    // one side's slot s: adds g = dq/dc_k, given as g.v and the direction sums of g.d
    auto slot = [&](int k, double gv, double s1d, double wkd) {
      L[HS::WDS + k] += s1d;
      L[HS::HDP + k] = fma(s2, gv, L[HS::HDP + k]);
      L[HS::HDS + k] += fma(s2, wkd, s2w * gv);
    };
    if (!fo) {
      const double e = x.EaR() * invT, beta = x.b() + e;
      const double gamma = beta - (s2 - x.dnu());   // T dln k_r/dT
      const double kr = x.rev() ? kb : 0.0;
      const double rf = kf * Pf.v, rb = x.rev() ? kr * Pb.v : 0.0;
      const double q0 = rf - rb, tq0 = x.rev() ? fma(rf, beta, -(rb * gamma)) : rf * beta;
      // T d(T dq/dT)/dT = rf (beta^2 - e) - rb (gamma^2 - e - s2t)
      double tt0 = rf * fma(beta, beta, -e);
      if (x.rev()) tt0 = fma(-rb, fma(gamma, gamma, -e) - s2t, tt0);
      const double bkf = beta * kf, gkr = gamma * kr;
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        double a = kf * Pf.d[i], b = bkf * Pf.d[i];
        if (x.rev()) {
          a = fma(-kr, Pb.d[i], a);
          b = fma(-gkr, Pb.d[i], b);
        }
        qd[i] = fma(tq0, tau[i], a);
        tqd[i] = fma(tt0, tau[i], b);
        if (euler) {
          // derivative part of (of - 2) rf - (ob - 2) rb
          double dg = 0.0;
          if (of != 2) dg = (double)(of - 2) * fma(rf * beta, tau[i], kf * Pf.d[i]);
          if (x.rev() && ob != 2) dg = fma((double)(2 - ob), fma(rb * gamma, tau[i], kr * Pb.d[i]), dg);
          dGd[i] = dg;
        }
      }
      if (euler) {
        if (of != 2) dG = (double)(of - 2) * rf;
        if (x.rev() && ob != 2) dG = fma((double)(2 - ob), rb, dG);
      }
      q = q0;
      tq = tq0;
      double mkf = kf, mkr = kr, s1m = 0.0, wkm = 0.0;   // tb: sum_i s1_i dM_i, sum_i w_T,i dM_i
      if (tb) {
        // by the product rule: M may be zero (no species of the cell is a third body)
        allc.v = q0;
        q = M.v * q0;
        tq = M.v * tq0;
#pragma unroll
        for (int i = 0; i < ND; ++i) {
          const double qd0 = qd[i];
          allc.d[i] = qd0;
          qd[i] = fma(q0, M.d[i], M.v * qd0);
          tqd[i] = fma(tq0, M.d[i], M.v * tqd[i]);
          dGd[i] = fma(M.v, dGd[i], fma(dG, M.d[i], qd[i]));
          s1m = fma(s1[i], M.d[i], s1m);
          wkm = fma(wK[i], M.d[i], wkm);
        }
        dG = fma(M.v, dG, q);
        mkf *= M.v;
        mkr *= M.v;
      }
      double s1t = 0.0;
#pragma unroll
      for (int i = 0; i < ND; ++i) s1t = fma(s1[i], tau[i], s1t);
      // a slot's g = M k O (O the other factors): sum_i s1_i g.d_i = M k sum s1 O.d + k O (M theta s1t + s1m)
#pragma unroll
      for (int s = 0; s < 2 * kMaxSide; ++s) {
        const bool fw = s < kMaxSide;
        const int j = fw ? s : s - kMaxSide;
        if (fw ? j < x.nf() : (x.rev() && j < x.nb())) {
          const int k = fw ? x.fi(j) : x.bi(j), o = fw ? x.fo(j) : x.bo(j), n = fw ? x.nf() : x.nb();
          const double k1 = fw ? kf : -kr, kk = fw ? mkf : -mkr, theta = fw ? beta : gamma;
          double Ov, s1o, wko;
          const int other = 1 - j;   // of a two-species side
          if (n == 1 && o == 1) {
            Ov = 1.0;
            s1o = wko = 0.0;
          } else if (o == 1 && n == 2 && (fw ? x.fo(other) : x.bo(other)) == 1) {
            const int ko = fw ? x.fi(other) : x.bi(other);
            Ov = L[HS::C + ko];
            s1o = 0.0;
#pragma unroll
            for (int i = 0; i < ND; ++i) s1o = fma(s1[i], L[HS::CD + i * K + ko], s1o);
            wko = L[HS::CWK + ko];
          } else {
            const D c = cget(k);
            D O = o == 1 ? cst<D>(1.0) : (o == 2 ? 2.0 * c : 3.0 * (c * c));
#pragma unroll
            for (int t = 0; t < kMaxSide; ++t)
              if (t != j && t < n) O = O * (fw ? pf[t] : pb[t]);
            Ov = O.v;
            s1o = wko = 0.0;
#pragma unroll
            for (int i = 0; i < ND; ++i) {
              s1o = fma(s1[i], O.d[i], s1o);
              wko = fma(wK[i], O.d[i], wko);
            }
          }
          const double g1 = (n == 1 && o == 1) ? k1 : k1 * Ov, gv = tb ? M.v * g1 : g1;
          double a = theta * s1t, b = theta * wkt;
          if (tb) {
            const double mt = M.v * theta;
            a = fma(mt, s1t, s1m);
            b = fma(mt, wkt, wkm);
          }
          slot(k, gv, fma(kk, s1o, g1 * a), fma(kk, wko, g1 * b));
        }
      }
      phiq_v = q;
#pragma unroll
      for (int i = 0; i < ND; ++i) phiq_d[i] = qd[i];
    } else {
      // falloff: dual numbers throughout
      D Td, lnT, iT, kfd, dlnkf, dkf_dM, phi, kinf, kr, dlnKc;
      Td.v = T;
      iT.v = invT;
      lnT.v = cx.lnT;
      kinf.v = kf;
      kr.v = kb;   // e^(-ln K_c)
      dlnKc.v = (s2 - x.dnu()) * invT;
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        Td.d[i] = T * tau[i];
        iT.d[i] = -(invT * tau[i]);
        lnT.d[i] = tau[i];
        kinf.d[i] = kf * fma(x.EaR(), invT, x.b()) * tau[i];
        kr.d[i] = -kb * (s2 - x.dnu()) * tau[i];
        dlnKc.d[i] = (s2t * invT - dlnKc.v) * tau[i];
      }
      kfd = falloff_s<D>(m, x, Td, lnT, iT, M, kinf, dlnkf, dkf_dM, phi);
      kr = x.rev() ? kfd * kr : cst<D>(0.0);
      const D rf = kfd * Pf, rb = x.rev() ? kr * Pb : cst<D>(0.0);
      const D q0 = rf - rb, dq = rf * dlnkf - rb * (dlnkf - dlnKc), tqn = Td * dq;
      allc = (kfd.v != 0.0) ? dkf_dM * (q0 / kfd) : cst<D>(0.0);
      const D dg = (double)(of - 2) * rf - (double)(ob - 2) * rb + allc * M;
      const D pq = phi * q0;
      q = q0.v;
      tq = tqn.v;
      dG = dg.v;
      phiq_v = pq.v;
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        qd[i] = q0.d[i];
        tqd[i] = tqn.d[i];
        dGd[i] = dg.d[i];
        phiq_d[i] = pq.d[i];
      }
#pragma unroll
      for (int s = 0; s < 2 * kMaxSide; ++s) {
        const bool fw = s < kMaxSide;
        const int j = fw ? s : s - kMaxSide;
        if (fw ? j < x.nf() : (x.rev() && j < x.nb())) {
          const int k = fw ? x.fi(j) : x.bi(j), o = fw ? x.fo(j) : x.bo(j), n = fw ? x.nf() : x.nb();
          const D c = cget(k);
          D G = fw ? kfd : -kr;
          if (o == 2) G = G * (2.0 * c);
          if (o == 3) G = G * (3.0 * (c * c));
#pragma unroll
          for (int t = 0; t < kMaxSide; ++t)
            if (t != j && t < n) G = G * (fw ? pf[t] : pb[t]);
          double s1d = 0.0, wkd = 0.0;
#pragma unroll
          for (int i = 0; i < ND; ++i) {
            s1d = fma(s1[i], G.d[i], s1d);
            wkd = fma(wK[i], G.d[i], wkd);
          }
          slot(k, G.v, s1d, wkd);
        }
      }
    }
    Vhw = fma(s2, q, Vhw);
    Vhwt = fma(s2t, q, Vhwt);
    Vcw = fma(sc, q, Vcw);
    Vcwt = fma(sct, q, Vcwt);
    Vht = fma(s2, tq, Vht);
    Vhtt = fma(s2t, tq, Vhtt);
    const double qe = euler ? q + dG : q;
    if (euler) {
      Vhg = fma(s2, dG, Vhg);
      Vhgt = fma(s2t, dG, Vhgt);
    }
    // w_i^T df/dq_r = a_i / rho, a_i = s1_i - facT_i s2;  d q / d ln A = phi q;  d q / d E = -phi q / (R T)
    double aq = 0.0, ar = 0.0, at = 0.0;
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      SHW[i] = fma(s2, qd[i], SHW[i]);
      SCW[i] = fma(sc, qd[i], SCW[i]);
      SE[i] = fma(s1[i], euler ? qd[i] + dGd[i] : qd[i], SE[i]);
      ST[i] = fma(s1[i], tqd[i], ST[i]);
      SHT[i] = fma(s2, tqd[i], SHT[i]);
      if (euler) SHG[i] = fma(s2, dGd[i], SHG[i]);
      Ve[i] = fma(s1[i], qe, Ve[i]);
      Vt[i] = fma(s1[i], tq, Vt[i]);
      const double a = fma(-facT[i], s2, s1[i]);
      aq = fma(a, phiq_d[i], aq);
      ar = fma(a, rl[i], ar);
      at = fma(a, tau[i], at);
    }
    if (x.type() != RX_ELEM) {
      double a1s = 0.0, a2s = 0.0;
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        a1s = fma(s1[i], allc.d[i], a1s);
        a2s = fma(wK[i], allc.d[i], a2s);
      }
      a2s = fma(s2, a2s, s2w * allc.v);
      const double a2 = s2 * allc.v;
      WDS_all += a1s;
      HDP_all += a2;
      HDS_all += a2s;
      for (int e = x.eff_begin(); e < x.eff_end(); ++e) {
        const int k = x.eff_k(m, e);
        const double am1 = x.eff_am1(m, e);
        L[HS::WDS + k] += a1s * am1;
        L[HS::HDP + k] += a2 * am1;
        L[HS::HDS + k] += a2s * am1;
      }
    }
    const double dA = invrho * (aq + phiq_v * (ar - fma(SF1, s2, SF2 * s2t)));
    thA[r * stride] += dA;
    thE[r * stride] -= invRT * (dA - invrho * phiq_v * at);
  });
  // final assembly of each direction as single dual numbers
  double Acoef = 0.0, AwHDc = 0.0, Afcp = 0.0, AT = 0.0, AcpW = 0.0, Bbeta = 0.0, coef_v = 0.0, wHDc_v = 0.0,
         fcp_v = 0.0, cpW_v = 0.0, gKs = 0.0;
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    const Dual RTi = mk(cx.RT, cx.RT * tau[i]), invrhoi = mk(invrho, invrho * rl[i]), invTi = mk(invT, -(invT * tau[i]));
    const Dual cpi = mk(cpm_J, cpd[i]), inv_cpi = mk(inv_cp, -(inv_cp * inv_cp) * cpd[i]);
    const Dual Wbari = mk(Wbar, -Wbar * (rl[i] - tau[i]));
    const Dual Xhw = mk(Vhw, fma(Vhwt, tau[i], SHW[i]));
    const Dual Xdc = mk(fma(2.0, Vhw, Vhg), fma(fma(2.0, Vhwt, Vhgt), tau[i], fma(2.0, SHW[i], SHG[i])));
    const Dual Xcw = mk(Vcw, fma(Vcwt, tau[i], SCW[i]));
    const Dual Xht = mk(Vht, fma(Vhtt, tau[i], SHT[i]));
    const Dual Ye = mk(-Ve[i], -SE[i]), Yt = mk(Vt[i], ST[i]);
    const Dual fT = -(RTi * Xhw * invrhoi * inv_cpi);
    const Dual wr = Wbari * invrhoi;
    const Dual beta = wr * Ye;
    const Dual coef = -(RTi * inv_cpi), wHDc = wr * Xdc, fcp = fT * inv_cpi, cpW = cpi * Wbari;
    const Dual HwT = (Xht - Xdc) * invTi;
    const Dual JTT = -((kRu * Xcw + RTi * HwT) * invrhoi * inv_cpi) + fT * invTi - fcp * mk(kRu * cx.dcpm, dcpd[i]);
    const Dual gT = invrhoi * ((Yt + Ye) * invTi) + wK[i] * JTT;
    Bbeta += beta.d;
    Acoef = fma(wK[i], coef.d, Acoef);
    AwHDc = fma(wK[i], wHDc.d, AwHDc);
    Afcp = fma(wK[i], fcp.d, Afcp);
    AT = fma(wK[i], tau[i], AT);
    AcpW = fma(wK[i], cpW.d, AcpW);
    coef_v = coef.v;
    wHDc_v = wHDc.v;
    fcp_v = fcp.v;
    cpW_v = cpW.v;
    gKs += gT.d;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double hdv = L[HS::HDP + k] + HDP_all;
    const double gi = Acoef * (hdv - wHDc_v) + coef_v * (L[HS::HDS + k] + HDS_all - AwHDc) -
                      Afcp * (kRu * L[HS::CPR + k] - cpW_v) - fcp_v * (kRu * L[HS::TP + k] * AT - AcpW);
    g[k] += sp[k].Winv * (L[HS::WDS + k] + WDS_all + Bbeta + gi);
  }
  g[K] += gKs;
}

// ---------------------------------------------------------------------------
// kernel 1: record the accepted steps of every cell's forward integration
// ---------------------------------------------------------------------------
struct AdjArgs {
  const unsigned char* mech;
  const unsigned char* plan;   // gather plan of the CTA-per-cell kernels (null for thread per cell)
  int mech_bytes;
  int K, R;
  long long n;
  const double* p;
  const double* T0;
  const double* Y0;
  long long ldY;
  double dt;
  rde_chem_options opt;
  const int* n_steps;          // [n] accepted steps of the forward pass
  long long total_steps;       // records the pool (and stages) hold
  const long long* order;      // [n] cells by accepted steps, most first (null: index order)
  long long* offsets;          // [n + 1] exclusive scan of n_steps
  double* pool;                // [sum n_steps][N + 1]: y_n then h_n
  double* stages;              // null, or [sum n_steps][N N + 4 N + 1]: the step's LU factors
                               // (1/U_kk on the diagonal), pivot word, u_1 .. u_4
  int* rec;                    // [n] steps recorded (or -status on failure)
  const double* gT;            // [n]
  const double* gY;            // [K][ldY]
  double* gT0;                 // [n]
  double* gY0;                 // [K][ldY]
  double* lane_scratch;        // [(8 N + 2 R) x lanes]
  double* rows;                // [2 R][n] per-cell parameter cotangents
  unsigned long long* queue;   // [2] work-queue counters (record, reverse)
  int* status;                 // optional [n]
  int num_sms;
  // self-checkpointing mode (n_steps == null: the step counts are not known in advance)
  int ckpt_S;                  // checkpoint entries per cell (a power of two), 0 otherwise
  int seg_max;                 // largest checkpoint stride the options allow (power of two)
  double* ckpt;                // [n][ckpt_S][N + 3]: y_n, t_n, the proposed step size at t_n, h_n
  double* seg;                 // [seg_max][N + 1][lanes]: the replayed y_n, h_n of one segment
  double* replay;              // [N + 6][lanes]: replay state y, t, h, rejected flag, count, target, attempts
};

// The adjoint's copy of the forward attempt, compiled once per kernel (not inlined).  Its
// rounding is explicit (chem_device.cuh), so the record pass, the forward kernels and the
// reverse sweep's segment replays take the same steps bit for bit.
template <int K, class RX>
__device__ __noinline__ bool adj_attempt(const MechView m, const Lane L, double invp, const double* y, double h,
                                         const Opts o, double* yn, double* err, bool* finite,
                                         unsigned long long* swaps, double* U) {
  constexpr int N = K + 1;
  double yv[N], ynv[N], Uv[4][N];
#pragma unroll
  for (int i = 0; i < N; ++i) yv[i] = y[i];
  const bool ok = rosenbrock_attempt<K, RhsOf<RX>, kMethodRodas3, true>(m, L, invp, yv, h, o, ynv, *err, *finite,
                                                                        *swaps, Uv);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    yn[i] = ynv[i];
    U[i] = Uv[0][i];
    U[N + i] = Uv[1][i];
    U[2 * N + i] = Uv[2][i];
    U[3 * N + i] = Uv[3][i];
  }
  return ok;
}

// Stride of a cell's checkpoints in self-checkpointing mode: the smallest power of two
// s with nrec <= S s (the record pass thins its S entries to every other one whenever
// they are full, so entry e holds step e s).
__host__ __device__ __forceinline__ int ckpt_stride(int nrec, int S) {
  int s = 1;
  while ((long long)S * s < (long long)nrec) s <<= 1;
  return s;
}

template <int K, class RX>
__device__ __forceinline__ void record_body(const AdjArgs& a) {
  using S = Slots<K>;
  constexpr int N = K + 1;
  extern __shared__ __align__(16) unsigned char smem[];
  {
    const int4* src = reinterpret_cast<const int4*>(a.mech);
    int4* dst = reinterpret_cast<int4*>(smem);
    for (int i = threadIdx.x; i < a.mech_bytes / 16; i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();
  const MechView m = mech_view(smem);
  const Lane L{reinterpret_cast<double*>(smem + a.mech_bytes) + threadIdx.x};
  const int lane = threadIdx.x & 31;
  const Opts o{a.opt.rtol, a.opt.atol, a.opt.h_min, a.opt.facmax, a.opt.facmin, a.opt.safety, a.opt.max_substeps, 0};
  const double dt = a.dt;
  bool active = false, exhausted = false;
  long long cell = 0, off = 0;
  int cap = 0, nrec = 0, attempts = 0;
  double y[N];
  double invp = 0.0, t = 0.0, h = 0.0;
  bool reject_prev = false;
  const bool self = a.ckpt_S > 0;
  int stride = 1;      // self mode: current checkpoint stride
  double hp0 = 0.0;    // self mode: the step size proposed for the next step (before any rejection)
  for (;;) {
    bool need = !active && !exhausted;
    while (__any_sync(kFullA, need)) {
      const unsigned mask = __ballot_sync(kFullA, need);
      const int leader = __ffs(mask) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(a.queue, (unsigned long long)__popc(mask));
      base = __shfl_sync(kFullA, base, leader);
      if (need) {
        const long long q = (long long)(base + __popc(mask & ((1u << lane) - 1u)));
        // queue position q holds the q-th cell of the cost order (most accepted steps first)
        const long long g = (q < a.n && a.order) ? a.order[q] : q;
        if (q >= a.n) {
          exhausted = true;
          need = false;
        } else if (g < 0 || g >= a.n) {
          // an order entry outside [0, n): nothing to do for this position
        } else {
          cell = g;
          const double p = a.p[g];
          bool good = isfinite(p) && p > 0.0;
#pragma unroll
          for (int k = 0; k < K; ++k) {
            y[k] = a.Y0[k * a.ldY + g];
            good = good && isfinite(y[k]);
          }
          y[K] = a.T0[g];
          good = good && isfinite(y[K]) && y[K] > 0.0;
          invp = 1.0 / p;
          t = 0.0;
          h = dt;
          nrec = attempts = 0;
          reject_prev = false;
          stride = 1;
          hp0 = h;
          bool room = true;
          if (!self) {
            off = a.offsets[g];
            cap = (int)(a.offsets[g + 1] - off);
            // the caller's total_steps is below the sum of n_steps: no room for this cell
            room = a.offsets[g + 1] <= a.total_steps;
          }
          if (!room) {
            a.rec[g] = -RDE_CELL_ADJ_MISMATCH;
          } else if (good) {
            active = true;
            need = false;
          } else {
            a.rec[g] = -RDE_CELL_BAD_STATE;
          }
        }
      }
    }
    // the CTA's warps stay in step (one barrier an iteration), so that they share the
    // instruction cache: the loop body is several times its size
    if (!__syncthreads_or(active ? 1 : 0)) break;
    if (active) {
      int fail = 0;
      if (attempts >= o.max_substeps) {
        fail = RDE_CELL_MAX_SUBSTEPS;
      } else {
        ++attempts;
        h = fmin(h, dt - t);
        // the forward kernel's attempt, in the one compiled copy the replays share
        double yn[N], err, U[4][N];
        bool finite;
        unsigned long long swaps;
        if (!adj_attempt<K, RX>(m, L, invp, y, h, o, yn, &err, &finite, &swaps, &U[0][0])) {
          fail = RDE_CELL_LU_SINGULAR;
        } else if (finite && err <= 1.0) {
          if (self) {
            // checkpoint of this step at every stride-th step; when the S entries are full,
            // keep every other one and double the stride
            if ((nrec & (stride - 1)) == 0) {
              double* base = a.ckpt + cell * (long long)a.ckpt_S * (N + 3);
              int e = nrec / stride;
              if (e == a.ckpt_S) {
#pragma unroll 1
                for (int q = 1; q < a.ckpt_S / 2; ++q) {
#pragma unroll
                  for (int f = 0; f < N + 3; ++f) base[q * (N + 3) + f] = base[2 * q * (N + 3) + f];
                }
                stride <<= 1;
                e = a.ckpt_S / 2;
              }
              double* en = base + (long long)e * (N + 3);
#pragma unroll
              for (int i = 0; i < N; ++i) en[i] = y[i];
              en[N] = t;
              en[N + 1] = hp0;
              en[N + 2] = h;
            }
          } else if (nrec < cap) {
            double* rec = a.pool + (off + nrec) * (N + 1);
#pragma unroll
            for (int i = 0; i < N; ++i) rec[i] = y[i];
            rec[N] = h;
            if (a.stages) {
              // stage checkpoint: the LU factors as lu_factor leaves them (1/U_kk on the
              // diagonal), the interchanges as 4-bit fields of one word, the four stages
              double* cp = a.stages + (off + nrec) * (long long)(N * N + 4 * N + 1);
#pragma unroll 1
              for (int r = 0; r < N; ++r) {
#pragma unroll 2
                for (int c = 0; c < N; ++c) cp[r * N + c] = L[S::MX + r * N + c];
              }
              cp[N * N] = __longlong_as_double((long long)swaps);
#pragma unroll
              for (int i = 0; i < N; ++i) {
                cp[N * N + 1 + i] = U[0][i];
                cp[N * N + 1 + N + i] = U[1][i];
                cp[N * N + 1 + 2 * N + i] = U[2][i];
                cp[N * N + 1 + 3 * N + i] = U[3][i];
              }
            }
          }
          ++nrec;
#pragma unroll
          for (int i = 0; i < N; ++i) y[i] = yn[i];
          t += h;
          h *= step_factor<kMethodRodas3>(err, finite, true, reject_prev, o);
          hp0 = h;
          reject_prev = false;
          if (dt - t <= 1e-14 * dt) {
            a.rec[cell] = (self || nrec == cap) ? nrec : -RDE_CELL_ADJ_MISMATCH;
            active = false;
          }
        } else {
          h *= step_factor<kMethodRodas3>(err, finite, false, reject_prev, o);
          reject_prev = true;
          if (h < o.hmin) fail = RDE_CELL_H_UNDERFLOW;
        }
      }
      if (fail) {
        a.rec[cell] = -fail;
        active = false;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// kernel 2: reverse sweep
// ---------------------------------------------------------------------------
template <int K, class RX, int ND = 1, bool SELF = false>
__device__ __forceinline__ void reverse_body(const AdjArgs& a) {
  static_assert(ND == 1 || ND == 2 || ND == 4, "the four stages split into evaluations of ND directions");
  using S = AdjSlots<K>;
  constexpr int N = K + 1;
  extern __shared__ __align__(16) unsigned char smem[];
  {
    const int4* src = reinterpret_cast<const int4*>(a.mech);
    int4* dst = reinterpret_cast<int4*>(smem);
    for (int i = threadIdx.x; i < a.mech_bytes / 16; i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();
  const MechView m = mech_view(smem);
  const Lane L{reinterpret_cast<double*>(smem + a.mech_bytes) + threadIdx.x};
  const int lane = threadIdx.x & 31;
  const long long nl = (long long)gridDim.x * blockDim.x;
  const long long me = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double* U = a.lane_scratch + me;                  // U[(i*N + e) * nl]
  double* W = a.lane_scratch + 4 * N * nl + me;     // W[(i*N + e) * nl]
  double* thA = a.lane_scratch + 8 * N * nl + me;   // thA[r * nl]
  double* thE = thA + (long long)a.R * nl;
  bool active = false, exhausted = false;
  long long cell = 0, off = 0;
  int s = 0;
  double lam[N];
  double invp = 0.0;
  // self-checkpointing mode: the cell's checkpoint stride, whether the lane is replaying
  // a segment, the first step the segment buffer holds and the cell's step count
  int cs = 1, seg0 = 0, ncell = 0;
  bool replaying = false;
  double* Rp = a.replay + me;                       // Rp[f * nl], f < N + 6
  double* Sg = a.seg + me;                          // Sg[(q * (N + 1) + f) * nl]
  const double* Ck = nullptr;                       // the cell's checkpoints
  // start replaying segment j (steps j cs .. ) from its checkpoint
  auto begin_replay = [&](int j) {
    const double* en = Ck + (long long)j * (N + 3);
#pragma unroll
    for (int i = 0; i < N; ++i) Rp[i * nl] = en[i];
    Rp[N * nl] = en[N];            // t
    Rp[(N + 1) * nl] = en[N + 1];  // proposed step size
    Rp[(N + 2) * nl] = 0.0;        // previous attempt rejected
    Rp[(N + 3) * nl] = 0.0;        // steps replayed
    Rp[(N + 4) * nl] = (double)min(cs, ncell - j * cs);
    Rp[(N + 5) * nl] = 0.0;        // attempts
    seg0 = j * cs;
    replaying = true;
  };
  // the cell's gradients are zero and its status `st` (failed forward or replay)
  auto fail_cell = [&](int st) {
    if (a.status) a.status[cell] = st;
#pragma unroll
    for (int k = 0; k < K; ++k) a.gY0[k * a.ldY + cell] = 0.0;
    a.gT0[cell] = 0.0;
    for (int j = 0; j < 2 * a.R; ++j) a.rows[(long long)j * a.n + cell] = 0.0;
    active = false;
  };
  for (;;) {
    bool need = !active && !exhausted;
    while (__any_sync(kFullA, need)) {
      const unsigned mask = __ballot_sync(kFullA, need);
      const int leader = __ffs(mask) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(a.queue + 1, (unsigned long long)__popc(mask));
      base = __shfl_sync(kFullA, base, leader);
      if (need) {
        const long long q = (long long)(base + __popc(mask & ((1u << lane) - 1u)));
        // queue position q holds the q-th cell of the cost order (most accepted steps first)
        const long long g = (q < a.n && a.order) ? a.order[q] : q;
        if (q >= a.n) {
          exhausted = true;
          need = false;
        } else if (g < 0 || g >= a.n) {
          // an order entry outside [0, n): nothing to do for this position
        } else {
          cell = g;
          const int nrec = a.rec[g];
          if (a.status) a.status[g] = nrec > 0 ? RDE_CELL_OK : -nrec;
          for (int j = 0; j < 2 * a.R; ++j) thA[(long long)j * nl] = 0.0;
          if (nrec <= 0) {
            // failed or inconsistent forward: no gradient
#pragma unroll
            for (int k = 0; k < K; ++k) a.gY0[k * a.ldY + g] = 0.0;
            a.gT0[g] = 0.0;
            for (int j = 0; j < 2 * a.R; ++j) a.rows[(long long)j * a.n + g] = 0.0;
          } else {
            s = nrec - 1;
#pragma unroll
            for (int k = 0; k < K; ++k) lam[k] = a.gY[k * a.ldY + g];
            lam[K] = a.gT[g];
            invp = 1.0 / a.p[g];
            active = true;
            need = false;
            if constexpr (SELF) {
              ncell = nrec;
              cs = ckpt_stride(nrec, a.ckpt_S);
              Ck = a.ckpt + g * (long long)a.ckpt_S * (N + 3);
              replaying = false;
              if (cs > 1) begin_replay(s / cs);
            } else {
              off = a.offsets[g];
            }
          }
        }
      }
    }
    // the CTA's warps stay in step (one barrier an iteration), so that they share the
    // instruction cache: the loop body is several times its size
    if (!__syncthreads_or(active ? 1 : 0)) break;
    if constexpr (SELF) {
      if (active && replaying) {
        // ---- one attempt of the segment's replay (the record pass's arithmetic) ----
        double ry[N], yn[N], err, unused[4][N];
#pragma unroll
        for (int i = 0; i < N; ++i) ry[i] = Rp[i * nl];
        const double rt = Rp[N * nl];
        const double hatt = fmin(Rp[(N + 1) * nl], a.dt - rt);
        const bool rrej = Rp[(N + 2) * nl] != 0.0;
        int rcnt = (int)Rp[(N + 3) * nl];
        const int rtarget = (int)Rp[(N + 4) * nl];
        const double ratt = Rp[(N + 5) * nl] + 1.0;
        Rp[(N + 5) * nl] = ratt;
        bool finite;
        unsigned long long swaps;
        const Opts o{a.opt.rtol, a.opt.atol, a.opt.h_min, a.opt.facmax, a.opt.facmin, a.opt.safety,
                     a.opt.max_substeps, 0};
        if (ratt > (double)o.max_substeps ||
            !adj_attempt<K, RX>(m, L, invp, ry, hatt, o, yn, &err, &finite, &swaps, &unused[0][0])) {
          fail_cell(RDE_CELL_ADJ_MISMATCH);
        } else if (finite && err <= 1.0) {
#pragma unroll
          for (int i = 0; i < N; ++i) Sg[(rcnt * (N + 1) + i) * nl] = ry[i];
          Sg[(rcnt * (N + 1) + N) * nl] = hatt;
          ++rcnt;
#pragma unroll
          for (int i = 0; i < N; ++i) Rp[i * nl] = yn[i];
          Rp[N * nl] = rt + hatt;
          Rp[(N + 1) * nl] = hatt * step_factor<kMethodRodas3>(err, finite, true, rrej, o);
          Rp[(N + 2) * nl] = 0.0;
          Rp[(N + 3) * nl] = (double)rcnt;
          if (rcnt == rtarget) {
            replaying = false;
            // the replayed segment must end on the next checkpoint, bit for bit
            const int jn = (seg0 + rcnt) / cs;
            if (seg0 + rcnt < ncell) {
              const double* en = Ck + (long long)jn * (N + 3);
              bool same = en[N] == rt + hatt;
#pragma unroll
              for (int i = 0; i < N; ++i) same = same && (__double_as_longlong(en[i]) == __double_as_longlong(yn[i]));
              if (!same) fail_cell(RDE_CELL_ADJ_MISMATCH);
            }
          }
        } else {
          const double hn = hatt * step_factor<kMethodRodas3>(err, finite, false, rrej, o);
          Rp[(N + 1) * nl] = hn;
          Rp[(N + 2) * nl] = 1.0;
          if (hn < o.hmin) fail_cell(RDE_CELL_ADJ_MISMATCH);
        }
        continue;
      }
    }
    if (active) {
      double y[N];
      const double* rec;
      int rstride = N + 1;
      if constexpr (SELF) {
        if (cs == 1) {
          rec = Ck + (long long)s * (N + 3);
          rstride = 1;
        } else {
          rec = Sg + (long long)(s - seg0) * (N + 1) * nl;
          rstride = 0;
        }
      } else {
        rec = a.pool + (off + s) * (N + 1);
        rstride = 1;
      }
      double h;
      if (rstride == 0) {
#pragma unroll
        for (int i = 0; i < N; ++i) y[i] = rec[i * nl];
        h = rec[N * nl];
      } else {
#pragma unroll
        for (int i = 0; i < N; ++i) y[i] = rec[i];
        h = (SELF) ? rec[N + 2] : rec[N];
      }
      const double invh = 1.0 / h;
      unsigned long long piv;
      if (a.stages) {
        // ---- the stages of this step from its checkpoint ----
        const double* cp = a.stages + (off + s) * (long long)(N * N + 4 * N + 1);
#pragma unroll 4
        for (int e = 0; e < N * N; ++e) L[S::MX + e] = cp[e];
        piv = (unsigned long long)__double_as_longlong(cp[N * N]);
#pragma unroll
        for (int i = 0; i < 4 * N; ++i) U[i * nl] = cp[N * N + 1 + i];
      } else {
        // ---- recompute the stages of this step ----
#pragma unroll
        for (int i = 0; i < N; ++i) L[S::ARG + i] = y[i];
        const MixState ms = RhsOf<RX>::template eval<K, true, S>(m, L, invp);
        double f0[N];
#pragma unroll
        for (int i = 0; i < N; ++i) f0[i] = L[S::VEC + i];
        constexpr unsigned IN = RX::kInert;
        assemble_matrix<K, S, IN, true>(m, L, y[K], ms, 1.0 / (kGamma * h), invp);
        unsigned long long perm;
        lu_factor<K, IN>(L, piv, perm);
        double u1[N], u2[N], u3[N], u4[N];
        lu_solve<K, IN, S>(L, perm, u1);
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (live<IN>(i)) L[S::VEC + i] = f0[i] + (kC21 * invh) * u1[i];
        lu_solve<K, IN, S>(L, perm, u2);
#pragma unroll
        for (int i = 0; i < N; ++i) u3[i] = u4[i] = 0.0;
        // stages 3 and 4 share one body, as in rosenbrock_attempt
#pragma unroll 1
        for (int st = 0; st < 2; ++st) {
#pragma unroll
          for (int i = 0; i < N; ++i) L[S::ARG + i] = live<IN>(i) ? y[i] + 2.0 * u1[i] + u3[i] : y[i];
          RhsOf<RX>::template eval<K, false, S>(m, L, invp);
          const double c3 = st ? kC43 : 0.0;
#pragma unroll
          for (int i = 0; i < N; ++i)
            if (live<IN>(i)) L[S::VEC + i] += invh * (u1[i] - u2[i] + c3 * u3[i]);
          double v[N];
          lu_solve<K, IN, S>(L, perm, v);
#pragma unroll
          for (int i = 0; i < N; ++i) {
            u3[i] = st ? u3[i] : v[i];
            u4[i] = st ? v[i] : u4[i];
          }
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
          U[(0 * N + i) * nl] = u1[i];
          U[(1 * N + i) * nl] = u2[i];
          U[(2 * N + i) * nl] = u3[i];
          U[(3 * N + i) * nl] = u4[i];
        }
      }
      auto solve_t = [&] { lu_solve_t<K, RX::kInert>(L, piv, kGamma * h); };
      // ---- adjoint of the stages: ybar = lam; ubar4 = lam, ubar3 = lam, ubar2 = 0, ubar1 = 2 lam ----
      double yb[N], ub1[N], ub2[N], ub3[N], g[N], arg[N], w[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        yb[i] = lam[i];
        ub1[i] = 2.0 * lam[i];
        ub2[i] = 0.0;
        ub3[i] = lam[i];
        L[S::VEC + i] = lam[i];
      }
      // stage 4: r4 = f(y + 2 u1 + u3) + (u1 - u2 + c43 u3)/h
      solve_t();
#pragma unroll
      for (int i = 0; i < N; ++i) {
        w[i] = L[S::VEC + i];
        W[(3 * N + i) * nl] = w[i];
        arg[i] = y[i] + 2.0 * U[(0 * N + i) * nl] + U[(2 * N + i) * nl];
      }
      jtw_value<K, RX>(m, L, invp, arg, w, g, thA, thE, nl);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        yb[i] += g[i];
        ub1[i] += 2.0 * g[i] + invh * w[i];
        ub2[i] -= invh * w[i];
        ub3[i] += g[i] + (kC43 * invh) * w[i];
        L[S::VEC + i] = ub3[i];
      }
      // stage 3: r3 = f(y + 2 u1) + (u1 - u2)/h
      solve_t();
#pragma unroll
      for (int i = 0; i < N; ++i) {
        w[i] = L[S::VEC + i];
        W[(2 * N + i) * nl] = w[i];
        arg[i] = y[i] + 2.0 * U[(0 * N + i) * nl];
      }
      jtw_value<K, RX>(m, L, invp, arg, w, g, thA, thE, nl);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        yb[i] += g[i];
        ub1[i] += 2.0 * g[i] + invh * w[i];
        ub2[i] -= invh * w[i];
        L[S::VEC + i] = ub2[i];
      }
      // stage 2: r2 = f(y) + (c21/h) u1
      solve_t();
#pragma unroll
      for (int i = 0; i < N; ++i) {
        w[i] = L[S::VEC + i];
        W[(1 * N + i) * nl] = w[i];
        ub1[i] += (kC21 * invh) * w[i];
        L[S::VEC + i] = ub1[i];
      }
      // stage 1: r1 = f(y)
      solve_t();
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const double w1 = L[S::VEC + i];
        W[(0 * N + i) * nl] = w1;
        w[i] = w1 + W[(1 * N + i) * nl];   // f(y) enters stages 1 and 2
      }
      jtw_value<K, RX>(m, L, invp, y, w, g, thA, thE, nl);
#pragma unroll
      for (int i = 0; i < N; ++i) yb[i] += g[i];
      // ---- M = I/(gamma h) - J(y): terms grad (w_i^T J(y) u_i) ----
      if constexpr (ND > 1) {
        // ND stages per evaluation, sharing its primal part
#pragma unroll 1
        for (int st = 0; st < 4; st += ND) hvp_sum<K, ND, RX>(m, L, invp, y, U, W, st, nl, yb, thA, thE, nl);
      } else {
        // one dual-number evaluation per stage
#pragma unroll 1
      for (int st = 0; st < 4; ++st) {
        Dual yd[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          yd[i] = mk(y[i], U[(st * N + i) * nl]);
          w[i] = W[(st * N + i) * nl];
        }
        jtw<K, RX>(m, L, 0, invp, yd, w, g, thA, thE, nl);
#pragma unroll
        for (int i = 0; i < N; ++i) yb[i] += g[i];
      }
      }
#pragma unroll
      for (int i = 0; i < N; ++i) lam[i] = yb[i];
      if (--s < 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) a.gY0[k * a.ldY + cell] = lam[k];
        a.gT0[cell] = lam[K];
        for (int j = 0; j < 2 * a.R; ++j) a.rows[(long long)j * a.n + cell] = thA[(long long)j * nl];
        active = false;
      } else if constexpr (SELF) {
        if (cs > 1 && s < seg0) begin_replay(s / cs);
      }
    }
  }
}

}  // namespace rde
