// Per-voxel and per-wave-vector steps of the 2D FP32 passes, shared by the row and Green passes
// (hom_fast2d.cu) and by the on-chip solver of small grids (hom_resident2d.cu).
#pragma once

#include "hom_em.cuh"
#include "hom_fast2d.h"
#include "hom_fastfft.cuh"
#include "hom_solve_args.cuh"

namespace hom {
namespace {

constexpr int NP = 3;  // lane pairs per position (2D Mandel components)

// ------------------------------------------------------------------ state layout
// The mixed-domain state of a cell (eps buffers and tau) is tiled by kx pairs: for load l, pair
// p = kx / 2 (T = Hp / 2 pairs) and row y, the three components are float4 lane pairs
// (re(kx = 2p), re(2p + 1), im(2p), im(2p + 1)).  A Green-pass task reads and writes one
// contiguous tile of n rows; a row-pass task reads 4 consecutive rows of every pair (192 bytes).
__device__ __forceinline__ size_t tile_index(const CellDev& c, int n, int l, int p, int y) {
  return (size_t)c.ws_off / 2 + (((size_t)l * (c.Hp / 2) + p) * n + y) * NP;
}

constexpr uint32_t kLabel8Mixed = 255;  // one-byte label of a mixed voxel

// Per local phase the pure-voxel constants: (lam - lam0, 2 mu - 2 mu0), for the output pass with a zero
// reference medium; EM (Eyre-Milton scheme): W = (c - c0)(c + c0)^-1 instead, and (c + c0)^-1 in sinv.
template <bool OUT, bool EM>
__device__ __forceinline__ void phase_constants(const SolveArgs& A, const CellDev& c, const CellConst<float>& cc,
                                                float2* sph, float2* sinv, int nthr) {
  const float lam0 = OUT ? 0.f : cc.lam0, mu2_0 = OUT ? 0.f : cc.mu2;
  for (int i = threadIdx.x; i < c.nph; i += nthr) {
    const float* pc = A.phase_c32 + (size_t)__ldg(A.cell_phases + c.ph_off + i) * 6;
    const float lam = __ldg(pc + 1);
    const float mu2 = __ldg(pc) - lam;
    sph[i] = make_float2(lam - lam0, mu2 - mu2_0);
    if (EM) {
      // (c + c0)^-1: volumetric eigenvalue 2 (lam + lam0) + (2 mu + 2 mu0), deviatoric 2 mu + 2 mu0
      const double l = (double)lam, m2 = (double)mu2, l0 = c.lam0, m20 = 2.0 * c.mu0;
      const double ms2 = m2 + m20, ks = 2.0 * (l + l0) + ms2;
      sinv[i] = make_float2((float)((1.0 / ks - 1.0 / ms2) * 0.5), (float)(1.0 / ms2));
      if (!OUT) {  // W = (c - c0)(c + c0)^-1: volumetric (k - k0)/(k + k0), deviatoric (2mu - 2mu0)/(2mu + 2mu0)
        const double aK = (m2 - m20) / ms2, aJ = (2.0 * (l - l0) + (m2 - m20)) / ks;
        sph[i] = make_float2((float)(0.5 * (aJ - aK)), (float)aK);
      }
    }
  }
}

// Constitutive update of the four voxels of one position (lanes (x, y, z, w) of a float4 are rows (0, 2, 1,
// 3)): lab holds their one-byte labels (the local phase index of a pure voxel, or kLabel8Mixed: full label
// read from the material, which also covers any voxel whose phase is not in the cell's list), e the
// strains (EM: the states u, turned into strains where the voxels are mixed or OUT), o the result tau
// (OUT: the stress).
template <bool OUT, bool SRC, bool EM>
__device__ __forceinline__ void tau_point(const SolveArgs& A, const CellDev& c, const FastPlanDev& fp, const float2* sph,
                                          const float2* sinv, const CellConst<float>& cc, int nr, int y0, int l, int pos,
                                          uint32_t (&lab)[kFastRows], float4 (&e)[NP], float4 (&o)[NP]) {
  // OUT: sigma = c~ : eps, i.e. the update with a zero reference medium
  const float lam0 = OUT ? 0.f : cc.lam0, mu2_0 = OUT ? 0.f : cc.mu2;
  const float lam_em = cc.lam0, mu2_em = cc.mu2;  // EM: the reference medium of (c + c0)^-1, also when OUT
  bool mixed = false;
#pragma unroll
  for (int r = 0; r < kFastRows; ++r) {
    // debug builds: a phase of the cell's list
    if (!HOM_CHECK(A, lab[r] == kLabel8Mixed || lab[r] < (uint32_t)c.nph, lab[r])) lab[r] = 0;
    mixed |= lab[r] == kLabel8Mixed;
  }
  uint32_t loc[kFastRows];  // the one-byte labels (EM: per-phase constants of pure voxels)
#pragma unroll
  for (int r = 0; r < kFastRows; ++r) loc[r] = lab[r];
  if (mixed) {  // full labels: the material's for mixed voxels, global phases for the others
    const int x = __ldg(fp.iperm + pos);
#pragma unroll
    for (int r = 0; r < kFastRows; ++r)
      lab[r] = lab[r] == kLabel8Mixed ? __ldg(A.label + c.vox_off + (size_t)(y0 + r) * c.n + x)
                                      : (uint32_t)__ldg(A.cell_phases + c.ph_off + lab[r]);
  }
  if (EM && (OUT || mixed)) {
    // e holds u: eps = (c~ + c0)^-1 u, per voxel (mixed: the per-call table; pure: in closed form)
    float ev[NP][kFastRows];
#pragma unroll
    for (int r = 0; r < kFastRows; ++r) {
      float u[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) u[k] = r == 0 ? e[k].x : r == 1 ? e[k].z : r == 2 ? e[k].y : e[k].w;
      if (mixed && (lab[r] & HOM_MIXED_BIT)) {
        const float* M = static_cast<const float*>(A.em_minv) + (size_t)(lab[r] & ~HOM_MIXED_BIT) * 6;
        ev[0][r] = __ldg(M) * u[0] + __ldg(M + 1) * u[1] + __ldg(M + 2) * u[2];
        ev[1][r] = __ldg(M + 1) * u[0] + __ldg(M + 3) * u[1] + __ldg(M + 4) * u[2];
        ev[2][r] = __ldg(M + 2) * u[0] + __ldg(M + 4) * u[1] + __ldg(M + 5) * u[2];
      } else {
        float2 d;
        if (loc[r] == kLabel8Mixed) {  // a pure voxel whose phase is not in the cell's list (rare)
          const float* pc = A.phase_c32 + (size_t)lab[r] * 6;
          const float l = __ldg(pc + 1), m2 = __ldg(pc) - l;
          const float ms2 = m2 + mu2_em, ks = 2.f * (l + lam_em) + ms2;
          d = make_float2((1.f / ks - 1.f / ms2) * 0.5f, 1.f / ms2);
        } else {
          d = sinv[loc[r]];
        }
        const float tr = u[0] + u[1];
        ev[0][r] = d.y * u[0] + d.x * tr;
        ev[1][r] = d.y * u[1] + d.x * tr;
        ev[2][r] = d.y * u[2];
      }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) e[k] = make_float4(ev[k][0], ev[k][2], ev[k][1], ev[k][3]);
  }
  if (!mixed) {
    // pure voxels: tau = (lam - lam0) tr(eps) I + (2 mu - 2 mu0) eps
    float dl[kFastRows], dm[kFastRows];
#pragma unroll
    for (int r = 0; r < kFastRows; ++r) {
      const float2 d = sph[lab[r]];
      dl[r] = d.x;
      dm[r] = d.y;
    }
    const float2 dl_lo = make_float2(dl[0], dl[2]), dl_hi = make_float2(dl[1], dl[3]);
    const float2 dm_lo = make_float2(dm[0], dm[2]), dm_hi = make_float2(dm[1], dm[3]);
    const float2 tr_lo = add2(make_float2(e[0].x, e[0].y), make_float2(e[1].x, e[1].y));
    const float2 tr_hi = add2(make_float2(e[0].z, e[0].w), make_float2(e[1].z, e[1].w));
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      float2 lo = mul2(dm_lo, make_float2(e[k].x, e[k].y));
      float2 hi = mul2(dm_hi, make_float2(e[k].z, e[k].w));
      if (k < 2) {
        lo = fma2(dl_lo, tr_lo, lo);
        hi = fma2(dl_hi, tr_hi, hi);
      }
      o[k] = make_float4(lo.x, lo.y, hi.x, hi.y);
    }
  } else {
    float out[NP][kFastRows];
#pragma unroll
    for (int r = 0; r < kFastRows; ++r) {
      float ev[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) ev[k] = r == 0 ? e[k].x : r == 1 ? e[k].z : r == 2 ? e[k].y : e[k].w;
      float C[6];
      const float* src = (lab[r] & HOM_MIXED_BIT) ? A.mixed_c32 + (size_t)(lab[r] & ~HOM_MIXED_BIT) * 6
                                                  : A.phase_c32 + (size_t)lab[r] * 6;
#pragma unroll
      for (int q = 0; q < 6; ++q) C[q] = __ldg(src + q);
      const float tr0 = ev[0] + ev[1];
      // packed upper triangle of the 3x3 Mandel matrix: (00, 01, 02, 11, 12, 22)
      const float sg0 = C[0] * ev[0] + C[1] * ev[1] + C[2] * ev[2];
      const float sg1 = C[1] * ev[0] + C[3] * ev[1] + C[4] * ev[2];
      const float sg2 = C[2] * ev[0] + C[4] * ev[1] + C[5] * ev[2];
      out[0][r] = sg0 - (mu2_0 * ev[0] + lam0 * tr0);
      out[1][r] = sg1 - (mu2_0 * ev[1] + lam0 * tr0);
      out[2][r] = sg2 - mu2_0 * ev[2];
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) o[k] = make_float4(out[k][0], out[k][2], out[k][1], out[k][3]);
  }
  if constexpr (SRC) {
    // adjoint solve: the stiffness acts on w - S, so tau = (c~ - c0) : w - c~ : S, with the
    // source S (real field, solver output layout) read at the rows' voxels
    const int x = __ldg(fp.iperm + pos);
    const float* S = static_cast<const float*>(A.src) + c.fld_off + (size_t)l * NP * c.nv + (size_t)y0 * c.n + x;
    float cs[NP][kFastRows];
#pragma unroll
    for (int r = 0; r < kFastRows; ++r) {
#pragma unroll
      for (int k = 0; k < NP; ++k) cs[k][r] = 0.f;
      if (r >= nr) continue;
      const uint32_t L = mixed ? lab[r] : (uint32_t)__ldg(A.cell_phases + c.ph_off + lab[r]);
      const float* C = (L & HOM_MIXED_BIT) ? A.mixed_c32 + (size_t)(L & ~HOM_MIXED_BIT) * 6 : A.phase_c32 + (size_t)L * 6;
      float sv[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) sv[k] = __ldg(S + (size_t)k * c.nv + (size_t)r * c.n);
      cs[0][r] = __ldg(C) * sv[0] + __ldg(C + 1) * sv[1] + __ldg(C + 2) * sv[2];
      cs[1][r] = __ldg(C + 1) * sv[0] + __ldg(C + 3) * sv[1] + __ldg(C + 4) * sv[2];
      cs[2][r] = __ldg(C + 2) * sv[0] + __ldg(C + 4) * sv[1] + __ldg(C + 5) * sv[2];
    }
#pragma unroll
    for (int k = 0; k < NP; ++k)
      o[k] = make_float4(o[k].x - cs[k][0], o[k].y - cs[k][2], o[k].z - cs[k][1], o[k].w - cs[k][3]);
  }
}

// Green step of one kx pair (lanes A, B = columns kx0, kx0 + 1) of one load: constants, and the Kahan sums
// (value, lost low part, per lane) of the equilibrium residuals of the points given to it.
struct GreenPair {
  float2 mu0, lpm, ratio, inv_mu0, X, X2, wgt;
  float inv_nv, nyq;
  bool even, deadA, deadB, first;
  const double* Eld;
  float2 r2s, r2c, rns, rnc;

  __device__ __forceinline__ GreenPair(const SolveArgs& A, const CellDev& c, const FastPlanDev& fp, int kx0, int cl) {
    CellConst<float> cc;
    cell_const(c, cc);
    mu0 = f2(0.5f * cc.mu2);
    lpm = f2(cc.lpm);
    ratio = f2(cc.ratio);
    inv_mu0 = f2(cc.inv_mu0);
    inv_nv = cc.inv_nv;
    // even grids: a wave vector with a Nyquist component (n/2) has no conjugate partner in the spectrum
    // of a real field; its strain is set to zero and it is left out of the residual
    even = !(c.n & 1);
    nyq = even ? __ldg(fp.xinat + c.n / 2) : 0.f;
    Eld = A.E + (size_t)cl * NP;
    r2s = r2c = rns = rnc = make_float2(0.f, 0.f);
    set_pair(c.n, fp, kx0);
  }
  __device__ __forceinline__ void set_pair(int N, const FastPlanDev& fp, int kx0) {
    const bool hasB = kx0 + 1 < N / 2 + 1;
    X = make_float2(__ldg(fp.xinat + kx0), hasB ? __ldg(fp.xinat + kx0 + 1) : 0.f);
    X2 = mul2(X, X);
    deadA = even && 2 * kx0 == N;
    deadB = !hasB || (even && 2 * kx0 + 2 == N);
    wgt = make_float2(deadA ? 0.f : kx0 == 0 ? 1.f : 2.f, deadB ? 0.f : 2.f);
    first = kx0 == 0;
  }

  // eps_hat = -sym(xi (x) g) / N_v of one position (k = 0 aside)
  __device__ __forceinline__ void strain(const P2& W0, const P2& W1, float2 Y, P2& E0, P2& E1, P2& E2) const {
    const float rs2 = 0.707106781186547524400844362105f;
    const float2 nx = mul2(X, f2(-inv_nv)), ny = mul2(Y, f2(-inv_nv));
    const float2 ns = f2(-rs2 * inv_nv);
    E0 = P2{mul2(nx, W0.re), mul2(nx, W0.im)};
    E1 = P2{mul2(ny, W1.re), mul2(ny, W1.im)};
    E2 = P2{mul2(ns, fma2(X, W1.re, mul2(Y, W0.re))), mul2(ns, fma2(X, W1.im, mul2(Y, W0.im)))};
  }

  // eps_hat of one position from its g (the two float4 that point() stored), k = 0 included
  __device__ __forceinline__ void spectrum(float4* T, float y, bool pos0, const float4& ga, const float4& gb) const {
    const P2 W0{make_float2(ga.x, gb.x), make_float2(ga.y, gb.y)}, W1{make_float2(ga.z, gb.z), make_float2(ga.w, gb.w)};
    P2 E0, E1, E2;
    strain(W0, W1, f2(y), E0, E1, E2);
    if (first && pos0) {
      E0.re.x = (float)Eld[0];
      E1.re.x = (float)Eld[1];
      E2.re.x = (float)Eld[2];
    }
    T[0] = stp(E0);
    T[1] = stp(E1);
    T[2] = stp(E2);
  }

  // One position: T (three lane pairs of tau_hat, overwritten by the new eps_hat), wave number y of the
  // last axis, its g (gin; the new one goes to gout).
  __device__ __forceinline__ void point(float4* T, float y, bool pos0, const float4 (&gin)[2], float4* gout) {
    const float4 ga = gin[0], gbv = gin[1];
    const float2 Y = f2(y);
    const P2 T0 = ldp(T[0]), T1 = ldp(T[1]), T2 = ldp(T[2]);
    const P2 G0{make_float2(ga.x, gbv.x), make_float2(ga.y, gbv.y)};
    const P2 G1{make_float2(ga.z, gbv.z), make_float2(ga.w, gbv.w)};
    const float rs2 = 0.707106781186547524400844362105f;
    // v = tau_hat . xi (tau_01 = T2 / sqrt 2)
    const P2 T01 = scale(rs2, T2);
    const P2 V0{fma2(Y, T01.re, mul2(X, T0.re)), fma2(Y, T01.im, mul2(X, T0.im))};
    const P2 V1{fma2(Y, T1.re, mul2(X, T01.re)), fma2(Y, T1.im, mul2(X, T01.im))};
    const float2 q2 = fma2(Y, Y, X2);
    const P2 XG{fma2(Y, G1.re, mul2(X, G0.re)), fma2(Y, G1.im, mul2(X, G0.im))};
    const P2 XV{fma2(Y, V1.re, mul2(X, V0.re)), fma2(Y, V1.im, mul2(X, V0.im))};
    // residual of the current iterate: r = tau_hat xi - K0 g, K0 g = mu0 q2 g + (lam0 + mu0) xi (xi . g)
    const float2 mq = mul2(mu0, q2);
    const float2 lx = mul2(lpm, X), ly = mul2(lpm, Y);
    const P2 R0{sub2(sub2(V0.re, mul2(mq, G0.re)), mul2(lx, XG.re)), sub2(sub2(V0.im, mul2(mq, G0.im)), mul2(lx, XG.im))};
    const P2 R1{sub2(sub2(V1.re, mul2(mq, G1.re)), mul2(ly, XG.re)), sub2(sub2(V1.im, mul2(mq, G1.im)), mul2(ly, XG.im))};
    float2 r2 = mul2(R0.re, R0.re);
    r2 = fma2(R0.im, R0.im, r2);
    r2 = fma2(R1.re, R1.re, r2);
    r2 = fma2(R1.im, R1.im, r2);
    const bool k0 = first && pos0;  // k = 0: eps_hat(0) = E, g = 0, no residual
    const bool dead = even && Y.x == nyq;  // the last axis at Nyquist
    const float2 iq = make_float2(k0 || deadA || dead ? 0.f : __fdividef(1.f, q2.x),
                                  deadB || dead ? 0.f : __fdividef(1.f, q2.y));
    // g' = K0^-1 (tau_hat xi), eps_hat' = -sym(xi (x) g') / N_v
    const float2 imq = mul2(inv_mu0, iq);
    const float2 rq = mul2(ratio, iq);
    const float2 rx = mul2(rq, X), ry = mul2(rq, Y);
    const P2 W0{mul2(imq, sub2(V0.re, mul2(rx, XV.re))), mul2(imq, sub2(V0.im, mul2(rx, XV.im)))};
    const P2 W1{mul2(imq, sub2(V1.re, mul2(ry, XV.re))), mul2(imq, sub2(V1.im, mul2(ry, XV.im)))};
    P2 E0, E1, E2;
    strain(W0, W1, Y, E0, E1, E2);
    float4 gna = make_float4(W0.re.x, W0.im.x, W1.re.x, W1.im.x);
    const float4 gnb = make_float4(W0.re.y, W0.im.y, W1.re.y, W1.im.y);
    float2 wr = dead ? make_float2(0.f, 0.f) : wgt;
    if (k0) {
      E0.re.x = (float)Eld[0]; E0.im.x = 0.f;
      E1.re.x = (float)Eld[1]; E1.im.x = 0.f;
      E2.re.x = (float)Eld[2]; E2.im.x = 0.f;
      gna = make_float4(0.f, 0.f, 0.f, 0.f);
      wr.x = 0.f;
    }
    T[0] = stp(E0);
    T[1] = stp(E1);
    T[2] = stp(E2);
    gout[0] = gna;
    gout[1] = gnb;
    // Kahan accumulation of wgt * r2 and wgt * r2 / q2, lane by lane
    const float2 a1 = mul2(wr, r2), a2 = mul2(a1, iq);
    {
      const float2 yv = sub2(a1, r2c), tv = add2(r2s, yv);
      r2c = sub2(sub2(tv, r2s), yv);
      r2s = tv;
    }
    {
      const float2 yv = sub2(a2, rnc), tv = add2(rns, yv);
      rnc = sub2(sub2(tv, rns), yv);
      rns = tv;
    }
  }

  // the two lanes of each sum (compensated pairs) as one compensated pair
  __device__ __forceinline__ void sums(Acc<float> (&vv)[2]) const {
    vv[0].s = r2s.x;
    vv[0].c = r2c.x;
    vv[0].add(r2s.y);
    vv[0].add(-r2c.y);
    vv[1].s = rns.x;
    vv[1].c = rnc.x;
    vv[1].add(rns.y);
    vv[1].add(-rnc.y);
  }
};

// The same for the Eyre-Milton scheme, lane by lane through em_core (hom_em.cuh).
struct GreenPairEm {
  CellConst<float> cc;
  float nvT, a0, inv_mu2_0, X[2], nyq;
  bool first;
  const double* Eld;
  __device__ __forceinline__ GreenPairEm(const SolveArgs& A, const CellDev& c, const FastPlanDev& fp, int kx0, const double* E) {
    const int N = c.n;
    // Nyquist bins of an even grid (a wave number no odd grid has)
    nyq = (N & 1) ? -1.f : __ldg(fp.xinat + N / 2);
    cell_const(c, cc);
    nvT = (float)c.nv;
    a0 = cc.lam0 / (cc.mu2 + 2.f * cc.lam0);
    inv_mu2_0 = 0.5f * cc.inv_mu0;
    Eld = E;
    set_pair(N, fp, kx0);
    (void)A;
  }
  __device__ __forceinline__ void set_pair(int N, const FastPlanDev& fp, int kx0) {
    X[0] = __ldg(fp.xinat + kx0);
    X[1] = kx0 + 1 < N / 2 + 1 ? __ldg(fp.xinat + kx0 + 1) : 0.f;
    first = kx0 == 0;
  }
  // Lane h of one position: T its lane pairs, uin u_hat of the current iterate, uout the new one.
  __device__ __forceinline__ void point(float* T, int h, float y, bool pos0, const float2* uin, float2* uout,
                                        Acc<float> (&acc)[3]) const {
    float2 th[NP], uh[NP], un[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      th[k] = make_float2(T[4 * k + h], T[4 * k + 2 + h]);  // (re A, re B, im A, im B)
      uh[k] = uin[k];
    }
    const float xi[2] = {h ? X[1] : X[0], y};
    em_core<float, 2>(th, uh, un, xi, h == 0 && first && pos0, xi[0] == nyq || xi[1] == nyq,
                      (h == 0 && first) || xi[0] == nyq, nvT, cc.inv_nv, cc.lam0, cc.mu2, a0, inv_mu2_0, cc.inv_mu0,
                      cc.ratio, Eld, acc[0], acc[1], acc[2]);
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      T[4 * k + h] = un[k].x;
      T[4 * k + 2 + h] = un[k].y;
      uout[k] = un[k];
    }
  }
};

}  // namespace
}  // namespace hom
