// Basic fixed-point scheme of section 2 (eqs. 1-a, 1-b, 2) for a batch of cells x load cases.
//
// State between passes lives in HBM in a "mixed" representation: transformed along x (half
// spectrum kx = 0..(n-1)/2, rows padded to Hp entries), real along y (and z); layout
// [load][z][y][kx][component] complex per cell.  One iteration (2D) is two passes:
//   row pass   : inverse x-DFT of eps (pairs of real rows packed into one complex line),
//                sigma = c~ : eps, FP64 partial sums of sigma, tau = sigma - c0 : eps,
//                forward x-DFT of tau (eq. 1-b)
//   Green pass : forward y-DFT of tau, then per wave vector xi on J (eq. 2):
//                   r = tau_hat . xi - K0(xi) g      (= sigma_hat . xi: equilibrium residual)
//                   g' = K0(xi)^-1 (tau_hat . xi)    eps_hat' = -sym(xi (x) g') (k != 0)
//                   eps_hat'(0) = E
//                then the inverse y-DFT, written to the other eps buffer.
// g is the displacement-like vector of the current iterate (eps_hat = -sym(xi (x) g)); keeping
// it lets the Green pass evaluate the equilibrium residual of the current iterate from tau_hat
// alone.  In 3D the y transforms are separate passes (forward before, inverse after the
// z-direction Green pass).  A small control kernel reduces the FP64 partial sums per
// (cell, load), applies the stopping rule and deactivates finished load cases; later passes
// skip inactive ones.
#define HOM_FILE_ID 1
#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "hom_internal.h"
#include "hom_plan.h"
#include "hom_solve_args.cuh"
#include "hom_em.cuh"
#include "hom_control.cuh"
#include "hom_fast2d.h"
#include "hom_cg.cuh"

namespace hom {
namespace {

template <typename T> __device__ __forceinline__ const T* mixed_tab(const SolveArgs& A);
template <> __device__ __forceinline__ const float* mixed_tab<float>(const SolveArgs& A) { return A.mixed_c32; }
template <> __device__ __forceinline__ const double* mixed_tab<double>(const SolveArgs& A) { return A.mixed_c64; }
template <typename T> __device__ __forceinline__ const T* phase_tab(const SolveArgs& A);
template <> __device__ __forceinline__ const float* phase_tab<float>(const SolveArgs& A) { return A.phase_c32; }
template <> __device__ __forceinline__ const double* phase_tab<double>(const SolveArgs& A) { return A.phase_c64; }

__device__ __forceinline__ void load_plan(const SolveArgs& A, int idx, Plan& sp) {
  if (threadIdx.x == 0) sp = A.plans[idx];
  __syncthreads();
}

// Shared-memory layout of the pass kernels: the length-n twiddle table, then the lines.
template <typename V>
__device__ __forceinline__ V* stage_twiddles(unsigned char* smem, const Plan& sp) {
  V* tw = reinterpret_cast<V*>(smem);
  const V* src = twiddles<V>(sp);
  for (int i = threadIdx.x; i < sp.n; i += blockDim.x) tw[i] = src[i];
  return tw;
}

// 1/x for |x| >= 4 pi^2 (no special values): the fast FP32 reciprocal (a few ulp) avoids the
// IEEE division sequence; FP64 keeps the correctly rounded division.
__device__ __forceinline__ float recip(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

template <typename T> __device__ __forceinline__ const T* xi_table(const Plan& p);
template <> __device__ __forceinline__ const float* xi_table<float>(const Plan& p) { return p.xi32; }
template <> __device__ __forceinline__ const double* xi_table<double>(const Plan& p) { return p.xi64; }
template <typename V> __device__ __forceinline__ const V* rot_table(const Plan& p);
template <> __device__ __forceinline__ const float2* rot_table<float2>(const Plan& p) { return p.rot32; }
template <> __device__ __forceinline__ const double2* rot_table<double2>(const Plan& p) { return p.rot64; }

// ------------------------------------------------------------------ row pass
// OUT = false: one iteration's row pass (eps -> tau).  OUT = true: final fields of the returned
// iterate (eps and sigma real, written to the output arrays), no forward transform.
// EM: the stored state is u = sigma + c0 : eps of the Eyre-Milton scheme; each voxel first solves
// (c~ + c0) : eps = u, and the row sums of sigma are (tau + u) / 2.
template <typename T, int DIM, bool OUT, int MAXR, bool EM = false>
__global__ void __launch_bounds__(kThreads) k_row(SolveArgs A) {
  using V = typename Cx<T>::V;
  constexpr int NC = DIM == 2 ? 3 : 6;
  constexpr int NS = DIM == 2 ? 6 : 21;
  HOM_DBG_POISON();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Plan sp;
  __shared__ int s_al[kMaxLoads], s_par[kMaxLoads], s_nal;
  const TaskR t = A.tR[blockIdx.x];
  const CellDev c = A.cells[t.cell];
  const int it = *A.it_dev;
  if (threadIdx.x == 0) {
    int nal = 0;
    for (int l = 0; l < A.L; ++l) {
      const int cl = t.cell * A.L + l;
      if (OUT || A.active[cl]) {
        s_al[nal] = l;
        s_par[nal] = OUT ? (A.iters[cl] & 1) : (it & 1);
        ++nal;
      }
    }
    s_nal = nal;
  }
  load_plan(A, c.plan, sp);
  const int nal = s_nal;
  if (nal == 0) return;
  const int n = c.n, H = c.H, Hp = c.Hp;
  const V* tw = stage_twiddles<V>(smem_raw, sp);
  V* s = reinterpret_cast<V*>(smem_raw) + n;
  const int nreal = t.nrows * nal * NC;
  const int nlines = (nreal + 1) >> 1;
  const size_t load_stride = (size_t)c.nrows * Hp * NC;
  const V zero = mk(T(0), T(0));
  // Real row q = (row, active load, component) -> element offset of its half spectrum at kx = 0;
  // the top bit carries the eps buffer parity of its load.
  long long* qbase = reinterpret_cast<long long*>(s + (size_t)nlines * n);
  // per real row: kx = 0 entry of the stored eps (the row mean) and of the transformed tau (the row sum)
  T* dc_eps = reinterpret_cast<T*>(qbase + nreal);
  T* dc_tau = dc_eps + nreal;
  for (int q = threadIdx.x; q < nreal; q += kThreads) {
    const int per_row = nal * NC;
    const int rl = q / per_row;
    const int rem = q - rl * per_row;
    const int la = rem / NC;
    const int comp = rem - la * NC;
    const long long off = (long long)(c.ws_off + (size_t)s_al[la] * load_stride + (size_t)(t.row0 + rl) * Hp * NC + comp);
    qbase[q] = off | ((long long)s_par[la] << 62);
  }
  __syncthreads();
  const long long kOffMask = (1LL << 62) - 1;

  // 1. two real rows per complex line, Hermitian-extended half spectra (four items per round so
  // that eight global loads are in flight per thread)
  {
    constexpr int U = 4;
    Iter2 it(threadIdx.x, kThreads, sp.div_h);
    while (it.a < nlines) {
      int line[U], kx[U];
      V a[U], b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        line[u] = it.a;
        kx[u] = it.b;
        a[u] = b[u] = zero;
        if (it.a < nlines) {
          const int q0 = 2 * it.a, q1 = q0 + 1;
          const long long b0 = qbase[q0];
          const size_t i0 = (b0 & kOffMask) + (size_t)it.b * NC;
          if (HOM_CHECK(A, i0 < A.n_ws, i0)) a[u] = static_cast<const V*>(A.eps[b0 >> 62])[i0];
          if (q1 < nreal) {
            const long long b1 = qbase[q1];
            const size_t i1 = (b1 & kOffMask) + (size_t)it.b * NC;
            if (HOM_CHECK(A, i1 < A.n_ws, i1)) b[u] = static_cast<const V*>(A.eps[b1 >> 62])[i1];
          }
        }
        it.next();
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (line[u] >= nlines) break;
        const int q0 = 2 * line[u], q1 = q0 + 1;
        V* z = s + (size_t)line[u] * n;
        if (kx[u] == 0) {
          z[0] = mk(a[u].x, b[u].x);
          dc_eps[q0] = a[u].x;
          if (q1 < nreal) dc_eps[q1] = b[u].x;
        } else {
          z[kx[u]] = mk(a[u].x - b[u].y, a[u].y + b[u].x);      // A + iB
          z[n - kx[u]] = mk(a[u].x + b[u].y, b[u].x - a[u].y);  // conj(A) + i conj(B)
        }
      }
    }
  }
  __syncthreads();
  // 2. inverse x-DFT (natural -> digit-reversed positions)
  fft_dif<false, MAXR, V, T>(s, nlines, n, sp, tw, threadIdx.x, kThreads);

  // 3. constitutive update at every grid point of the task's rows: the material is read once per
  // voxel for all loads; pure voxels use sigma = lam tr(eps) I + 2 mu eps, mixed ones the packed c~.
  CellConst<T> cc;
  cell_const(c, cc);
  const T lam0 = cc.lam0, mu2_0 = cc.mu2;
  for (Iter2 it(threadIdx.x, kThreads, sp.div_n); it.a < t.nrows; it.next()) {
    const int rl = it.a, x = it.b;
    const int pos = HOM_LDG(sp.perm + x);
    const size_t vox = (size_t)(t.row0 + rl) * n + x;
    if (!HOM_CHECK(A, c.vox_off + vox < A.n_lab, c.vox_off + vox)) continue;
    const uint32_t lab = HOM_LDG(A.label + c.vox_off + vox);
    const bool mixed = (lab & HOM_MIXED_BIT) != 0;
    T C[NS];
    T lam = T(0), mu2 = T(0);
    if (mixed) {
      const T* src = mixed_tab<T>(A) + (size_t)(lab & ~HOM_MIXED_BIT) * NS;
#pragma unroll
      for (int k = 0; k < NS; ++k) C[k] = HOM_LDG(src + k);
    } else {
      const T* src = phase_tab<T>(A) + (size_t)lab * NS;
      lam = HOM_LDG(src + 1);                 // c_01 = lambda
      mu2 = HOM_LDG(src) - lam;               // c_00 - c_01 = 2 mu
    }
    // EM, pure voxel: (c + c0)^-1 u = (u - a tr(u) I) / (2 mu + 2 mu0), a = lam_s / (2 mu_s + DIM lam_s)
    T em_inv2 = T(0), em_a = T(0);
    const T* em_m = nullptr;
    if (EM) {
      if (mixed) {
        em_m = static_cast<const T*>(A.em_minv) + (size_t)(lab & ~HOM_MIXED_BIT) * NS;
      } else {
        const T ls = lam + lam0, ms2 = mu2 + mu2_0;
        em_inv2 = T(1) / ms2;
        em_a = ls / (ms2 + T(DIM) * ls);
      }
    }
    for (int la = 0; la < nal; ++la) {
      const int l = s_al[la];
      T e[NC];
      const int q0 = (rl * nal + la) * NC;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int q = q0 + k;
        const V zz = s[(size_t)(q >> 1) * n + pos];
        e[k] = (q & 1) ? zz.y : zz.x;
      }
      if (EM) {  // e holds u: the strain of the iterate is (c~ + c0)^-1 : u
        T u[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) u[k] = e[k];
        if (mixed) {
#pragma unroll
          for (int I = 0; I < NC; ++I) {
            T acc_i = T(0);
#pragma unroll
            for (int J = 0; J < NC; ++J) acc_i += HOM_LDG(em_m + packed_index(NC, I, J)) * u[J];
            e[I] = acc_i;
          }
        } else {
          T tr = T(0);
#pragma unroll
          for (int k = 0; k < DIM; ++k) tr += u[k];
          const T atr = em_a * tr;
#pragma unroll
          for (int k = 0; k < NC; ++k) e[k] = em_inv2 * (u[k] - (k < DIM ? atr : T(0)));
        }
      }
      T ee[NC];  // strain the stiffness acts on: eps, or w - S in the adjoint solve
#pragma unroll
      for (int k = 0; k < NC; ++k) ee[k] = e[k];
      if (A.src) {
        const T* S = static_cast<const T*>(A.src) + c.fld_off + (size_t)l * NC * c.nv + vox;
#pragma unroll
        for (int k = 0; k < NC; ++k) ee[k] -= S[(size_t)k * c.nv];
      }
      T sg[NC];
      if (mixed) {
#pragma unroll
        for (int I = 0; I < NC; ++I) {
          T acc_i = T(0);
#pragma unroll
          for (int J = 0; J < NC; ++J) acc_i += C[packed_index(NC, I, J)] * ee[J];
          sg[I] = acc_i;
        }
      } else {
        T tr = T(0);
#pragma unroll
        for (int k = 0; k < DIM; ++k) tr += ee[k];
        const T ltr = lam * tr;
#pragma unroll
        for (int k = 0; k < NC; ++k) sg[k] = mu2 * ee[k] + (k < DIM ? ltr : T(0));
      }
      if (OUT) {
        const size_t base = c.fld_off + (size_t)l * NC * c.nv + vox;
        T* oe = static_cast<T*>(A.out_eps);
        T* os = static_cast<T*>(A.out_sig);
        if (HOM_CHECK(A, base + (size_t)(NC - 1) * c.nv < A.n_fld, base + (size_t)(NC - 1) * c.nv))
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            if (oe) oe[base + (size_t)k * c.nv] = e[k];
            if (os) os[base + (size_t)k * c.nv] = sg[k];
          }
      } else {
        T tr = T(0);
#pragma unroll
        for (int k = 0; k < DIM; ++k) tr += e[k];
        const T ltr0 = lam0 * tr;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          const T tau = sg[k] - (mu2_0 * e[k] + (k < DIM ? ltr0 : T(0)));
          const int q = q0 + k;
          V* zz = s + (size_t)(q >> 1) * n + pos;
          if (q & 1) zz->y = tau; else zz->x = tau;
        }
      }
    }
  }
  if (OUT) {
    if (threadIdx.x == 0)
      atomicAdd(A.bytes + HOM_K_OUTPUT,
                (unsigned long long)((size_t)nal * t.nrows * NC * (H * sizeof(V) + 2 * (size_t)n * sizeof(T)) +
                                     (size_t)t.nrows * n * 4));
    return;
  }
  __syncthreads();
  // 4. forward x-DFT (digit-reversed -> natural)
  fft_dit<true, MAXR, V, T>(s, nlines, n, sp, tw, threadIdx.x, kThreads);
  // 5. split the two real rows of each line and store the half spectra of tau
  V* tau = static_cast<V*>(A.tau);
  for (Iter2 it(threadIdx.x, kThreads, sp.div_h); it.a < nlines; it.next()) {
    const int line = it.a, kx = it.b;
    const V* z = s + (size_t)line * n;
    const V zk = z[kx];
    const V zm = z[kx == 0 ? 0 : n - kx];
    const V a = mk(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));   // (Z[k] + conj Z[n-k]) / 2
    const V b = mk(T(0.5) * (zk.y + zm.y), T(0.5) * (zm.x - zk.x));   // (Z[k] - conj Z[n-k]) / 2i
    const int q0 = 2 * line;
    const size_t i0 = (qbase[q0] & kOffMask) + (size_t)kx * NC;
    if (HOM_CHECK(A, i0 < A.n_ws, i0)) tau[i0] = a;
    if (q0 + 1 < nreal) {
      const size_t i1 = (qbase[q0 + 1] & kOffMask) + (size_t)kx * NC;
      if (HOM_CHECK(A, i1 < A.n_ws, i1)) tau[i1] = b;
    }
    if (kx == 0) {
      dc_tau[q0] = a.x;
      if (q0 + 1 < nreal) dc_tau[q0 + 1] = b.x;
    }
  }
  __syncthreads();
  // Sum of sigma over the task's rows, per load and component, from the kx = 0 bins:
  //   sum_x sigma = sum_x tau + c0 : sum_x eps, with sum_x tau the (tree-summed) DFT bin of tau and
  //   sum_x eps = n times the stored row mean.  Rows are combined in FP64.
  if (threadIdx.x < nal * NC) {
    const int la = threadIdx.x / NC, k = threadIdx.x - la * NC;
    double acc = 0.0;
    for (int rl = 0; rl < t.nrows; ++rl) {
      const int q0 = (rl * nal + la) * NC;
      if (EM) {  // sigma = (tau + u) / 2, sum_x u = n times the stored row mean of u
        acc += 0.5 * ((double)dc_tau[q0 + k] + (double)n * (double)dc_eps[q0 + k]);
        continue;
      }
      double tr = 0.0;
#pragma unroll
      for (int j = 0; j < DIM; ++j) tr += (double)dc_eps[q0 + j];
      const double se = (double)n * (2.0 * c.mu0 * (double)dc_eps[q0 + k] + (k < DIM ? c.lam0 * tr : 0.0));
      acc += (double)dc_tau[q0 + k] + se;
    }
    A.partR[((size_t)blockIdx.x * A.L + s_al[la]) * NC + k] = acc;
  }
  if (threadIdx.x == 0)
    atomicAdd(A.bytes + HOM_K_ROW,
              (unsigned long long)(2 * (size_t)nreal * H * sizeof(V) + (size_t)t.nrows * n * 4));
}

// ------------------------------------------------------------------ Green pass
// One wave vector of the Eyre-Milton Green pass (see k_green and em_core): tv holds the nc
// entries of tau_hat (overwritten by the new u_hat for the inverse transform), up the stored u_hat
// of the current iterate (overwritten with the new one); uh is its value, read ahead.
template <typename T, int DIM, typename V>
__device__ __forceinline__ void em_point(V* const (&tv)[DIM == 2 ? 3 : 6], const V* uh, V* up, const T* xi, bool k0,
                                         bool nyq, bool self_conj, T nvT, T inv_nv, T lam0, T mu2_0, T a0,
                                         T inv_mu2_0, T inv_mu0, T ratio, const double* Eld, Acc<T>& r2acc,
                                         Acc<T>& rnacc, Acc<T>& c2acc) {
  constexpr int NC = DIM == 2 ? 3 : 6;
  V th[NC], un[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) th[k] = *tv[k];
  em_core<T, DIM>(th, uh, un, xi, k0, nyq, self_conj, nvT, inv_nv, lam0, mu2_0, a0, inv_mu2_0, inv_mu0, ratio, Eld,
                  r2acc, rnacc, c2acc);
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    *tv[k] = un[k];
    up[k] = un[k];
  }
}

// Lines along the last axis (y in 2D, z in 3D with ky fixed) for a tile of kx and one load.
// EM (Eyre-Milton): the private state beside the lines is u_hat of the current iterate (nc
// components per wave vector, 1/N_v-scaled) instead of g.  With tau_hat of the row pass,
// sigma_hat = (N_v u_hat + tau_hat) / 2 and c0 : eps_hat = (N_v u_hat - tau_hat) / 2 give the
// equilibrium residual sigma_hat . xi and the compatibility residual eps_hat - Gamma0 c0 eps_hat of
// the current iterate; the new state is tau_hat - 2 c0 Gamma0 tau_hat (k != 0), tau_hat(0) + 2 c0 E.
template <typename T, int DIM, int MAXR, bool EM = false>
__global__ void __launch_bounds__(kThreads) k_green(SolveArgs A) {
  using V = typename Cx<T>::V;
  constexpr int NC = DIM == 2 ? 3 : 6;
  constexpr int GC = EM ? NC : DIM;  // components of the private state per wave vector
  HOM_DBG_POISON();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Plan sp;
  const TaskL t = A.tC[blockIdx.x];
  const int cl = t.cell * A.L + t.load;
  if (!A.active[cl]) return;
  const CellDev c = A.cells[t.cell];
  load_plan(A, c.plan, sp);
  const int it = *A.it_dev;
  const int n = c.n, Hp = c.Hp, ntk = t.ntk;
  const V* tw = stage_twiddles<V>(smem_raw, sp);
  V* s = reinterpret_cast<V*>(smem_raw) + n;
  const int nl = ntk * NC;
  const size_t rowstride = DIM == 2 ? (size_t)Hp * NC : (size_t)n * Hp * NC;
  const size_t base = c.ws_off + (size_t)t.load * c.nrows * Hp * NC +
                      (DIM == 3 ? (size_t)t.fixed * Hp * NC : 0) + (size_t)t.kx0 * NC;
  const V* in = static_cast<const V*>(A.tau);
  V* out = DIM == 2 ? static_cast<V*>(A.eps[(it + 1) & 1]) : static_cast<V*>(A.tau);

  {
    constexpr int U = 4;
    Iter2 it(threadIdx.x, kThreads, t.d_nl);
    while (it.a < n) {
      int jj[U], ww[U];
      V v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        jj[u] = it.a;
        ww[u] = it.b;
        if (it.a < n) {
          const size_t i0 = base + (size_t)it.a * rowstride + it.b;
          v[u] = HOM_CHECK(A, i0 < A.n_ws, i0) ? in[i0] : mk(T(0), T(0));
        }
        it.next();
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (jj[u] < n) s[(size_t)ww[u] * n + jj[u]] = v[u];
    }
  }
  __syncthreads();
  fft_dif<true, MAXR, V, T>(s, nl, n, sp, tw, threadIdx.x, kThreads);

  // Green operator at every wave vector of the tile (spectrum at digit-reversed positions)
  CellConst<T> cc;
  cell_const(c, cc);
  const T mu0 = T(0.5) * cc.mu2;
  const T lpm = cc.lpm;
  const T ratio = cc.ratio;
  const T inv_nv = cc.inv_nv;
  const T inv_mu0 = cc.inv_mu0;
  // 2 pi a(k) of the transformed axis, one entry per bin (after the lines in shared memory); the
  // rotated scheme takes the factors (2n sin(pi a/n), cos(pi a/n)) of its wave vector instead
  const bool rotated = A.green == HOM_GREEN_ROTATED;
  T* xi_tab = reinterpret_cast<T*>(s + (size_t)nl * n);
  V* rot_tab = reinterpret_cast<V*>(s + (size_t)nl * n);
  const T* xi_src = xi_table<T>(sp);
  const V* rot_src = rot_table<V>(sp);
  if (rotated) {
    for (int k = threadIdx.x; k < n; k += kThreads) rot_tab[k] = rot_src[k];
  } else {
    for (int k = threadIdx.x; k < n; k += kThreads) xi_tab[k] = xi_src[k];
  }
  const T xi_fixed = DIM == 3 ? xi_src[t.fixed] : T(0);
  const V rot_fixed = DIM == 3 ? rot_src[t.fixed] : mk(T(0), T(1));
  __syncthreads();
  const T rs2 = T(0.707106781186547524400844362105);
  const double* Eld = A.E + ((size_t)t.cell * A.L + t.load) * NC;
  V* gbuf = static_cast<V*>(A.g);
  const size_t gbase = c.g_off + (size_t)t.load * c.nrows * Hp * GC + (size_t)t.kx0 * GC;
  const size_t grow_stride = DIM == 2 ? (size_t)Hp * GC : (size_t)n * Hp * GC;
  const size_t gfix = DIM == 3 ? (size_t)t.fixed * Hp * GC : 0;
  Acc<T> r2acc, rnacc, c2acc;
  // g of the next point is loaded while the current one is processed
  Iter2 gi(threadIdx.x, kThreads, t.d_ntk);
  V gnext[GC];
  // every g index of the task lies below the one of its last point
  if (!HOM_CHECK(A, gbase + gfix + (size_t)(n - 1) * grow_stride + (size_t)(ntk * GC) <= A.n_g,
                 gbase + gfix + (size_t)(n - 1) * grow_stride + (size_t)(ntk * GC)))
    gi.a = n;
  if (gi.a < n) {
    const V* gp0 = gbuf + gbase + gfix + (size_t)gi.a * grow_stride + (size_t)gi.b * GC;
#pragma unroll
    for (int d = 0; d < GC; ++d) gnext[d] = gp0[d];
  }
  // EM constants: N_v, 2 lam0, and c0^-1 s = (s - a0 tr(s) I) / (2 mu0), a0 = lam0 / (2 mu0 + DIM lam0)
  const T nvT = EM ? T(c.nv) : T(0);
  const T em_a0 = EM ? cc.lam0 / (cc.mu2 + T(DIM) * cc.lam0) : T(0);
  const T inv_mu2_0 = T(0.5) * inv_mu0;
  for (; gi.a < n;) {
    const int kk = gi.a, kxl = gi.b;
    V gv[GC];
#pragma unroll
    for (int d = 0; d < GC; ++d) gv[d] = gnext[d];
    gi.next();
    if (gi.a < n) {
      const V* gpn = gbuf + gbase + gfix + (size_t)gi.a * grow_stride + (size_t)gi.b * GC;
#pragma unroll
      for (int d = 0; d < GC; ++d) gnext[d] = gpn[d];
    }
    const int kx = t.kx0 + kxl;
    const int pos = HOM_LDG(sp.perm + kk);
    V* tv[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) tv[k] = s + (size_t)(kxl * NC + k) * n + pos;
    V* gp = gbuf + gbase + gfix + (size_t)kk * grow_stride + (size_t)kxl * GC;
    T xi[DIM];
    if (rotated) {  // q_j = 2n sin(pi a_j / n) prod_{m != j} cos(pi a_m / n)
      const V fx = rot_tab[kx], fl = rot_tab[kk];
      if (DIM == 2) {
        xi[0] = fx.x * fl.y;
        xi[1] = fx.y * fl.x;
      } else {
        xi[0] = fx.x * rot_fixed.y * fl.y;
        xi[1] = fx.y * rot_fixed.x * fl.y;
        xi[DIM - 1] = fx.y * rot_fixed.y * fl.x;
      }
    } else {
      xi[0] = xi_tab[kx];  // kx <= (n-1)/2: the table entry is 2 pi kx
      if (DIM == 2) {
        xi[1] = xi_tab[kk];
      } else {
        xi[1] = xi_fixed;
        xi[DIM - 1] = xi_tab[kk];
      }
    }
    const bool k0 = kx == 0 && kk == 0 && (DIM == 2 || t.fixed == 0);
    // even grids: a wave vector with a Nyquist component (n/2) has no conjugate partner in the
    // spectrum of a real field; its strain is set to zero and it is left out of the residual
    const bool nyq = (n & 1) == 0 && (kx == (n >> 1) || kk == (n >> 1) || (DIM == 3 && t.fixed == (n >> 1)));
    if (EM) {
      em_point<T, DIM>(tv, gv, gp, xi, k0, nyq, kx == 0 || 2 * kx == n, nvT, inv_nv, cc.lam0, cc.mu2, em_a0,
                       inv_mu2_0, inv_mu0, ratio, Eld, r2acc, rnacc, c2acc);
      continue;
    }
    if (k0 || nyq) {
#pragma unroll
      for (int k = 0; k < NC; ++k) *tv[k] = k0 ? mk((T)Eld[k], T(0)) : mk(T(0), T(0));
#pragma unroll
      for (int d = 0; d < DIM; ++d) gp[d] = mk(T(0), T(0));
      continue;
    }
    // tensor components of tau_hat
    V tt[DIM][DIM];
    if (DIM == 2) {
      tt[0][0] = *tv[0];
      tt[1][1] = *tv[1];
      tt[0][1] = tt[1][0] = rs2 * *tv[2];
    } else {
      tt[0][0] = *tv[0];
      tt[1][1] = *tv[1];
      tt[DIM - 1][DIM - 1] = *tv[2];
      tt[1][DIM - 1] = tt[DIM - 1][1] = rs2 * *tv[3];
      tt[0][DIM - 1] = tt[DIM - 1][0] = rs2 * *tv[4];
      tt[0][1] = tt[1][0] = rs2 * *tv[5];
    }
    V v[DIM];
    T q2 = T(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      q2 += xi[a] * xi[a];
      V acc = mk(T(0), T(0));
#pragma unroll
      for (int b = 0; b < DIM; ++b) acc = acc + xi[b] * tt[a][b];
      v[a] = acc;
    }
    V xg = mk(T(0), T(0)), xv = mk(T(0), T(0));
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      xg = xg + xi[a] * gv[a];
      xv = xv + xi[a] * v[a];
    }
    // equilibrium residual of the current iterate: r = tau_hat xi - K0 g
    T r2 = T(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const V r = v[a] - (mu0 * q2) * gv[a] - (lpm * xi[a]) * xg;
      r2 += r.x * r.x + r.y * r.y;
    }
    const T wgt = kx == 0 ? T(1) : T(2);
    const T inv_q2 = recip(q2);
    r2acc.add(wgt * r2);
    rnacc.add(wgt * r2 * inv_q2);
    // g' = K0^-1 (tau_hat xi);  eps_hat' = -sym(xi (x) g') / N_v
    const T inv_mq = inv_mu0 * inv_q2;
    const T rq = ratio * inv_q2;
    V w[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      w[a] = inv_mq * (v[a] - (rq * xi[a]) * xv);
      gp[a] = w[a];
    }
    if (DIM == 2) {
      *tv[0] = (-xi[0] * inv_nv) * w[0];
      *tv[1] = (-xi[1] * inv_nv) * w[1];
      *tv[2] = (-rs2 * inv_nv) * (xi[0] * w[1] + xi[1] * w[0]);
    } else {
      *tv[0] = (-xi[0] * inv_nv) * w[0];
      *tv[1] = (-xi[1] * inv_nv) * w[1];
      *tv[2] = (-xi[2] * inv_nv) * w[2];
      *tv[3] = (-rs2 * inv_nv) * (xi[1] * w[2] + xi[2] * w[1]);
      *tv[4] = (-rs2 * inv_nv) * (xi[0] * w[2] + xi[2] * w[0]);
      *tv[5] = (-rs2 * inv_nv) * (xi[0] * w[1] + xi[1] * w[0]);
    }
  }
  if (EM) {
    const Acc<T> vv[3] = {r2acc, rnacc, c2acc};
    double tot[3];
    block_sum<T, 3>(vv, tot);  // contains the barrier before the inverse transform
    if (threadIdx.x == 0) {
      A.partC[2 * (size_t)blockIdx.x] = tot[0];
      A.partC[2 * (size_t)blockIdx.x + 1] = tot[1];
      A.partE[blockIdx.x] = tot[2];
    }
  } else {
    const Acc<T> vv[2] = {r2acc, rnacc};
    double tot[2];
    block_sum<T, 2>(vv, tot);  // contains the barrier before the inverse transform
    if (threadIdx.x == 0) {
      A.partC[2 * (size_t)blockIdx.x] = tot[0];
      A.partC[2 * (size_t)blockIdx.x + 1] = tot[1];
    }
  }
  fft_dit<false, MAXR, V, T>(s, nl, n, sp, tw, threadIdx.x, kThreads);
  // defect correction (2D): the new iterate takes the fixed source strain (3D: in the inverse y pass)
  const V* srcm = DIM == 2 ? static_cast<const V*>(A.src_mixed) : nullptr;
  for (Iter2 it(threadIdx.x, kThreads, t.d_nl); it.a < n; it.next()) {
    const int j = it.a, w = it.b;
    const size_t ad = base + (size_t)j * rowstride + w;
    if (HOM_CHECK(A, ad < A.n_ws, ad)) out[ad] = srcm ? s[(size_t)w * n + j] + srcm[ad] : s[(size_t)w * n + j];
  }
  if (threadIdx.x == 0)
    atomicAdd(A.bytes + HOM_K_GREEN,
              (unsigned long long)(2 * (size_t)n * nl * sizeof(V) + 2 * (size_t)n * ntk * GC * sizeof(V)));
}

// ------------------------------------------------------------------ 3D y passes
template <typename T, bool FWD, int MAXR>
__global__ void __launch_bounds__(kThreads) k_ypass(SolveArgs A) {
  using V = typename Cx<T>::V;
  constexpr int NC = 6;
  HOM_DBG_POISON();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Plan sp;
  const TaskL t = A.tY[blockIdx.x];
  const int cl = t.cell * A.L + t.load;
  if (!A.active[cl]) return;
  const CellDev c = A.cells[t.cell];
  load_plan(A, c.plan, sp);
  const int it = *A.it_dev;
  const int n = c.n, Hp = c.Hp, nl = t.ntk * NC;
  const V* tw = stage_twiddles<V>(smem_raw, sp);
  V* s = reinterpret_cast<V*>(smem_raw) + n;
  const size_t rowstride = (size_t)Hp * NC;
  const size_t base = c.ws_off + (size_t)t.load * c.nrows * Hp * NC + (size_t)t.fixed * n * Hp * NC +
                      (size_t)t.kx0 * NC;
  const V* in = static_cast<const V*>(A.tau);
  V* out = FWD ? static_cast<V*>(A.tau) : static_cast<V*>(A.eps[(it + 1) & 1]);
  for (Iter2 it(threadIdx.x, kThreads, t.d_nl); it.a < n; it.next()) {
    const int j = it.a, w = it.b;
    const int pos = FWD ? j : HOM_LDG(sp.perm + j);
    const size_t i0 = base + (size_t)j * rowstride + w;
    s[(size_t)w * n + pos] = HOM_CHECK(A, i0 < A.n_ws, i0) ? in[i0] : mk(T(0), T(0));
  }
  __syncthreads();
  if (FWD) fft_dif<true, MAXR, V, T>(s, nl, n, sp, tw, threadIdx.x, kThreads);
  else fft_dit<false, MAXR, V, T>(s, nl, n, sp, tw, threadIdx.x, kThreads);
  const V* srcm = FWD ? nullptr : static_cast<const V*>(A.src_mixed);  // defect correction (3D)
  for (Iter2 it(threadIdx.x, kThreads, t.d_nl); it.a < n; it.next()) {
    const int j = it.a, w = it.b;
    const int pos = FWD ? HOM_LDG(sp.perm + j) : j;
    const size_t ad = base + (size_t)j * rowstride + w;
    if (HOM_CHECK(A, ad < A.n_ws, ad)) out[ad] = srcm ? s[(size_t)w * n + pos] + srcm[ad] : s[(size_t)w * n + pos];
  }
  if (threadIdx.x == 0)
    atomicAdd(A.bytes + (FWD ? HOM_K_YFWD : HOM_K_YINV), (unsigned long long)(2 * (size_t)n * nl * sizeof(V)));
}

// ------------------------------------------------------------------ control
// One CTA per (cell, load): FP64 sums of the pair's partials (per-task partials of the row pass
// and of the Green pass, summed in a fixed order: deterministic), equilibrium errors, stopping
// rule.  The last CTA to finish counts the active pairs and advances the iteration.
// Bound by latency (a chain of a few dependent loads) and, for pairs of many tasks, by FP64 additions: an
// SM does two per cycle.  Each thread keeps several tasks' loads in flight; the block sums go through shared
// memory, one warp per total (a shuffle tree in every warp would spend 32 lanes on every addition); a pair of
// more than kCtlSlice tasks is split over CTAs, the last of which adds the slices in order.  Launches of
// 128 threads and one CTA per pair took 56 us at 135^3 (6 pairs of 4590 + 4590 tasks), 1024 threads 32 us;
// now 16 us.
constexpr int kCtlThreads = 256;
constexpr int kCtlSlice = 1024;
constexpr int kCtlMaxSlices = 16;
inline unsigned ctl_slices(int most_tasks) {
  return (unsigned)std::min(kCtlMaxSlices, std::max(1, (most_tasks + kCtlSlice / 2) / kCtlSlice));
}
template <int NC>
__global__ void __launch_bounds__(kCtlThreads) k_control(SolveArgs A) {
  constexpr int K = NC + 3;
  __shared__ double s_val[K][kCtlThreads];
  __shared__ double s_tot[K];
  __shared__ int s_last;
  const int pair = blockIdx.x, slice = blockIdx.y, slices = gridDim.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int it = *A.it_dev;
  int still = 0;  // thread 0: the pair stays active
  if (A.active[pair]) {
    const PairDev pr = A.pairs[pair];
    // v[0..NC): sigma sums, v[NC]: residual sum, v[NC + 1]: normalised residual sum, v[NC + 2]:
    // compatibility residual sum (Eyre-Milton scheme)
    double v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.0;
    const double* pR = A.partR + (size_t)pr.load * NC;
    const size_t rs = (size_t)A.L * NC;
    const int nr = pr.rtask1 - pr.rtask0, nc = pr.ctask1 - pr.ctask0;
    const int r1 = pr.rtask0 + (int)((long long)nr * (slice + 1) / slices);
    const int c1 = pr.ctask0 + (int)((long long)nc * (slice + 1) / slices);
#pragma unroll 4
    for (int tk = pr.rtask0 + (int)((long long)nr * slice / slices) + (int)threadIdx.x; tk < r1; tk += kCtlThreads) {
      const double* p = pR + (size_t)tk * rs;
#pragma unroll
      for (int k = 0; k < NC; ++k) v[k] += p[k];
    }
    const double2* pC = reinterpret_cast<const double2*>(A.partC);
    const bool em = A.partE != nullptr;
#pragma unroll 4
    for (int tk = pr.ctask0 + (int)((long long)nc * slice / slices) + (int)threadIdx.x; tk < c1; tk += kCtlThreads) {
      const double2 q = pC[tk];
      v[NC] += q.x;
      v[NC + 1] += q.y;
      if (em) v[NC + 2] += A.partE[tk];
    }
#pragma unroll
    for (int k = 0; k < K; ++k) s_val[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int k = wid; k < K; k += kCtlThreads / 32) {
      double x = 0.0;
#pragma unroll
      for (int i = 0; i < kCtlThreads / 32; ++i) x += s_val[k][i * 32 + lane];
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) s_tot[k] = x;
    }
    __syncthreads();
    bool last = true;
    if (slices > 1) {
      if (threadIdx.x < K) {
        A.ctl_part[((size_t)pair * slices + slice) * K + threadIdx.x] = s_tot[threadIdx.x];
        __threadfence();
      }
      __syncthreads();
      if (threadIdx.x == 0) s_last = atomicAdd(A.ctl_cnt + pair, 1) == slices - 1;
      __syncthreads();
      last = s_last;
    }
    if (!last) return;
    if (wid == 0) {
      double sum = lane < K ? s_tot[lane] : 0.0;  // lane k: total k
      if (slices > 1) {
        __threadfence();
        sum = 0.0;
        if (lane < K)
          for (int q = 0; q < slices; ++q) sum += __ldcg(A.ctl_part + ((size_t)pair * slices + q) * K + lane);
        if (lane == 0) A.ctl_cnt[pair] = 0;
      }
      still = control_pair<NC>(A, pair, (double)A.cells[pr.cell].nv, sum, it);
    }
  } else if (slice > 0) {
    return;
  }
  if (threadIdx.x == 0) {
    // arrivals in the low half, active pairs in the high half: the last CTA has both
    const unsigned long long mine = 1ull + ((unsigned long long)still << 32);
    const unsigned long long all = atomicAdd(A.done, mine) + mine;
    if ((unsigned)all == gridDim.x) {
      const int tot = (int)(all >> 32);
      *A.nactive = tot;
      *A.it_dev = it + 1;
      *A.done = 0ull;
      // whole-solve graph: run another iteration while a pair is active and the budget allows
      // (the host loop's bound: at most max_iter + 1 iterations)
      if (A.use_cond) cudaGraphSetConditional(A.cond, (tot > 0 && it + 1 <= A.max_iter) ? 1u : 0u);
    }
  }
}

// ------------------------------------------------------------------ initial state
// eps = E: the stored x-spectrum holds E at kx = 0 of every row (see the scaling convention in
// the row pass: stored = (1/n) x-DFT, so the unnormalised inverse gives eps back).
// EM: the state u = 2 c0 : E instead, and its (1/N_v-scaled) spectrum at k = 0 in the private state
// of the Green pass (zero elsewhere: the caller clears it).
template <typename T, bool EM = false>
__global__ void k_init(SolveArgs A, int ncells, int nc) {
  using V = typename Cx<T>::V;
  for (int cell = blockIdx.y; cell < ncells; cell += gridDim.y) {
    const CellDev c = A.cells[cell];
    const long long items = (long long)A.L * c.nrows * nc;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < items; i += (long long)gridDim.x * blockDim.x) {
      const int comp = (int)(i % nc);
      const long long r = i / nc;
      const long long row = r % c.nrows;
      const int l = (int)(r / c.nrows);
      const size_t ad = c.ws_off + ((size_t)l * c.nrows + row) * c.Hp * nc + comp;
      const double* El = A.E + ((size_t)cell * A.L + l) * nc;
      double v = El[comp];
      if (EM) {
        double trE = 0.0;
        for (int k = 0; k < c.dim; ++k) trE += El[k];
        v = 2.0 * (2.0 * c.mu0 * El[comp] + (comp < c.dim ? c.lam0 * trE : 0.0));
        const size_t gi = c.g_off + (size_t)l * c.nrows * c.Hp * nc + comp;
        if (row == 0 && HOM_CHECK(A, gi < A.n_g, gi)) static_cast<V*>(A.g)[gi] = mk((T)v, T(0));
      }
      if (HOM_CHECK(A, ad < A.n_ws, ad)) static_cast<V*>(A.eps[0])[ad] = mk((T)v, T(0));
    }
  }
}

// Warm start: the caller's real strain field of every (cell, load) [nc][voxels] (field precision,
// layout of hom_result.eps) into the stored state eps[0]: per row the half spectrum of its
// (1/n)-scaled x-DFT, two real rows per complex line (the row pass's transform); one task = rows x
// every load.
template <typename T, int DIM, int MAXR>
__global__ void __launch_bounds__(kThreads) k_state_in(SolveArgs A, const T* eps_in) {
  using V = typename Cx<T>::V;
  constexpr int NC = DIM == 2 ? 3 : 6;
  HOM_DBG_POISON();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Plan sp;
  const TaskR t = A.tR[blockIdx.x];
  const CellDev c = A.cells[t.cell];
  load_plan(A, c.plan, sp);
  const int n = c.n, Hp = c.Hp, L = A.L;
  const V* tw = stage_twiddles<V>(smem_raw, sp);
  V* s = reinterpret_cast<V*>(smem_raw) + n;
  const int nreal = t.nrows * L * NC;
  const int nlines = (nreal + 1) >> 1;
  const size_t load_stride = (size_t)c.nrows * Hp * NC;
  // real row q = (row, load, component), as in the row pass with every load active
  auto rowq = [&](int q, int& rl, int& l, int& comp) {
    rl = q / (L * NC);
    const int rem = q - rl * L * NC;
    l = rem / NC;
    comp = rem - l * NC;
  };
  for (Iter2 it(threadIdx.x, kThreads, sp.div_n); it.a < nlines; it.next()) {
    const int line = it.a, x = it.b;
    T v[2] = {T(0), T(0)};
    for (int h = 0; h < 2; ++h) {
      const int q = 2 * line + h;
      if (q >= nreal) break;
      int rl, l, comp;
      rowq(q, rl, l, comp);
      const size_t vox = (size_t)(t.row0 + rl) * n + x;
      const size_t i0 = c.fld_off + ((size_t)l * NC + comp) * c.nv + vox;
      if (HOM_CHECK(A, i0 < A.n_fld, i0)) v[h] = eps_in[i0];
    }
    s[(size_t)line * n + HOM_LDG(sp.perm + x)] = mk(v[0], v[1]);
  }
  __syncthreads();
  fft_dit<true, MAXR, V, T>(s, nlines, n, sp, tw, threadIdx.x, kThreads);
  V* out = static_cast<V*>(A.eps[0]);
  const T inv_n = T(1) / T(n);
  for (Iter2 it(threadIdx.x, kThreads, sp.div_h); it.a < nlines; it.next()) {
    const int line = it.a, kx = it.b;
    const V* z = s + (size_t)line * n;
    const V zk = z[kx];
    const V zm = z[kx == 0 ? 0 : n - kx];
    const V a = mk(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));
    const V b = mk(T(0.5) * (zk.y + zm.y), T(0.5) * (zm.x - zk.x));
    for (int h = 0; h < 2; ++h) {
      const int q = 2 * line + h;
      if (q >= nreal) break;
      int rl, l, comp;
      rowq(q, rl, l, comp);
      const size_t ad = c.ws_off + (size_t)l * load_stride + (size_t)(t.row0 + rl) * Hp * NC + (size_t)kx * NC + comp;
      if (HOM_CHECK(A, ad < A.n_ws, ad)) out[ad] = inv_n * (h == 0 ? a : b);
    }
  }
}

// EM: (c~ + c0)^-1 of every mixed voxel of every cell (c0 of the voxel's cell), by Cholesky
// factorisation in FP64, packed like the mixed stiffness table; blockIdx.y = cell.  The few mixed
// voxels of each run of kMinvRun labels are listed first, so that the FP64 work runs in full warps:
// factorising voxel by voxel where the labels lie, mostly one lane of a warp at a time, took 0.97 ms for
// the 64 cells (2.3 M voxels) of a random-disk ensemble, this 0.057 ms.
constexpr int kMinvThreads = 128;
constexpr int kMinvRun = 1024;
template <typename T, int NC>
__global__ void __launch_bounds__(kMinvThreads) k_em_minv(SolveArgs A, T* minv) {
  constexpr int NS = NC * (NC + 1) / 2;
  __shared__ uint32_t s_list[kMinvRun];
  __shared__ int s_cnt;
  const CellDev c = A.cells[blockIdx.y];
  const double* tab = A.mixed_c64;
  for (long long v0 = (long long)blockIdx.x * kMinvRun; v0 < c.nv; v0 += (long long)gridDim.x * kMinvRun) {
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const int run = (int)min((long long)kMinvRun, c.nv - v0);
    for (int i = threadIdx.x; i < run; i += kMinvThreads) {
      const uint32_t lab = A.label[c.vox_off + v0 + i];
      if (lab & HOM_MIXED_BIT) s_list[atomicAdd(&s_cnt, 1)] = lab & ~HOM_MIXED_BIT;
    }
    __syncthreads();
    const int cnt = s_cnt;
    for (int i = threadIdx.x; i < cnt; i += kMinvThreads) {
      const size_t m = s_list[i];
      double a[NC][NC];  // lower triangle: a = L L^T in place, 1 / L_jj on the diagonal
#pragma unroll
      for (int r = 0; r < NC; ++r)
#pragma unroll
        for (int q = r; q < NC; ++q) {
          double x = tab[m * NS + packed_index(NC, r, q)];
          if (r == q) x += 2.0 * c.mu0;
          if (r < (NC == 3 ? 2 : 3) && q < (NC == 3 ? 2 : 3)) x += c.lam0;
          a[q][r] = x;
        }
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        double d = a[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) d -= a[j][k] * a[j][k];
        const double id = 1.0 / sqrt(d);
        a[j][j] = id;
#pragma unroll
        for (int r = j + 1; r < NC; ++r) {
          double x = a[r][j];
#pragma unroll
          for (int k = 0; k < j; ++k) x -= a[r][k] * a[j][k];
          a[r][j] = x * id;
        }
      }
      // L^-1 in place (column by column), then the inverse as L^-T L^-1
#pragma unroll
      for (int j = 0; j < NC; ++j)
#pragma unroll
        for (int r = j + 1; r < NC; ++r) {
          double x = 0.0;
#pragma unroll
          for (int k = j; k < r; ++k) x -= a[r][k] * a[k][j];
          a[r][j] = x * a[r][r];
        }
#pragma unroll
      for (int r = 0; r < NC; ++r)
#pragma unroll
        for (int q = r; q < NC; ++q) {
          double x = 0.0;
#pragma unroll
          for (int k = q; k < NC; ++k) x += a[k][r] * a[k][q];
          minv[m * NS + packed_index(NC, r, q)] = (T)x;
        }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ defect correction
// Element ranges of pair p's strain state (ε layout) and displacement-like state (g layout).
__device__ __forceinline__ void pair_ranges(const SolveArgs& A, int p, size_t& e0, size_t& ne, size_t& g0, size_t& ng) {
  const PairDev pd = A.pairs[p];
  const CellDev c = A.cells[pd.cell];
  ne = (size_t)c.nrows * c.Hp * c.nc;
  e0 = c.ws_off + (size_t)pd.load * ne;
  ng = (size_t)c.nrows * c.Hp * c.dim;
  g0 = c.g_off + (size_t)pd.load * ng;
}

enum RefineOp {
  kRefStart,   // eps64 = eps32[(iters + 1) & 1], g64 = g32  (the last FP32 iterate and its g)
  kRefResid,   // r32 = eps64[1] - eps64[0]                   (F(eps) - eps, rounded to FP32)
  kRefUpdate,  // eps64[0] += eps32[(k + 1) & 1], g64 += g32  (the correction after k inner steps)
  kRefFinal    // eps32[iters & 1] = eps64[0]                 (the returned iterate, for the output pass)
};

// One element-wise step of the defect correction over the pairs with mask[p] != 0; blockIdx.y = pair.
template <int OP>
__global__ void k_refine(SolveArgs A, const int* mask, const float2* eps32a, const float2* eps32b, float2* g32,
                         double2* eps64a, const double2* eps64b, double2* g64, float2* r32, int kinner) {
  const int p = blockIdx.y;
  if (!mask[p]) return;
  size_t e0, ne, g0, ng;
  pair_ranges(A, p, e0, ne, g0, ng);
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (OP == kRefStart) {
    const float2* e32 = ((A.iters[p] + 1) & 1) ? eps32b : eps32a;
    for (size_t i = i0; i < ne; i += stride) eps64a[e0 + i] = make_double2(e32[e0 + i].x, e32[e0 + i].y);
    for (size_t i = i0; i < ng; i += stride) g64[g0 + i] = make_double2(g32[g0 + i].x, g32[g0 + i].y);
  } else if (OP == kRefResid) {
    for (size_t i = i0; i < ne; i += stride) {
      const double2 a = eps64b[e0 + i], b = eps64a[e0 + i];
      r32[e0 + i] = make_float2((float)(a.x - b.x), (float)(a.y - b.y));
    }
  } else if (OP == kRefUpdate) {
    const float2* d32 = ((A.kinner[p] + 1) & 1) ? eps32b : eps32a;
    for (size_t i = i0; i < ne; i += stride) {
      double2 a = eps64a[e0 + i];
      a.x += d32[e0 + i].x;
      a.y += d32[e0 + i].y;
      eps64a[e0 + i] = a;
    }
    for (size_t i = i0; i < ng; i += stride) {
      double2 a = g64[g0 + i];
      a.x += g32[g0 + i].x;
      a.y += g32[g0 + i].y;
      g64[g0 + i] = a;
    }
  } else {
    float2* e32 = const_cast<float2*>((A.iters[p] & 1) ? eps32b : eps32a);
    for (size_t i = i0; i < ne; i += stride) e32[e0 + i] = make_float2((float)eps64a[e0 + i].x, (float)eps64a[e0 + i].y);
  }
}

// The start of the inner solve of pair p: delta^0 = r (in eps32[0]), bookkeeping of pair p reset.
__global__ void k_refine_inner_start(SolveArgs A, const int* mask, const float2* r32, float2* eps32a) {
  const int p = blockIdx.y;
  if (!mask[p]) return;
  size_t e0, ne, g0, ng;
  pair_ranges(A, p, e0, ne, g0, ng);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < ne; i += (size_t)gridDim.x * blockDim.x)
    eps32a[e0 + i] = r32[e0 + i];
}

// Bookkeeping of a refinement phase: pairs with mask[p] start active, the others stay inactive.
__global__ void k_init_pairs_masked(SolveArgs A, const int* mask) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < A.npairs) {
    A.active[p] = mask[p] ? 1 : 0;
    A.iters[p] = 0;
    A.status[p] = -1;
    A.grow[p] = 0;
    A.last_err[p] = INFINITY;
    A.best_err[p] = INFINITY;
    A.best_it[p] = 0;
  }
  if (p == 0) {
    int cnt = 0;
    for (int q = 0; q < A.npairs; ++q) cnt += mask[q] ? 1 : 0;
    *A.it_dev = 0;
    *A.nactive = cnt;
    *A.done = 0ull;
  }
}

__global__ void k_init_pairs(SolveArgs A) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < A.npairs) {
    A.active[p] = 1;
    A.iters[p] = 0;
    A.status[p] = -1;
    A.grow[p] = 0;
    A.last_err[p] = INFINITY;
    A.best_err[p] = INFINITY;
    A.best_it[p] = 0;
  }
  if (p == 0) {
    *A.it_dev = 0;
    *A.nactive = A.npairs;
    *A.done = 0ull;
  }
}

// ------------------------------------------------------------------ host side
// Opt a kernel in to `bytes` of dynamic shared memory (needed above 48 KB).
template <typename K>
int allow_smem(K kernel, size_t bytes) {
  cudaFuncAttributes fa{};
  HOM_CUDA_TRY(cudaFuncGetAttributes(&fa, kernel));
  int dev = 0, optin = 0;
  HOM_CUDA_TRY(cudaGetDevice(&dev));
  HOM_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  if (bytes + fa.sharedSizeBytes > (size_t)optin)
    return set_error(HOM_ERR_UNSUPPORTED_SIZE, "kernel needs %zu bytes of shared memory, device allows %d",
                     bytes + fa.sharedSizeBytes, optin);
  if ((int)bytes > fa.maxDynamicSharedSizeBytes)
    HOM_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return HOM_OK;
}

struct Layout {
  std::vector<CellDev> cells;
  std::vector<Plan> plans;
  std::vector<HostPlan> host_plans;  // external workspace only: tables to upload with the call
  std::vector<TaskR> tR;
  std::vector<TaskL> tC, tY;
  std::vector<PairDev> pairs;
  std::vector<FastPlanDev> fplans;  // specialised FP32 passes: per-size tables
  std::vector<std::vector<unsigned char>> fplan_host;  // external workspace: their host copies
  bool fast = false;
  bool compact = false;  // the least scratch: no smaller tasks than fit on chip, one control CTA per pair
  bool run = false;  // fast, with radices read from the plans (a size without compiled ones)
  int run_max = 0;   // the largest of them (0: compiled radices)
  size_t ws_elems = 0, g_elems = 0, fld_elems = 0;
  size_t smem_row = 0, smem_green = 0, smem_y = 0;
};


// The control kernel's arrival word: 64 bits after the pair bookkeeping of npairs pairs at `ib`.
unsigned long long* done_word(int* ib, int npairs) {
  return reinterpret_cast<unsigned long long*>((reinterpret_cast<uintptr_t>(ib + 5 * npairs + 2) + 7) & ~(uintptr_t)7);
}

// Most tasks of one pair in one pass (sizes the control kernel's CTAs).
int most_tasks(const Layout& lay) {
  int m = 1;
  for (const PairDev& p : lay.pairs) m = std::max(m, std::max(p.rtask1 - p.rtask0, p.ctask1 - p.ctask0));
  return m;
}

// Control CTAs per pair.
unsigned control_slices(const Layout& lay) { return lay.compact ? 1u : ctl_slices(most_tasks(lay)); }

template <int DIM> constexpr int nc_of_dim() { return DIM == 2 ? 3 : 6; }

long long vox_total(const Layout& lay) {
  long long v = 0;
  for (const CellDev& c : lay.cells) v += c.nv;
  return v;
}

TaskL make_task(int cell, int load, int kx0, int ntk, int fixed, int nc, int dim) {
  TaskL t{};
  t.cell = cell;
  t.load = load;
  t.kx0 = kx0;
  t.ntk = ntk;
  t.fixed = fixed;
  t.d_ntk = make_fastdiv(ntk);
  t.d_nl = make_fastdiv(ntk * nc);
  t.d_ng = make_fastdiv(ntk * dim);
  return t;
}

// Per-CTA shared-memory budgets of the generic passes: the Green and y passes take three kx
// columns of a 1215 line in FP32 (nine lines, two CTAs per SM), the row pass two CTAs per SM
// (both measured best on the 2D sweep).
constexpr size_t kGreenBudget = (size_t)110 * 1024;
constexpr size_t kRowBudget = (size_t)96 * 1024;

// A batch of few or small cells leaves most of the chip idle when every CTA of the generic passes takes as much
// as its shared memory holds; smaller tasks spread it, but each has a start of its own (task words, twiddles,
// labels, a barrier per stage), and one task more than the SMs share out evenly costs a whole turn.  Below four
// tasks per SM the sizes are therefore chosen by an estimate of the busiest SM's time.
//   One grid size: a task of `lines` complex lines of length n costs n lines + fixed; of T tasks the SM gets
//   ceil(T / SMs), two at a time in `pair` times the time of one (FP64 keeps an SM busy with one task, FP32 does
//   not); over every size of task.
//   Several: a task costs n (lines + start) + fixed; the larger of the largest task and of pair / 2 times the mean
//   load plus `tail` mean tasks, over the sizes that bring two, three, four or six tasks to an SM.
// Smaller tasks are taken where the estimate falls by more than `gain`.  The constants fit launches of 32 batches of
// one size (2D 45 to 512, 3D 13 to 81, one to six loads, one to sixteen cells, up to 18 task sizes each) and of 19 of
// several (2 to 61 cells): the sizes chosen take 0.2 to 4 % more than the best of those tried, and none more than
// tasks as large as fit.  Us per launch, as large as fit -> chosen: FP64 45^3, 1 load: row 129 -> 50, Green 133 ->
// 58; 26^3, 3 loads: 122 -> 39, 60 -> 51; 405^2, 3 loads: 153 and 184, both kept (a fixed target of four tasks
// per SM gave 193 and 215); the 61 cells of a convergence study: 156 -> 137, 184 -> 148.
struct TaskModel {
  struct {
    double fixed, pair, gain;
  } one;
  struct {
    double fixed, start, pair, tail, gain;
  } several;
};
constexpr TaskModel kRow64{{150.0, 1.8, 0.0}, {400.0, 1.0, 1.4, 1.0, 0.2}};
constexpr TaskModel kCol64{{900.0, 1.9, 0.0}, {150.0, 0.5, 2.0, 0.5, 0.2}};
constexpr TaskModel kRow32{{100.0, 1.0, 0.0}, {300.0, 0.0, 2.0, 0.5, 0.15}};
constexpr TaskModel kCol32{{900.0, 1.4, 0.05}, {500.0, 3.0, 2.0, 0.5, 0.1}};
struct PassCell {  // one cell's lines in a pass: `mult` times `units` rows or kx columns, at most `fit` a task
  int n, fit;
  long long units, mult;
};
// Rows (columns) per task of every cell.  `lines(k)`: complex lines of a task of k; `even`: tasks of an even number
// where they are smaller (an odd number of real rows leaves half of a complex line empty).
template <typename F>
std::vector<int> task_sizes(const std::vector<PassCell>& cells, const TaskModel& m, int sms, bool even, F lines) {
  auto tasks = [](const PassCell& c, int k) { return c.mult * ((c.units + k - 1) / k); };
  std::vector<int> pick;
  long long full = 0;
  bool alike = true;
  for (const PassCell& c : cells) {
    pick.push_back(c.fit);
    full += tasks(c, c.fit);
    alike = alike && c.n == cells[0].n && c.fit == cells[0].fit;
  }
  if (full >= 4ll * sms) return pick;
  double whole, best;
  if (alike) {
    const PassCell& c = cells[0];
    auto estimate = [&](int k) {
      const long long turns = (tasks(c, k) * (long long)cells.size() + sms - 1) / sms;
      return ((double)(turns / 2) * m.one.pair + (double)(turns % 2)) * (c.n * lines(k) + m.one.fixed);
    };
    whole = best = estimate(c.fit);
    for (int k = c.fit - 1; k >= 1; --k) {
      const double t = estimate(k);
      if (t < best && t < (1.0 - m.one.gain) * whole) {
        best = t;
        std::fill(pick.begin(), pick.end(), k);
      }
    }
    return pick;
  }
  auto estimate = [&](const std::vector<int>& k) {
    double sum = 0.0, most = 0.0;
    long long T = 0;
    for (size_t i = 0; i < cells.size(); ++i) {
      const double c = cells[i].n * (lines(k[i]) + m.several.start) + m.several.fixed;
      const long long t = tasks(cells[i], k[i]);
      T += t;
      sum += (double)t * c;
      most = std::max(most, c);
    }
    return std::max(0.5 * m.several.pair * sum / sms + m.several.tail * sum / (double)T, most);
  };
  whole = best = estimate(pick);
  std::vector<int> k(cells.size());
  for (const int per : {2, 3, 4, 6}) {
    const long long few = (long long)per * sms;
    for (size_t i = 0; i < cells.size(); ++i) {
      const int fit = cells[i].fit;
      k[i] = full >= few ? fit : (int)std::max<long long>(1, fit * full / few);
      if (even && k[i] < fit && (k[i] & 1)) ++k[i];
    }
    const double t = estimate(k);
    if (t < best && t < (1.0 - m.several.gain) * whole) {
      best = t;
      pick = k;
    }
  }
  return pick;
}
// One load per row task on the specialised passes, in place of every load (labels and twiddles are then read once):
// `groups` tasks of L loads, or groups L of one.  In 2D in turns of what the SMs hold at once (three CTAs up to
// radix 9 or with compiled radices, else two), a task's start costing about a load; 3D lines are short, and single
// loads keep the SMs busier up to as many groups.  Us per launch, every load -> one load: 45^2, 3
// loads: 16.5 -> 12.5; 405^2, 2 cells: 32 -> 28, 4 cells: 39.5, 44; 33^3, 6 loads: 38 -> 32; 45^3: 30, 32.
bool one_load_tasks(long long groups, int L, int dim, int run, int sms) {
  if (L < 2 || groups >= 4ll * sms) return false;
  const long long slots = (long long)sms * (run > 9 ? 2 : 3);
  auto turns = [&](long long tasks) { return (tasks + slots - 1) / slots; };
  return dim == 3 ? groups <= slots : 2 * turns(groups * L) <= (L + 1) * turns(groups);
}

// Whether the FP32 passes with radices from a plan are the faster ones, for batches that do not run on chip.  They
// keep a lane pair of lines per thread, with little per task; the generic ones hold many lines and radices up to 27
// per task.  While the plan-read tasks fit the chip at once (two or three CTAs an SM in 2D, four or six in 3D, by
// their registers) they win (325^2, 3 loads: 34 us an iteration against 45).  Beyond, they win where the generic
// passes' lines fall on the same banks (512^2, 8 cells, 3 loads: 229 against 552; 208^2, 64 cells: 582 against 829;
// 64^3, 6 loads: 232 against 381), on long lines (507^2, 8 cells: 276 against 306; 98^3: 679 against 946), and with
// three stages of radices up to 9 (2D: 343^2, 8 cells: 136 against 148); and lose elsewhere (143^2, 64 cells, 3
// loads: 362 against 174; 44^3, 6 loads: 149 against 96).  A batch goes as most of its voxels do.
bool plan_reads_win(int dim, int n, int largest, int stages) {
  if (dim == 2)
    return n >= 455 || (n >= 128 && n % (n <= 256 || n >= 400 ? 16 : 32) == 0) ||
           (n >= 243 && largest <= 9 && stages <= 3);
  return (n >= 32 && n % 8 == 0) || (n >= 70 && (largest <= 9 || stages <= 2 || n >= 100));
}
bool plan_passes_faster(const std::vector<int>& sizes, const std::vector<int>& largest, const std::vector<int>& stages, int L,
                        int dim, int run, int sms) {
  long long tasks = 0;
  double all = 0.0, good = 0.0;
  for (size_t i = 0; i < sizes.size(); ++i) {
    const int n = sizes[i];
    const long long groups = (n + kFastRows - 1) / kFastRows;
    tasks += L * groups * (dim == 2 ? 1 : n);
    const double voxels = (double)n * n * (dim == 2 ? 1 : n);
    all += voxels;
    good += plan_reads_win(dim, n, largest[i], stages[i]) ? voxels : 0.0;
  }
  const long long slots = (long long)sms * (run > 9 ? 2 : 3) * (dim == 2 ? 1 : 2);
  return tasks <= slots || 2.0 * good >= all;
}

int build_layout(const hom_cell* cells, int ncells, int L, int dim, size_t vsize, int max_radix, const double* c0,
                 bool external, Layout& lay, bool em, bool chip) {
  const int nc = nc_of(dim);
  const size_t budget = kRowBudget;
  const size_t kMaxSmem = 227 * 1024;
  // The specialised passes take 4-row and 2-column tasks; the output pass (generic row kernel)
  // then needs 4 rows of every load on chip.
  // The radices are compiled in where every size of the batch has them, else read from plans.
  if (lay.fast) {
    for (int ci = 0; ci < ncells; ++ci) {
      const int n = cells[ci].n;
      if (!(dim == 2 ? fast2d_size(n) : fast3d_size(n))) lay.run = true;
      if (!(dim == 2 ? run2d_size(n) : run3d_size(n))) lay.fast = false;
    }
    if (lay.run) {  // what the one-byte labels and their kernel cannot hold stays on the generic passes
      if (ncells > 65535) lay.fast = false;
      size_t nph_max = 1;
      for (int ci = 0; ci < ncells && lay.fast; ++ci) {
        std::vector<int> ph{cells[ci].matrix_phase};
        for (int p = 0; p < cells[ci].nprim; ++p) ph.push_back(cells[ci].prims[p].phase);
        std::sort(ph.begin(), ph.end());
        nph_max = std::max(nph_max, (size_t)(std::unique(ph.begin(), ph.end()) - ph.begin()));
        if (nph_max > 254) lay.fast = false;
      }
      if (lay.fast) {
        std::vector<int> sizes(ncells), largest(ncells), stages(ncells);
        for (int ci = 0; ci < ncells; ++ci) {
          sizes[ci] = cells[ci].n;
          run_plan_shape(sizes[ci], &largest[ci], &stages[ci]);
        }
        const int run = *std::max_element(largest.begin(), largest.end());
        if (!(chip && resident2d_takes(sizes, stages, L, run, (int)nph_max, em)))
          lay.fast = plan_passes_faster(sizes, largest, stages, L, dim, run, sm_count());
      }
    }
    lay.run = lay.run && lay.fast;
  }
  long long vox = 0;
  std::vector<int> plan_n;
  // rows per row task and kx columns per Green/y task that fit on chip, and the passes' tasks with them
  auto row_lines = [&](int rows) { return (size_t)((rows * L * nc + 1) / 2) + 1; };
  // (compiled sizes: four rows of every load, also where the generic kernel would hold fewer)
  auto rows_fit = [&](int n) {
    const int nrows = dim == 2 ? n : n * n;
    if (lay.fast && !lay.run) return std::min(kFastRows, nrows);
    const size_t line_bytes = (size_t)n * vsize;  // one line; the twiddle table is one more
    int r = 1;
    while (r < nrows &&
           row_lines(r + 1) * line_bytes + (size_t)(r + 1) * L * nc * (sizeof(long long) + vsize) <= budget)
      ++r;
    return r;
  };
  auto cols_fit = [&](int n) {
    const size_t line_bytes = (size_t)n * vsize, gbudget = kGreenBudget;
    int ntk = (int)std::max<size_t>(1, (gbudget - std::min(gbudget, 2 * line_bytes)) / ((size_t)nc * line_bytes));
    return std::min(lay.fast ? kFastCols : ntk, n / 2 + 1);
  };
  std::vector<int> task_rows, task_cols;
  std::vector<PassCell> row_cells, col_cells;
  long long groups = 0;  // of rows, on the specialised passes
  for (int ci = 0; ci < ncells; ++ci) {
    const int n = cells[ci].n, nrows = dim == 2 ? n : n * n;
    groups += (long long)((n + kFastRows - 1) / kFastRows) * (dim == 2 ? 1 : n);
    row_cells.push_back(PassCell{n, rows_fit(n), nrows, 1});
    col_cells.push_back(PassCell{n, cols_fit(n), n / 2 + 1, (long long)L * (dim == 2 ? 1 : n)});
  }
  if (!lay.fast && !lay.compact) {
    const bool f64 = vsize == sizeof(double2);
    const int sms = sm_count();
    task_rows = task_sizes(row_cells, f64 ? kRow64 : kRow32, sms, (L * nc & 1) != 0,
                           [&](int k) { return (double)((k * L * nc + 1) / 2); });
    task_cols = task_sizes(col_cells, f64 ? kCol64 : kCol32, sms, false, [&](int k) { return (double)(k * nc); });
  } else {
    for (int ci = 0; ci < ncells; ++ci) {
      task_rows.push_back(row_cells[ci].fit);
      task_cols.push_back(col_cells[ci].fit);
    }
  }
  for (int ci = 0; ci < ncells; ++ci) {
    const hom_cell& k = cells[ci];
    CellDev c{};
    c.dim = dim;
    c.n = k.n;
    c.H = k.n / 2 + 1;  // kx = 0 .. n/2: (n+1)/2 bins for odd n, n/2 + 1 (with the Nyquist bin) for even n
    c.Hp = (c.H + 7) / 8 * 8;
    c.nc = nc;
    c.nrows = dim == 2 ? k.n : k.n * k.n;
    c.nv = (long long)c.nrows * k.n;
    auto itp = std::find(plan_n.begin(), plan_n.end(), k.n);
    if (itp == plan_n.end()) {
      Plan p{};
      if (external) {
        HostPlan hp;
        if (!build_host_plan(k.n, hp, max_radix) || (int)hp.radix.size() > kMaxStages)
          return set_error(HOM_ERR_UNSUPPORTED_SIZE, "grid size %d has a prime factor above 13", k.n);
        p.n = k.n;
        p.nstage = (int)hp.radix.size();
        for (int s2 = 0; s2 < p.nstage; ++s2) {
          p.radix[s2] = hp.radix[s2];
          p.span[s2] = hp.span[s2];
        }
        plan_dividers(p);
        lay.host_plans.push_back(hp);  // table pointers are set once the scratch is carved
      } else {
        int rc = get_plan(k.n, max_radix, &p);
        if (rc != HOM_OK) return rc;
      }
      plan_n.push_back(k.n);
      lay.plans.push_back(p);
      c.plan = (int)lay.plans.size() - 1;
    } else {
      c.plan = (int)(itp - plan_n.begin());
    }
    c.fplan = -1;
    if (lay.fast) {
      int idx = -1;
      for (size_t i = 0; i < lay.fplans.size(); ++i)
        if (lay.fplans[i].n == k.n) idx = (int)i;
      if (idx < 0) {
        FastPlanDev fp{};
        int rc;
        if (external) {  // host tables, uploaded into the caller's workspace with the call
          lay.fplan_host.emplace_back();
          rc = fast2d_plan_host(k.n, lay.run, lay.fplan_host.back(), &fp);
        } else {
          rc = fast2d_plan(k.n, lay.run, &fp);
        }
        if (rc != HOM_OK) return rc;
        lay.fplans.push_back(fp);
        if (lay.run)
          for (int st = 0; st < fp.run.m; ++st) lay.run_max = std::max(lay.run_max, fp.run.r[st]);
        idx = (int)lay.fplans.size() - 1;
      }
      c.fplan = idx;
    }
    c.vox_off = vox;
    c.fld_off = (long long)lay.fld_elems;
    c.ws_off = (long long)lay.ws_elems;
    c.g_off = (long long)lay.g_elems;
    c.lam0 = c0[2 * ci];
    c.mu0 = c0[2 * ci + 1];
    c.d_lam0 = c.lam0;
    c.d_mu2 = 2.0 * c.mu0;
    c.d_lpm = c.lam0 + c.mu0;
    c.d_ratio = (c.lam0 + c.mu0) / (c.lam0 + 2.0 * c.mu0);
    c.d_inv_mu0 = 1.0 / c.mu0;
    c.d_inv_nv = 1.0 / (double)((long long)(dim == 2 ? k.n : k.n * k.n) * k.n);
    c.f_lam0 = (float)c.d_lam0;
    c.f_mu2 = (float)c.d_mu2;
    c.f_lpm = (float)c.d_lpm;
    c.f_ratio = (float)c.d_ratio;
    c.f_inv_mu0 = (float)c.d_inv_mu0;
    c.f_inv_nv = (float)c.d_inv_nv;
    vox += c.nv;
    lay.fld_elems += (size_t)L * nc * c.nv;
    lay.ws_elems += (size_t)L * c.nrows * c.Hp * nc;
    lay.g_elems += (size_t)L * c.nrows * c.Hp * (em ? nc : dim);  // EM: u_hat (nc) instead of g (dim)
    // row-pass tasks: as many rows as fit in the shared-memory budget with every load active
    const size_t line_bytes = (size_t)k.n * vsize;
    int r = task_rows[ci];
    // (passes with run-time radices refuse what the generic ones do, although they would hold it)
    const size_t need_r = row_lines(r) * line_bytes + (size_t)r * L * nc * (sizeof(long long) + 2 * vsize / 2);
    if (need_r > kMaxSmem) return set_error(HOM_ERR_UNSUPPORTED_SIZE, "row of n = %d with %d loads does not fit on chip", k.n, L);
    lay.smem_row = std::max(lay.smem_row, need_r);
    if (lay.fast) r = std::min(kFastRows, c.nrows);
    const int ntk = task_cols[ci];
    const size_t need_l = ((size_t)ntk * nc + 2) * line_bytes;
    lay.smem_green = std::max(lay.smem_green, need_l);
    lay.smem_y = std::max(lay.smem_y, need_l);
    task_rows[ci] = r;
    lay.cells.push_back(c);
  }
  const bool split_loads = lay.fast && !lay.compact && one_load_tasks(groups, L, dim, lay.run_max, sm_count());
  // tasks, largest grids first: the small cells' tasks fill the end of each launch
  std::vector<int> order(ncells);
  for (int ci = 0; ci < ncells; ++ci) order[ci] = ci;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cells[a].n > cells[b].n; });
  lay.pairs.resize((size_t)ncells * L);
  for (int ci : order) {
    const hom_cell& k = cells[ci];
    CellDev& c = lay.cells[ci];
    const int r = task_rows[ci], ntk = task_cols[ci];
    // row tasks: every load per task (one load per task measured 3 % slower on the 2D sweep: labels and
    // twiddles are shared across the loads), or one load per task where the batch has few (split_loads)
    c.rtask0 = (int)lay.tR.size();
    std::vector<int> rt0(L, c.rtask0), rt1(L, c.rtask0);
    for (int l = 0; l < (split_loads ? L : 1); ++l) {
      rt0[l] = (int)lay.tR.size();
      const int load = split_loads ? l : -1;
      if (lay.fast && dim == 3) {  // groups of 4 rows (consecutive y) within each z plane
        for (int z = 0; z < k.n; ++z)
          for (int y0 = 0; y0 < k.n; y0 += r) lay.tR.push_back(TaskR{ci, z * k.n + y0, std::min(r, k.n - y0), load});
      } else {
        for (int r0 = 0; r0 < c.nrows; r0 += r) lay.tR.push_back(TaskR{ci, r0, std::min(r, c.nrows - r0), load});
      }
      rt1[l] = (int)lay.tR.size();
    }
    if (!split_loads)
      for (int l = 1; l < L; ++l) {
        rt0[l] = rt0[0];
        rt1[l] = rt1[0];
      }
    c.rtask1 = (int)lay.tR.size();
    // Green-pass and y-pass tiles of kx: ntk kx columns x nc lines, plus the twiddle table and the
    // wave-number table
    for (int l = 0; l < L; ++l) {
      PairDev pd{ci, l, (int)lay.tC.size(), 0, rt0[l], rt1[l]};
      const int nfix = dim == 2 ? 1 : k.n;
      for (int f = 0; f < nfix; ++f)
        for (int kx0 = 0; kx0 < c.H; kx0 += ntk) lay.tC.push_back(make_task(ci, l, kx0, std::min(ntk, c.H - kx0), f, nc, dim));
      pd.ctask1 = (int)lay.tC.size();
      lay.pairs[(size_t)ci * L + l] = pd;
      if (dim == 3)
        for (int z = 0; z < k.n; ++z)
          for (int kx0 = 0; kx0 < c.H; kx0 += ntk) lay.tY.push_back(make_task(ci, l, kx0, std::min(ntk, c.H - kx0), z, nc, dim));
    }
  }
  return HOM_OK;
}

// CUDA events around every launch when statistics are requested.  Events come from a pool kept
// per device and reused across calls, so recording them costs no event creation on the timed path.
struct EventPool {
  std::vector<cudaEvent_t> ev;
  size_t next = 0;
};
EventPool g_event_pool[64];

struct Timer {
  hom_kernel_stats* stats;
  cudaStream_t st;
  std::vector<std::pair<int, std::pair<size_t, size_t>>> marks;  // kernel kind, event indices
  EventPool* pool = nullptr;
  cudaEvent_t take() {
    if (!pool) {
      int dev = 0;
      cudaGetDevice(&dev);
      pool = &g_event_pool[dev & 63];
      pool->next = 0;
    }
    if (pool->next == pool->ev.size()) {
      cudaEvent_t e;
      cudaEventCreate(&e);
      pool->ev.push_back(e);
    }
    return pool->ev[pool->next++];
  }
  void begin(int kind) {
    if (!stats) return;
    const size_t a = pool ? pool->next : 0;
    cudaEventRecord(take(), st);
    marks.push_back({kind, {a, 0}});
  }
  void end() {
    if (!stats) return;
    marks.back().second.second = pool->next;
    cudaEventRecord(take(), st);
  }
  void collect() {
    if (!stats) return;
    for (auto& m : marks) {
      float ms = 0.f;
      cudaEventSynchronize(pool->ev[m.second.second]);
      cudaEventElapsedTime(&ms, pool->ev[m.second.first], pool->ev[m.second.second]);
      stats->ms[m.first] += ms;
      stats->launches[m.first] += 1;
    }
    marks.clear();
    pool->next = 0;
  }
};

// Instantiated whole-solve graphs, kept across calls.  A graph bakes in the kernel arguments
// (pointers into the workspace and the caller's material, sizes, options) and launch shapes, so
// the key is those bytes; a call with the same key replays the cached graph.
struct GraphEntry {
  int dev;
  std::string key;
  cudaGraphExec_t exec;
};
std::mutex g_graph_mu;
std::vector<GraphEntry> g_graphs;  // most recently used last
constexpr size_t kMaxGraphs = 8;

cudaGraphExec_t find_graph(int dev, const std::string& key) {
  std::lock_guard<std::mutex> lk(g_graph_mu);
  for (size_t i = 0; i < g_graphs.size(); ++i)
    if (g_graphs[i].dev == dev && g_graphs[i].key == key) {
      GraphEntry e = g_graphs[i];
      g_graphs.erase(g_graphs.begin() + i);
      g_graphs.push_back(e);
      return e.exec;
    }
  return nullptr;
}

void keep_graph(int dev, const std::string& key, cudaGraphExec_t exec) {
  std::lock_guard<std::mutex> lk(g_graph_mu);
  if (g_graphs.size() >= kMaxGraphs) {
    cudaGraphExecDestroy(g_graphs.front().exec);
    g_graphs.erase(g_graphs.begin());
  }
  g_graphs.push_back(GraphEntry{dev, key, exec});
}

// Autotuner choices per batch shape (device, dimension, loads, Green operator, grid sizes), with the
// timings that decided them.
struct TuneChoice {
  int passes, radix;
};
struct TuneEntry {
  std::string key;
  TuneChoice choice;
  std::string report;
};
std::mutex g_tune_mu;
std::vector<TuneEntry> g_tuned;

bool find_tuned(const std::string& key, TuneChoice* out) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (const auto& e : g_tuned)
    if (e.key == key) {
      *out = e.choice;
      return true;
    }
  return false;
}

void keep_tuned(const std::string& key, TuneChoice c, const std::string& report) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tuned.push_back(TuneEntry{key, c, report});
}

bool is_device_ptr(const void* p) {
  if (!p) return false;
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Defect correction of the pairs the FP32 iteration left stalled (or at max_iter): from their last
// FP32 iterate eps (and its g), repeat up to opts->refine times
//   one FP64 iteration of the basic scheme on eps: its equilibrium error (FP64; the pair stops
//     when it passes opts->tol) and F(eps);
//   r = F(eps) - eps, rounded to FP32;
//   K + 1 FP32 iterations of the correction's fixed point delta <- r + F0(delta), delta^0 = r
//     (F0: the map with zero mean strain; the Green pass adds r to every new iterate);
//   eps <- eps + delta and g <- g(F(eps)) + g', in FP64.
// FP32 rounding then acts on the correction, not on the strain, so the FP32 iteration's floor no
// longer limits the attainable error.  On return the refined pairs' results (mean stress, errors,
// status, Green-operator applications) replace the FP32 ones and their iterate, rounded to FP32,
// sits where the output pass reads it.
template <typename T, int DIM, int MAXR>
int refine_solve(SolveArgs& A, unsigned char* ws, int npairs, int nc, const hom_solve_opts* opts, const Layout& lay,
                 size_t o_e64a, size_t o_e64b, size_t o_t64, size_t o_g64, size_t o_r32, size_t o_int2, size_t o_dbl2,
                 size_t o_mask, size_t o_plans64, size_t o_E0, cudaStream_t st) {
  if constexpr (!std::is_same<T, float>::value) {
    return HOM_OK;
  } else {
    std::vector<int> h_st(npairs), h_it(npairs), mask(npairs, 0);
    HOM_CUDA_TRY(cudaMemcpyAsync(h_st.data(), A.status, npairs * sizeof(int), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(h_it.data(), A.iters, npairs * sizeof(int), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<double> h_e(npairs);
    HOM_CUDA_TRY(cudaMemcpyAsync(h_e.data(), opts->criterion == HOM_CRIT_E ? A.err : A.errn, npairs * sizeof(double),
                                 cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));
    // inner iterations: the FP32 iteration took it_p steps to bring the error from about 1 to e_p,
    // a contraction of e_p^(1/it_p) per step; one correction should shrink the error to a fifth of
    // tol, i.e. by f_p = tol / (5 e_p): K_p = it_p ln f_p / ln e_p (the largest over the pairs)
    int nref = 0, K = 0;
    std::vector<int> kin(npairs, 0);
    for (int p = 0; p < npairs; ++p)
      if (h_st[p] == HOM_STATUS_STALLED || h_st[p] == HOM_STATUS_MAX_ITER) {
        mask[p] = 1;
        ++nref;
        const double e = h_e[p], f = opts->tol / (5.0 * e);
        double kd = h_it[p];
        if (e > 0.0 && e < 0.5 && f < 1.0 && f > 0.0) kd = h_it[p] * std::log(f) / std::log(e);
        kin[p] = opts->refine_inner > 0 ? opts->refine_inner
                                        : (int)std::ceil(std::min(std::max(kd, 10.0), 2.0 * std::max(h_it[p], 5)));
        K = std::max(K, kin[p]);
      }
    if (nref == 0) return HOM_OK;
    int* d_mask = reinterpret_cast<int*>(ws + o_mask);
    int* d_kin = d_mask + npairs;
    HOM_CUDA_TRY(cudaMemcpyAsync(d_mask, mask.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(d_kin, kin.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, st));
    auto book = [&](SolveArgs& X, int which) {  // bookkeeping block `which` (0: FP64 checks, 1: inner solves)
      int* ib = reinterpret_cast<int*>(ws + o_int2 + (size_t)which * ((size_t)npairs * 5 * sizeof(int) + 64));
      X.active = ib;
      X.iters = ib + npairs;
      X.status = ib + 2 * npairs;
      X.grow = ib + 3 * npairs;
      X.best_it = ib + 4 * npairs;
      X.it_dev = ib + 5 * npairs;
      X.nactive = ib + 5 * npairs + 1;
      X.done = done_word(ib, npairs);
      double* db = reinterpret_cast<double*>(ws + o_dbl2) + (size_t)which * npairs * (4 + nc);
      X.err = db;
      X.errn = db + npairs;
      X.last_err = db + 2 * (size_t)npairs;
      X.best_err = db + 3 * (size_t)npairs;
      X.mean_sigma = db + 4 * (size_t)npairs;
      X.diverge_window = 0;
      X.stall_window = 0;
      X.quiet = 0;  // the last check's mean stress and errors are the results, above tol too
      X.cond = 0;
      X.use_cond = 0;
    };
    SolveArgs A64 = A;  // FP64 checks: eps[0] = eps, eps[1] = F(eps)
    A64.hist = nullptr;  // the history holds the FP32 iteration only
    book(A64, 0);
    A64.plans = reinterpret_cast<const Plan*>(ws + o_plans64);
    A64.eps[0] = ws + o_e64a;
    A64.eps[1] = ws + o_e64b;
    A64.tau = ws + o_t64;
    A64.g = ws + o_g64;
    A64.max_iter = 1 << 30;
    A64.inner = 0;
    SolveArgs Ain = A;  // inner solves: FP32 buffers of the forward solve, zero mean strain, source r
    Ain.hist = nullptr;
    book(Ain, 1);
    Ain.E = reinterpret_cast<const double*>(ws + o_E0);
    Ain.src_mixed = ws + o_r32;
    Ain.tol = -1.0;
    Ain.max_iter = K;
    Ain.inner = 1;
    Ain.kinner = d_kin;
    A.kinner = d_kin;  // read by the update step
    const size_t smem_row64 = 2 * lay.smem_row, smem_green64 = 2 * lay.smem_green, smem_y64 = 2 * lay.smem_y;
    int rc;
    if ((rc = allow_smem(k_row<double, DIM, false, 15>, smem_row64)) != HOM_OK) return rc;
    if ((rc = allow_smem(k_green<double, DIM, 15>, smem_green64)) != HOM_OK) return rc;
    if (DIM == 3) {
      if ((rc = allow_smem(k_ypass<double, true, 15>, smem_y64)) != HOM_OK) return rc;
      if ((rc = allow_smem(k_ypass<double, false, 15>, smem_y64)) != HOM_OK) return rc;
    }
    const unsigned nR = (unsigned)lay.tR.size(), nC = (unsigned)lay.tC.size(), nY = (unsigned)lay.tY.size();
    const unsigned nctl = control_slices(lay);
    auto iter64 = [&]() {
      k_row<double, DIM, false, 15><<<nR, kThreads, smem_row64, st>>>(A64);
      if (DIM == 3) k_ypass<double, true, 15><<<nY, kThreads, smem_y64, st>>>(A64);
      k_green<double, DIM, 15><<<nC, kThreads, smem_green64, st>>>(A64);
      if (DIM == 3) k_ypass<double, false, 15><<<nY, kThreads, smem_y64, st>>>(A64);
      k_control<nc_of_dim<DIM>()><<<dim3((unsigned)npairs, nctl), kCtlThreads, 0, st>>>(A64);
    };
    auto iter32 = [&]() {
      k_row<float, DIM, false, MAXR><<<nR, kThreads, lay.smem_row, st>>>(Ain);
      if (DIM == 3) k_ypass<float, true, MAXR><<<nY, kThreads, lay.smem_y, st>>>(Ain);
      k_green<float, DIM, MAXR><<<nC, kThreads, lay.smem_green, st>>>(Ain);
      if (DIM == 3) k_ypass<float, false, MAXR><<<nY, kThreads, lay.smem_y, st>>>(Ain);
      k_control<nc_of_dim<DIM>()><<<dim3((unsigned)npairs, nctl), kCtlThreads, 0, st>>>(Ain);
    };
    const dim3 eg(64, (unsigned)npairs);
    float2* e32a = static_cast<float2*>(A.eps[0]);
    float2* e32b = static_cast<float2*>(A.eps[1]);
    float2* g32 = static_cast<float2*>(A.g);
    double2* e64a = reinterpret_cast<double2*>(ws + o_e64a);
    double2* e64b = reinterpret_cast<double2*>(ws + o_e64b);
    double2* g64 = reinterpret_cast<double2*>(ws + o_g64);
    float2* r32 = reinterpret_cast<float2*>(ws + o_r32);
    k_refine<kRefStart><<<eg, 256, 0, st>>>(A, d_mask, e32a, e32b, g32, e64a, e64b, g64, r32, 0);
    std::vector<int> h_st64(npairs), extra(npairs, 0), conv(npairs, 0);
    int steps = 0;
    for (;;) {
      // FP64 check of the current iterate (and F of it)
      k_init_pairs_masked<<<(npairs + 255) / 256, 256, 0, st>>>(A64, d_mask);
      iter64();
      HOM_CUDA_TRY(cudaGetLastError());
      HOM_CUDA_TRY(cudaMemcpyAsync(h_st64.data(), A64.status, npairs * sizeof(int), cudaMemcpyDeviceToHost, st));
      HOM_CUDA_TRY(cudaStreamSynchronize(st));
      int left = 0;
      for (int p = 0; p < npairs; ++p)
        if (mask[p]) {
          extra[p] += 1;
          if (h_st64[p] == HOM_STATUS_CONVERGED) {
            mask[p] = 0;
            conv[p] = 1;  // its FP64 results stay in the check's arrays: later checks skip it
          } else {
            ++left;
          }
        }
      if (left == 0 || steps >= opts->refine) break;
      HOM_CUDA_TRY(cudaMemcpyAsync(d_mask, mask.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, st));
      // the correction: K + 1 FP32 iterations of delta <- r + F0(delta) from delta = r
      k_refine<kRefResid><<<eg, 256, 0, st>>>(A, d_mask, e32a, e32b, g32, e64a, e64b, g64, r32, 0);
      k_refine_inner_start<<<eg, 256, 0, st>>>(A, d_mask, r32, e32a);
      k_init_pairs_masked<<<(npairs + 255) / 256, 256, 0, st>>>(Ain, d_mask);
      for (int k = 0; k <= K; ++k) iter32();
      k_refine<kRefUpdate><<<eg, 256, 0, st>>>(A, d_mask, e32a, e32b, g32, e64a, e64b, g64, r32, K);
      HOM_CUDA_TRY(cudaGetLastError());
      for (int p = 0; p < npairs; ++p)
        if (mask[p]) extra[p] += kin[p] + 1;
      ++steps;
    }
    // results of the refined pairs: the FP64 check's mean stress and errors, the iterate rounded to
    // FP32 in the buffer the output pass reads, status converged or (after opts->refine corrections)
    // the one the FP32 iteration had
    std::vector<int> all(npairs, 0);
    for (int p = 0; p < npairs; ++p)
      if (h_st[p] == HOM_STATUS_STALLED || h_st[p] == HOM_STATUS_MAX_ITER) all[p] = 1;
    HOM_CUDA_TRY(cudaMemcpyAsync(d_mask, all.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, st));
    std::vector<double> ms((size_t)npairs * nc), err(npairs), errn(npairs), ms64((size_t)npairs * nc), e64(npairs),
        en64(npairs);
    HOM_CUDA_TRY(cudaMemcpyAsync(ms.data(), A.mean_sigma, ms.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(err.data(), A.err, npairs * sizeof(double), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(errn.data(), A.errn, npairs * sizeof(double), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(ms64.data(), A64.mean_sigma, ms64.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(e64.data(), A64.err, npairs * sizeof(double), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(en64.data(), A64.errn, npairs * sizeof(double), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));
    for (int p = 0; p < npairs; ++p)
      if (all[p]) {
        for (int k = 0; k < nc; ++k) ms[(size_t)p * nc + k] = ms64[(size_t)p * nc + k];
        err[p] = e64[p];
        errn[p] = en64[p];
        if (conv[p]) h_st[p] = HOM_STATUS_CONVERGED;
        h_it[p] += extra[p];
      }
    HOM_CUDA_TRY(cudaMemcpyAsync(A.mean_sigma, ms.data(), ms.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(A.err, err.data(), npairs * sizeof(double), cudaMemcpyHostToDevice, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(A.errn, errn.data(), npairs * sizeof(double), cudaMemcpyHostToDevice, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(A.status, h_st.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(A.iters, h_it.data(), npairs * sizeof(int), cudaMemcpyHostToDevice, st));
    k_refine<kRefFinal><<<eg, 256, 0, st>>>(A, d_mask, e32a, e32b, g32, e64a, e64b, g64, r32, 0);
    HOM_CUDA_TRY(cudaGetLastError());
    HOM_CUDA_TRY(cudaStreamSynchronize(st));  // the host vectors above go out of scope
    return HOM_OK;
  }
}

template <typename T, int DIM, int MAXR>
int run_solve(const hom_cell* cells, int ncells, const hom_material* mat, const double* E, int L, const double* c0,
              const hom_solve_opts* opts, hom_result* out, cudaStream_t st, const ExternalWorkspace* ext,
              const AdjointSpec* adj, bool cg) {
  using V = typename Cx<T>::V;
  const int nc = nc_of(DIM);
  Layout lay;
  // Conjugate gradients run on the generic passes with the reference medium c0 = s I per cell, s the
  // smallest eigenvalue of the cell's phase stiffnesses (isotropic: min(2 mu, dim lambda + 2 mu))
  std::vector<double> c0_cg;
  if (cg) {
    const int ns = DIM == 2 ? 6 : 21;
    std::vector<double> ph((size_t)mat->nphase * ns);
    HOM_CUDA_TRY(cudaMemcpy(ph.data(), mat->phase_c64, ph.size() * sizeof(double), cudaMemcpyDeviceToHost));
    auto smin = [&](int q) {
      const double lam = ph[(size_t)q * ns + 1], mu2 = ph[(size_t)q * ns] - lam;
      return std::min(mu2, DIM * lam + mu2);
    };
    c0_cg.resize(2 * (size_t)ncells);
    for (int i = 0; i < ncells; ++i) {
      double sm = smin(cells[i].matrix_phase);
      for (int q = 0; q < cells[i].nprim; ++q) sm = std::min(sm, smin(cells[i].prims[q].phase));
      if (!(sm > 0.0)) return set_error(HOM_ERR_INVALID_ARG, "hom_solve_cg: cell %d has a phase that is not positive definite", i);
      c0_cg[2 * i] = 0.0;
      c0_cg[2 * i + 1] = 0.5 * sm;
    }
    c0 = c0_cg.data();
  }
  // opts->passes == HOM_PASSES_GENERIC keeps every solve on the generic passes
  // defect correction (FP32 with FP64 residuals) runs on the generic passes: FP32 and FP64 states
  // then share one layout
  const bool refine = std::is_same<T, float>::value && opts->refine > 0 && !cg && !adj && !ext;
  const bool em = opts->scheme == HOM_SCHEME_EYRE_MILTON && !cg && !adj && !ext;
  // a warm start converts the caller's real field on the generic passes' layout
  const bool warm = opts->warm_start != 0 && !cg && !adj && !ext;
  if (warm && !out->eps) return set_error(HOM_ERR_INVALID_ARG, "hom_solve: a warm start without an initial field");
  lay.fast = std::is_same<T, float>::value && !cg && opts->passes != HOM_PASSES_GENERIC &&
             opts->green == HOM_GREEN_CONTINUOUS && !refine && !warm;
  lay.compact = ext && ext->compact;
  const bool chip = DIM == 2 && !adj && !out->stats && !lay.compact;  // the on-chip solver may run
  int rc = build_layout(cells, ncells, L, DIM, sizeof(V), MAXR, c0, ext != nullptr, lay, em, chip);
  if (rc != HOM_OK) return rc;
  const int npairs = ncells * L;
  const bool want_fields = out->eps || out->sigma;
  const bool eps_dev = is_device_ptr(out->eps), sig_dev = is_device_ptr(out->sigma);
  const bool need_stage = want_fields && ((out->eps && !eps_dev) || (out->sigma && !sig_dev));

  // workspace carve-up
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  };
  const size_t o_eps0 = take(lay.ws_elems * sizeof(V)), o_eps1 = take(lay.ws_elems * sizeof(V)),
               o_tau = take(lay.ws_elems * sizeof(V)), o_g = take(lay.g_elems * sizeof(V));
  const size_t o_partR = take(lay.tR.size() * (size_t)L * nc * sizeof(double));
  const size_t o_partC = take(lay.tC.size() * 2 * sizeof(double));
  const size_t o_cells = take(lay.cells.size() * sizeof(CellDev)), o_plans = take(lay.plans.size() * sizeof(Plan));
  const size_t o_tR = take(lay.tR.size() * sizeof(TaskR)), o_tC = take(lay.tC.size() * sizeof(TaskL)),
               o_tY = take(std::max<size_t>(1, lay.tY.size()) * sizeof(TaskL));
  const size_t o_pairs = take(lay.pairs.size() * sizeof(PairDev));
  const size_t o_E = take((size_t)npairs * nc * sizeof(double));
  const size_t o_int = take((size_t)npairs * 5 * sizeof(int) + 64);
  const size_t o_dbl = take((size_t)npairs * (4 + nc) * sizeof(double));
  const size_t o_bytes = take(HOM_NKERNEL * sizeof(unsigned long long));
  const unsigned slices = control_slices(lay);  // only pairs of many tasks have partial sums to exchange
  const size_t o_ctlp = slices > 1 ? take((size_t)npairs * slices * (nc + 3) * sizeof(double)) : 0;
  const size_t o_ctlc = slices > 1 ? take((size_t)npairs * sizeof(int)) : 0;
  const size_t o_res0 = adj ? take((size_t)npairs * 2 * sizeof(double)) : 0;
  constexpr int NS = DIM == 2 ? 6 : 21;
  const size_t o_partE = em ? take(lay.tC.size() * sizeof(double)) : 0;
  const size_t o_errc = em ? take((size_t)npairs * sizeof(double)) : 0;
  const size_t o_minv = em ? take((size_t)std::max<int64_t>(1, mat->mixed_count) * NS * sizeof(T)) : 0;
  const size_t o_dbg = take(4 * sizeof(unsigned int));
  const bool hist_dev = is_device_ptr(out->history);
  const size_t hist_elems = out->history ? (size_t)npairs * ((size_t)opts->max_iter + 1) : 0;
  const size_t o_hist = out->history && !hist_dev ? take(hist_elems * sizeof(double)) : 0;
  int cg_nchunk = 1;
  for (const CellDev& c : lay.cells)
    cg_nchunk = std::max(cg_nchunk, (c.nrows + cg_rows_per_cta(c.Hp, nc, c.nrows) - 1) / cg_rows_per_cta(c.Hp, nc, c.nrows));
  if (cg && cg_nchunk > 65535) return set_error(HOM_ERR_UNSUPPORTED_SIZE, "hom_solve_cg: cell too large");
  const size_t o_cgx = cg ? take(lay.ws_elems * sizeof(V)) : 0, o_cgr = cg ? take(lay.ws_elems * sizeof(V)) : 0;
  const size_t o_cgpart = cg ? take((size_t)npairs * cg_nchunk * sizeof(double)) : 0;
  const size_t o_cgsc = cg ? take((size_t)npairs * (3 + nc) * sizeof(double)) : 0;
  const size_t o_cgint = cg ? take((size_t)npairs * 2 * sizeof(int)) : 0;
  const size_t o_E0 = cg || refine ? take((size_t)npairs * nc * sizeof(double)) : 0;
  // defect correction: FP64 strain state (current and F of it), FP64 tau and g, the FP32 residual,
  // FP64 plans (register radix 15), and bookkeeping of the FP64 checks and of the inner solves
  const size_t o_e64a = refine ? take(lay.ws_elems * sizeof(double2)) : 0;
  const size_t o_e64b = refine ? take(lay.ws_elems * sizeof(double2)) : 0;
  const size_t o_t64 = refine ? take(lay.ws_elems * sizeof(double2)) : 0;
  const size_t o_g64 = refine ? take(lay.g_elems * sizeof(double2)) : 0;
  const size_t o_r32 = refine ? take(lay.ws_elems * sizeof(V)) : 0;
  const size_t o_int2 = refine ? take(2 * ((size_t)npairs * 5 * sizeof(int) + 64)) : 0;
  const size_t o_dbl2 = refine ? take(2 * (size_t)npairs * (4 + nc) * sizeof(double)) : 0;
  const size_t o_mask = refine ? take(2 * (size_t)npairs * sizeof(int)) : 0;
  const size_t o_plans64 = refine ? take(lay.plans.size() * sizeof(Plan)) : 0;
  long long nv_all = 0, nv_max = 0;
  for (CellDev& c : lay.cells) {
    c.lp_off = nv_all;  // one-byte labels, rows padded to 16 bytes
    nv_all += (long long)c.nrows * ((c.n + 15) / 16 * 16);
    nv_max = std::max(nv_max, c.nv);
  }
  const size_t o_lperm = lay.fast ? take((size_t)nv_all) : 0;
  // pure-voxel phases of each cell: the matrix phase and its primitives' phases (one-byte local index)
  std::vector<int> cell_phases;
  int nph_max = 1;
  if (lay.fast) {
    for (int ci = 0; ci < ncells; ++ci) {
      std::vector<int> ph{cells[ci].matrix_phase};
      for (int p = 0; p < cells[ci].nprim; ++p) ph.push_back(cells[ci].prims[p].phase);
      std::sort(ph.begin(), ph.end());
      ph.erase(std::unique(ph.begin(), ph.end()), ph.end());
      if (ph.size() > 254) return set_error(HOM_ERR_UNSUPPORTED_SIZE, "cell %d holds more than 254 phases", ci);
      lay.cells[ci].ph_off = (int)cell_phases.size();
      lay.cells[ci].nph = (int)ph.size();
      nph_max = std::max(nph_max, (int)ph.size());
      cell_phases.insert(cell_phases.end(), ph.begin(), ph.end());
    }
  }
  const size_t o_cphase = lay.fast ? take(cell_phases.size() * sizeof(int)) : 0;
  const bool on_chip = lay.fast && chip;
  const size_t o_reslist = on_chip ? take((size_t)npairs * sizeof(int)) : 0;
  const size_t o_fplans = lay.fast ? take(lay.fplans.size() * sizeof(FastPlanDev)) : 0;
  const size_t o_stage_e = need_stage && out->eps && !eps_dev ? take(lay.fld_elems * sizeof(T)) : 0;
  const size_t o_stage_s = need_stage && out->sigma && !sig_dev ? take(lay.fld_elems * sizeof(T)) : 0;
  const size_t host_lo = o_cells, host_hi = o_int;  // tables uploaded in one copy
  // external workspace: the plan tables follow the scratch
  std::vector<size_t> o_plan_tab(lay.host_plans.size()), o_fplan_tab(lay.fplan_host.size());
  for (size_t i = 0; i < lay.host_plans.size(); ++i) o_plan_tab[i] = take(plan_table_bytes(lay.host_plans[i].n));
  for (size_t i = 0; i < lay.fplan_host.size(); ++i) o_fplan_tab[i] = take(lay.fplan_host[i].size());
  void* wsv = nullptr;
  if (ext) {
    // What speed costs in scratch goes first (partial sums of more tasks and control CTAs), then the passes
    // with plan-read radices: the generic ones take less (no one-byte labels).
    if (off > ext->capacity && (!ext->compact || lay.run)) {
      ExternalWorkspace least = *ext;
      hom_solve_opts g = *opts;
      if (ext->compact) g.passes = HOM_PASSES_GENERIC;
      least.compact = true;
      return run_solve<T, DIM, MAXR>(cells, ncells, mat, E, L, c0, &g, out, st, &least, adj, cg);
    }
    if (off > ext->capacity)
      return set_error(HOM_ERR_UNSUPPORTED_SIZE,
                       "this batch needs %zu bytes of solver scratch; the fixed scratch array holds %zu bytes", off,
                       ext->capacity);
    wsv = ext->base;
  } else {
    rc = get_workspace(off, &wsv);
    if (rc != HOM_OK) return rc;
  }
  unsigned char* ws = static_cast<unsigned char*>(wsv);
  std::vector<unsigned char> plan_host;
  for (size_t i = 0; i < lay.host_plans.size(); ++i) {
    const HostPlan& hp = lay.host_plans[i];
    plan_host.assign(plan_table_bytes(hp.n), 0);
    fill_plan_tables(hp, plan_host.data());
    HOM_CUDA_TRY(cudaMemcpyAsync(ws + o_plan_tab[i], plan_host.data(), plan_host.size(), cudaMemcpyHostToDevice, st));
    if (ext) HOM_CUDA_TRY(cudaStreamSynchronize(st));  // plan_host is reused for the next table
    set_plan_pointers(lay.plans[i], ws + o_plan_tab[i]);
  }
  for (size_t i = 0; i < lay.fplan_host.size(); ++i) {
    HOM_CUDA_TRY(cudaMemcpyAsync(ws + o_fplan_tab[i], lay.fplan_host[i].data(), lay.fplan_host[i].size(),
                                 cudaMemcpyHostToDevice, st));
    fast2d_plan_rebase(lay.fplans[i], ws + o_fplan_tab[i]);
  }
  if (ext) HOM_CUDA_TRY(cudaStreamSynchronize(st));  // the host staging vectors above go out of scope
  {
    std::vector<unsigned char> h(host_hi - host_lo, 0);
    auto put = [&](size_t o, const void* src, size_t b) {
      if (b) std::memcpy(h.data() + (o - host_lo), src, b);
    };
    put(o_cells, lay.cells.data(), lay.cells.size() * sizeof(CellDev));
    put(o_plans, lay.plans.data(), lay.plans.size() * sizeof(Plan));
    put(o_tR, lay.tR.data(), lay.tR.size() * sizeof(TaskR));
    put(o_tC, lay.tC.data(), lay.tC.size() * sizeof(TaskL));
    put(o_tY, lay.tY.data(), lay.tY.size() * sizeof(TaskL));
    put(o_pairs, lay.pairs.data(), lay.pairs.size() * sizeof(PairDev));
    put(o_E, E, (size_t)npairs * nc * sizeof(double));
    HOM_CUDA_TRY(cudaMemcpyAsync(ws + host_lo, h.data(), h.size(), cudaMemcpyHostToDevice, st));
    if (lay.fast) {
      HOM_CUDA_TRY(cudaMemcpyAsync(ws + o_fplans, lay.fplans.data(), lay.fplans.size() * sizeof(FastPlanDev),
                                   cudaMemcpyHostToDevice, st));
      HOM_CUDA_TRY(cudaMemcpyAsync(ws + o_cphase, cell_phases.data(), cell_phases.size() * sizeof(int),
                                   cudaMemcpyHostToDevice, st));
      HOM_CUDA_TRY(cudaStreamSynchronize(st));  // the staging vector goes out of scope
    }
  }
  HOM_CUDA_TRY(cudaMemsetAsync(ws + o_eps0, 0, lay.ws_elems * sizeof(V), st));
  HOM_CUDA_TRY(cudaMemsetAsync(ws + o_g, 0, lay.g_elems * sizeof(V), st));
  HOM_CUDA_TRY(cudaMemsetAsync(ws + o_bytes, 0, HOM_NKERNEL * sizeof(unsigned long long), st));
  if (slices > 1) HOM_CUDA_TRY(cudaMemsetAsync(ws + o_ctlc, 0, (size_t)npairs * sizeof(int), st));
  HOM_CUDA_TRY(cudaMemsetAsync(ws + o_dbg, 0, 4 * sizeof(unsigned int), st));
  if (out->history && !hist_dev)  // staged: the entries the solve does not write keep the caller's values
    HOM_CUDA_TRY(cudaMemcpyAsync(ws + o_hist, out->history, hist_elems * sizeof(double), cudaMemcpyHostToDevice, st));
  if (refine) {
    HOM_CUDA_TRY(cudaMemsetAsync(ws + o_E0, 0, (size_t)npairs * nc * sizeof(double), st));
    std::vector<Plan> p64(lay.plans.size());
    for (size_t i = 0; i < lay.plans.size(); ++i)
      if ((rc = get_plan(lay.plans[i].n, 15, &p64[i])) != HOM_OK) return rc;
    HOM_CUDA_TRY(cudaMemcpyAsync(ws + o_plans64, p64.data(), p64.size() * sizeof(Plan), cudaMemcpyHostToDevice, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));  // p64 goes out of scope
  }
  if (cg) {
    HOM_CUDA_TRY(cudaMemsetAsync(ws + o_E0, 0, (size_t)npairs * nc * sizeof(double), st));
    HOM_CUDA_TRY(cudaMemsetAsync(ws + o_cgint, 0, (size_t)npairs * 2 * sizeof(int), st));
  }

  SolveArgs A;
  std::memset(&A, 0, sizeof(A));  // the bytes of A key the graph cache: no stray padding
  A.cells = reinterpret_cast<const CellDev*>(ws + o_cells);
  A.plans = reinterpret_cast<const Plan*>(ws + o_plans);
  A.label = mat->label;
  A.mixed_c32 = mat->mixed_c32;
  A.mixed_c64 = mat->mixed_c64;
  A.phase_c32 = mat->phase_c32;
  A.phase_c64 = mat->phase_c64;
  A.E = reinterpret_cast<const double*>(ws + o_E);
  A.eps[0] = ws + o_eps0;
  A.eps[1] = ws + o_eps1;
  A.tau = ws + o_tau;
  A.g = ws + o_g;
  A.partR = reinterpret_cast<double*>(ws + o_partR);
  A.partC = reinterpret_cast<double*>(ws + o_partC);
  A.tR = reinterpret_cast<const TaskR*>(ws + o_tR);
  A.tC = reinterpret_cast<const TaskL*>(ws + o_tC);
  A.tY = reinterpret_cast<const TaskL*>(ws + o_tY);
  A.pairs = reinterpret_cast<const PairDev*>(ws + o_pairs);
  A.npairs = npairs;
  int* ib = reinterpret_cast<int*>(ws + o_int);
  A.active = ib;
  A.iters = ib + npairs;
  A.status = ib + 2 * npairs;
  A.grow = ib + 3 * npairs;
  A.best_it = ib + 4 * npairs;
  A.it_dev = ib + 5 * npairs;
  A.nactive = ib + 5 * npairs + 1;
  A.done = done_word(ib, npairs);
  double* db = reinterpret_cast<double*>(ws + o_dbl);
  A.err = db;
  A.errn = db + npairs;
  A.last_err = db + 2 * npairs;
  A.best_err = db + 3 * npairs;
  A.mean_sigma = db + 4 * npairs;
  A.bytes = reinterpret_cast<unsigned long long*>(ws + o_bytes);
  A.ctl_part = slices > 1 ? reinterpret_cast<double*>(ws + o_ctlp) : nullptr;
  A.ctl_cnt = slices > 1 ? reinterpret_cast<int*>(ws + o_ctlc) : nullptr;
  A.L = L;
  A.criterion = opts->criterion;
  A.max_iter = opts->max_iter;
  A.green = opts->green;
  A.diverge_window = opts->diverge_window;
  // defect correction starts from where the FP32 iteration stagnates (30 iterations by default)
  A.stall_window = opts->stall_window > 0 ? opts->stall_window : (refine ? 30 : 0);
  A.tol = opts->tol;
  A.out_eps = out->eps ? (eps_dev ? out->eps : (void*)(ws + o_stage_e)) : nullptr;
  A.out_sig = out->sigma ? (sig_dev ? out->sigma : (void*)(ws + o_stage_s)) : nullptr;
  A.src = adj ? adj->source : nullptr;
  A.res0 = adj ? reinterpret_cast<double*>(ws + o_res0) : nullptr;
  A.scheme = em ? HOM_SCHEME_EYRE_MILTON : HOM_SCHEME_BASIC;
  A.warm = warm ? 1 : 0;
  A.dbg = reinterpret_cast<unsigned int*>(ws + o_dbg);
  A.n_ws = lay.ws_elems;
  A.n_g = lay.g_elems;
  A.n_fld = lay.fld_elems;
  A.n_lab = (size_t)vox_total(lay);
  A.hist = out->history ? (hist_dev ? out->history : reinterpret_cast<double*>(ws + o_hist)) : nullptr;
  A.partE = em ? reinterpret_cast<double*>(ws + o_partE) : nullptr;
  A.errc = em ? reinterpret_cast<double*>(ws + o_errc) : nullptr;
  A.em_minv = em ? ws + o_minv : nullptr;
  A.quiet = !adj && !warm && !A.hist && A.diverge_window == 0 && A.stall_window == 0;
  A.fplans = lay.fast ? reinterpret_cast<const FastPlanDev*>(ws + o_fplans) : nullptr;
  A.label8 = lay.fast ? reinterpret_cast<const uint8_t*>(ws + o_lperm) : nullptr;
  A.cell_phases = lay.fast ? reinterpret_cast<const int*>(ws + o_cphase) : nullptr;
  CgArgs G{};
  if (cg) {
    G.x = ws + o_cgx;
    G.r = ws + o_cgr;
    G.part = reinterpret_cast<double*>(ws + o_cgpart);
    double* sc = reinterpret_cast<double*>(ws + o_cgsc);
    G.rr = sc;
    G.alpha = sc + npairs;
    G.beta = sc + 2 * (size_t)npairs;
    G.ssum = sc + 3 * (size_t)npairs;
    G.vmode = reinterpret_cast<int*>(ws + o_cgint);
    G.steps = G.vmode + npairs;
    G.E = A.E;
    G.nchunk = cg_nchunk;
  }
  size_t smem_frow = 0, smem_fout = 0, smem_fgreen = 0, smem_fy = 0;  // the largest over the batch's sizes
  for (const FastPlanDev& fp : lay.fplans) {
    smem_frow = std::max(smem_frow, DIM == 2 ? fast2d_smem_row(fp.n, nph_max) : fast3d_smem_row(fp.n, nph_max));
    smem_fout = std::max(smem_fout, smem_frow + ((size_t)fp.n * sizeof(uint16_t) + 15) / 16 * 16);
    smem_fgreen = std::max(smem_fgreen, DIM == 2 ? fast2d_smem_green(fp.n) : fast3d_smem_green(fp.n));
    if (DIM == 3) smem_fy = std::max(smem_fy, fast3d_smem_y(fp.n));
  }
  if (lay.fast && (rc = fast2d_permute_labels(A, ncells, nv_max, st)) != HOM_OK) return rc;

  if (warm && (rc = allow_smem(k_state_in<T, DIM, MAXR>, lay.smem_row)) != HOM_OK) return rc;
  if (em) {
    if ((rc = allow_smem(k_row<T, DIM, false, MAXR, true>, lay.smem_row)) != HOM_OK) return rc;
    if ((rc = allow_smem(k_row<T, DIM, true, MAXR, true>, lay.smem_row)) != HOM_OK) return rc;
    if ((rc = allow_smem(k_green<T, DIM, MAXR, true>, lay.smem_green)) != HOM_OK) return rc;
  } else {
    if ((rc = allow_smem(k_row<T, DIM, false, MAXR>, lay.smem_row)) != HOM_OK) return rc;
    if ((rc = allow_smem(k_row<T, DIM, true, MAXR>, lay.smem_row)) != HOM_OK) return rc;
    if ((rc = allow_smem(k_green<T, DIM, MAXR>, lay.smem_green)) != HOM_OK) return rc;
  }
  if (DIM == 3) {
    if ((rc = allow_smem(k_ypass<T, true, MAXR>, lay.smem_y)) != HOM_OK) return rc;
    if ((rc = allow_smem(k_ypass<T, false, MAXR>, lay.smem_y)) != HOM_OK) return rc;
  }

  Timer tm{out->stats, st, {}};
  const unsigned nR = (unsigned)lay.tR.size(), nC = (unsigned)lay.tC.size(), nY = (unsigned)lay.tY.size();
  NvtxRange nvtx_init_("hom_solve: initial state");
  const unsigned nCtl = (unsigned)npairs, nctl = control_slices(lay);  // control CTAs: (cell, load) pairs x slices
  tm.begin(HOM_K_INIT);
  k_init_pairs<<<(npairs + 255) / 256, 256, 0, st>>>(A);
  if (em) {
    if (ncells > 65535) return set_error(HOM_ERR_UNSUPPORTED_SIZE, "Eyre-Milton scheme: more than 65535 cells");
    HOM_CUDA_TRY(cudaMemsetAsync(ws + o_errc, 0, (size_t)npairs * sizeof(double), st));
    k_em_minv<T, DIM == 2 ? 3 : 6><<<dim3(64, (unsigned)ncells), kMinvThreads, 0, st>>>(A, reinterpret_cast<T*>(ws + o_minv));
  }
  if (lay.fast && DIM == 3) {
    fast3d_init(A, ncells, st);
  } else if (lay.fast) {
    fast2d_init(A, ncells, st);
  } else if (warm) {
    k_state_in<T, DIM, MAXR><<<nR, kThreads, lay.smem_row, st>>>(A, static_cast<const T*>(out->eps));
  } else if (em) {
    dim3 grid(64, (unsigned)std::min(ncells, 65535));
    k_init<T, true><<<grid, 256, 0, st>>>(A, ncells, nc);
  } else {
    dim3 grid(64, (unsigned)std::min(ncells, 65535));
    k_init<T><<<grid, 256, 0, st>>>(A, ncells, nc);
  }
  tm.end();
  nvtx_init_.end();
  HOM_CUDA_TRY(cudaGetLastError());

  const int check = opts->check_every > 0 ? opts->check_every : 8;
  int host_nactive = npairs;
  if (on_chip) {
    // pairs on small grids run to their own stopping point on chip; the passes below see them inactive
    int nres = 0;
    if ((rc = resident2d_solve(A, lay.cells, lay.fplans, L, lay.run_max, reinterpret_cast<int*>(ws + o_reslist),
                               nph_max, st, &nres)) != HOM_OK)
      return rc;
    host_nactive -= nres;
  }
  int launched = 0;
  const dim3 cg_grid((unsigned)npairs, (unsigned)cg_nchunk);
  int pass_rc = HOM_OK;  // the first pass that could not be launched
  auto launched_ok = [&](int r) {
    if (pass_rc == HOM_OK) pass_rc = r;
  };
  auto one_pass = [&]() {
    NvtxRange r_("hom_solve: passes");
    tm.begin(HOM_K_ROW);
    if (lay.fast && DIM == 3) launched_ok(fast3d_row(A, nR, smem_frow, false, lay.run_max, st));
    else if (lay.fast) launched_ok(fast2d_row(A, nR, smem_frow, lay.run_max, st));
    else if (em) k_row<T, DIM, false, MAXR, true><<<nR, kThreads, lay.smem_row, st>>>(A);
    else k_row<T, DIM, false, MAXR><<<nR, kThreads, lay.smem_row, st>>>(A);
    tm.end();
    if (DIM == 3) {
      tm.begin(HOM_K_YFWD);
      if (lay.fast) launched_ok(fast3d_ypass(A, nY, smem_fy, true, lay.run_max, st));
      else k_ypass<T, true, MAXR><<<nY, kThreads, lay.smem_y, st>>>(A);
      tm.end();
    }
    tm.begin(HOM_K_GREEN);
    if (lay.fast && DIM == 3) launched_ok(fast3d_green(A, nC, smem_fgreen, lay.run_max, st));
    else if (lay.fast) launched_ok(fast2d_green(A, nC, smem_fgreen, lay.run_max, st));
    else if (em) k_green<T, DIM, MAXR, true><<<nC, kThreads, lay.smem_green, st>>>(A);
    else k_green<T, DIM, MAXR><<<nC, kThreads, lay.smem_green, st>>>(A);
    tm.end();
    if (DIM == 3) {
      tm.begin(HOM_K_YINV);
      if (lay.fast) launched_ok(fast3d_ypass(A, nY, smem_fy, false, lay.run_max, st));
      else k_ypass<T, false, MAXR><<<nY, kThreads, lay.smem_y, st>>>(A);
      tm.end();
    }
  };
  auto one_iteration = [&]() {
    one_pass();
    tm.begin(HOM_K_CONTROL);
    if (cg) {
      k_cg_elems<T, DIM, kCgPq><<<cg_grid, kCgThreads, 0, st>>>(A, G);
      k_cg_control<kCgPq><<<nCtl, kCgCtlThreads, 0, st>>>(A, G, nc);
      k_cg_elems<T, DIM, kCgUpdate><<<cg_grid, kCgThreads, 0, st>>>(A, G);
      k_cg_control<kCgUpdate><<<nCtl, kCgCtlThreads, 0, st>>>(A, G, nc);
      k_cg_elems<T, DIM, kCgDir><<<cg_grid, kCgThreads, 0, st>>>(A, G);
    } else {
      k_control<nc_of_dim<DIM>()><<<dim3(nCtl, nctl), kCtlThreads, 0, st>>>(A);
    }
    tm.end();
  };
  if (cg) {
    // start: the passes on the uniform field E with zero mean strain give the first residual
    A.E = reinterpret_cast<const double*>(ws + o_E0);
    one_pass();
    tm.begin(HOM_K_CONTROL);
    k_cg_elems<T, DIM, kCgStart><<<cg_grid, kCgThreads, 0, st>>>(A, G);
    k_cg_control<kCgStart><<<nCtl, kCgCtlThreads, 0, st>>>(A, G, nc);
    tm.end();
    HOM_CUDA_TRY(cudaGetLastError());
    HOM_CUDA_TRY(cudaMemcpyAsync(&host_nactive, A.nactive, sizeof(int), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));
  }
  NvtxRange nvtx_iter_("hom_solve: iterations");
  if (opts->use_graph && !out->stats && !cg && host_nactive > 0) {
    // The whole solve as one graph launch: a conditional WHILE node whose body is one iteration
    // (the passes and the control kernel); the control kernel clears the condition once no pair is
    // active or max_iter + 1 iterations ran, so the host waits once instead of polling.  The body
    // is captured on a private stream (the legacy default stream cannot be captured); the
    // instantiated graph is cached across calls with the same arguments.
    int dev = 0;
    HOM_CUDA_TRY(cudaGetDevice(&dev));
    SolveArgs K = A;  // the output buffers are not used by the iterations: not part of the key
    K.out_eps = K.out_sig = nullptr;
    std::string key(reinterpret_cast<const char*>(&K), sizeof(K));
    const size_t dims[] = {nR, nC, nY, nCtl, nctl, lay.smem_row, lay.smem_green, lay.smem_y, smem_frow, smem_fgreen,
                           smem_fy, (size_t)lay.fast, (size_t)lay.run_max, (size_t)DIM, sizeof(T), (size_t)MAXR};
    key.append(reinterpret_cast<const char*>(dims), sizeof(dims));
    cudaGraphExec_t gexec = find_graph(dev, key);
    if (!gexec) {
      cudaGraph_t graph = nullptr;
      cudaStream_t cap = nullptr;
      HOM_CUDA_TRY(cudaGraphCreate(&graph, 0));
      cudaGraphConditionalHandle h{};
      cudaGraphNode_t node{};
      cudaGraphNodeParams cp{};
      cudaError_t ce = cudaGraphConditionalHandleCreate(&h, graph, 1u, cudaGraphCondAssignDefault);
      if (ce == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        ce = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &cp);
      }
      if (ce == cudaSuccess) ce = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
      if (ce == cudaSuccess)
        ce = cudaStreamBeginCaptureToGraph(cap, cp.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                           cudaStreamCaptureModeThreadLocal);
      if (ce == cudaSuccess) {
        const cudaStream_t user = st;
        st = cap;  // the launch lambdas use `st`
        A.cond = h;
        A.use_cond = 1;
        one_iteration();
        A.cond = 0;
        A.use_cond = 0;
        st = user;
        cudaGraph_t body = nullptr;
        ce = cudaStreamEndCapture(cap, &body);
      }
      if (ce == cudaSuccess && pass_rc == HOM_OK) ce = cudaGraphInstantiate(&gexec, graph, 0);
      if (cap) cudaStreamDestroy(cap);
      cudaGraphDestroy(graph);
      if (pass_rc != HOM_OK) {
        cudaGetLastError();
        return pass_rc;
      }
      if (ce != cudaSuccess) {
        cudaGetLastError();
        return set_error(HOM_ERR_CUDA, "whole-solve graph: %s", cudaGetErrorString(ce));
      }
      keep_graph(dev, key, gexec);
    }
    HOM_CUDA_TRY(cudaGraphLaunch(gexec, st));
    HOM_CUDA_TRY(cudaMemcpyAsync(&host_nactive, A.nactive, sizeof(int), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));
  }
  while (host_nactive > 0 && !(opts->use_graph && !out->stats && !cg)) {
    // CG: a verification pass takes a launch without a step, and is followed by a step or a stop
    const int remaining = (cg ? 2 * opts->max_iter + 2 : opts->max_iter + 1) - launched;
    if (remaining <= 0) break;  // the control kernel has stopped every pair by now
    const int k = std::min(check, remaining);
    for (int i = 0; i < k; ++i) one_iteration();
    launched += k;
    if (pass_rc != HOM_OK) return pass_rc;
    HOM_CUDA_TRY(cudaGetLastError());
    HOM_CUDA_TRY(cudaMemcpyAsync(&host_nactive, A.nactive, sizeof(int), cudaMemcpyDeviceToHost, st));
    HOM_CUDA_TRY(cudaStreamSynchronize(st));
  }
  nvtx_iter_.end();
  if (host_nactive > 0) return set_error(HOM_ERR_TIMEOUT, "iteration control did not terminate");
  if (cg) {
    // the returned iterate E + x, in the buffer the output pass reads for each pair
    k_cg_elems<T, DIM, kCgFinal><<<cg_grid, kCgThreads, 0, st>>>(A, G);
    HOM_CUDA_TRY(cudaGetLastError());
  }

  if (refine) {
    NvtxRange r_("hom_solve: defect correction");
    rc = refine_solve<T, DIM, MAXR>(A, ws, npairs, nc, opts, lay, o_e64a, o_e64b, o_t64, o_g64, o_r32, o_int2, o_dbl2,
                                    o_mask, o_plans64, o_E0, st);
    if (rc != HOM_OK) return rc;
  }

  if (want_fields) {
    NvtxRange r_("hom_solve: output fields");
    tm.begin(HOM_K_OUTPUT);
    if (lay.fast && DIM == 3) launched_ok(fast3d_row(A, nR, smem_fout, true, lay.run_max, st));
    else if (lay.fast) launched_ok(fast2d_out(A, nR, smem_fout, lay.run_max, st));
    else if (em) k_row<T, DIM, true, MAXR, true><<<nR, kThreads, lay.smem_row, st>>>(A);
    else k_row<T, DIM, true, MAXR><<<nR, kThreads, lay.smem_row, st>>>(A);
    tm.end();
    HOM_CUDA_TRY(cudaGetLastError());
    if (pass_rc != HOM_OK) return pass_rc;
    if (out->eps && !eps_dev)
      HOM_CUDA_TRY(cudaMemcpyAsync(out->eps, ws + o_stage_e, lay.fld_elems * sizeof(T), cudaMemcpyDeviceToHost, st));
    if (out->sigma && !sig_dev)
      HOM_CUDA_TRY(cudaMemcpyAsync(out->sigma, ws + o_stage_s, lay.fld_elems * sizeof(T), cudaMemcpyDeviceToHost, st));
  }
  std::vector<int> h_it(npairs), h_st(npairs);
  std::vector<double> h_e(npairs), h_en(npairs);
  unsigned long long h_bytes[HOM_NKERNEL];
  HOM_CUDA_TRY(cudaMemcpyAsync(out->mean_sigma, A.mean_sigma, (size_t)npairs * nc * sizeof(double), cudaMemcpyDefault, st));
  HOM_CUDA_TRY(cudaMemcpyAsync(h_it.data(), A.iters, npairs * sizeof(int), cudaMemcpyDeviceToHost, st));
  HOM_CUDA_TRY(cudaMemcpyAsync(h_st.data(), A.status, npairs * sizeof(int), cudaMemcpyDeviceToHost, st));
  HOM_CUDA_TRY(cudaMemcpyAsync(h_e.data(), A.err, npairs * sizeof(double), cudaMemcpyDeviceToHost, st));
  HOM_CUDA_TRY(cudaMemcpyAsync(h_en.data(), A.errn, npairs * sizeof(double), cudaMemcpyDeviceToHost, st));
  HOM_CUDA_TRY(cudaMemcpyAsync(h_bytes, A.bytes, sizeof(h_bytes), cudaMemcpyDeviceToHost, st));
  HOM_CUDA_TRY(cudaStreamSynchronize(st));
  tm.collect();
  if (out->iterations) std::memcpy(out->iterations, h_it.data(), npairs * sizeof(int));
  if (out->status) std::memcpy(out->status, h_st.data(), npairs * sizeof(int));
  if (out->err) std::memcpy(out->err, h_e.data(), npairs * sizeof(double));
  if (out->err_n) std::memcpy(out->err_n, h_en.data(), npairs * sizeof(double));
  if (out->err_c) {
    if (em) HOM_CUDA_TRY(cudaMemcpy(out->err_c, A.errc, npairs * sizeof(double), cudaMemcpyDeviceToHost));
    else std::memset(out->err_c, 0, npairs * sizeof(double));
  }
  if (out->history && !hist_dev)
    HOM_CUDA_TRY(cudaMemcpy(out->history, A.hist, hist_elems * sizeof(double), cudaMemcpyDeviceToHost));
  if (out->stats) {
    for (int k = 0; k < HOM_NKERNEL; ++k) out->stats->bytes[k] += (double)h_bytes[k];
    double vi = 0.0;
    for (int p = 0; p < npairs; ++p) vi += (double)lay.cells[lay.pairs[p].cell].nv * h_it[p];
    out->stats->voxel_iterations += vi;
  }
  {
    // the error word: a bounded wait that ran out (every build), a failed bounds check (debug builds)
    unsigned int w[4];
    HOM_CUDA_TRY(cudaMemcpy(w, A.dbg, sizeof(w), cudaMemcpyDeviceToHost));
    if (w[0] == 0xFFFFFFFFu) return set_error(HOM_ERR_TIMEOUT, "a shared-memory bulk copy did not complete in time");
    if (w[0])
      return set_error(HOM_ERR_BOUNDS, "bounds check failed in a solver kernel: file %u, line %u, index %llu", w[1],
                       w[0], ((unsigned long long)w[2] << 32) | w[3]);
  }
  int worst = HOM_OK;
  for (int p = 0; p < npairs; ++p) {
    if (h_st[p] == HOM_STATUS_DIVERGED) worst = HOM_ERR_DIVERGED;
    else if ((h_st[p] == HOM_STATUS_MAX_ITER || h_st[p] == HOM_STATUS_STALLED) && worst == HOM_OK)
      worst = HOM_ERR_NOT_CONVERGED;
  }
  if (worst == HOM_ERR_DIVERGED) set_error(worst, "a load case diverged");
  if (worst == HOM_ERR_NOT_CONVERGED) set_error(worst, "a load case reached max_iter or stalled");
  return worst;
}

}  // namespace

std::string tune_report() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  std::string r;
  for (const auto& e : g_tuned) {
    char c[96];
    std::snprintf(c, sizeof(c), " -> %s r%d", e.choice.passes == HOM_PASSES_AUTO ? "specialised" : "generic",
                  e.choice.radix);
    r += e.key + ": " + e.report + c + "\n";
  }
  return r;
}

void release_graphs() {
  std::lock_guard<std::mutex> lk(g_graph_mu);
  for (auto& e : g_graphs) cudaGraphExecDestroy(e.exec);
  g_graphs.clear();
}

}  // namespace hom

using namespace hom;

namespace hom {

int solve_entry(const hom_cell* cells, int ncells, const hom_material* mat, const double* E, int L,
                const double* c0, const hom_solve_opts* opts, hom_result* out, void* stream,
                const ExternalWorkspace* ext, const AdjointSpec* adj, bool cg) {
  if (!cells || ncells <= 0 || !mat || !E || !c0 || !opts || !out || !out->mean_sigma)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: null or empty argument");
  if (L < 1 || L > kMaxLoads) return set_error(HOM_ERR_INVALID_ARG, "hom_solve: L must be in [1, %d]", kMaxLoads);
  if (opts->precision != HOM_FP32 && opts->precision != HOM_FP64)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: unknown precision");
  if (opts->criterion != HOM_CRIT_E && opts->criterion != HOM_CRIT_EN)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: unknown criterion");
  if (opts->max_iter < 0 || opts->check_every < 0 || opts->diverge_window < 0 || opts->stall_window < 0)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: negative option");
  if (opts->passes != HOM_PASSES_AUTO && opts->passes != HOM_PASSES_GENERIC)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: unknown passes option %d", opts->passes);
  if (opts->max_radix != 0 && opts->max_radix != 15 && opts->max_radix != 27 && opts->max_radix != 45)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: max_radix must be 0, 15, 27 or 45");
  if (opts->green != HOM_GREEN_CONTINUOUS && opts->green != HOM_GREEN_ROTATED)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: unknown Green operator %d", opts->green);
  if (cg && opts->green != HOM_GREEN_CONTINUOUS)
    return set_error(HOM_ERR_NOT_IMPL, "hom_solve_cg: only the continuous Green operator");
  if (opts->refine < 0 || opts->refine_inner < 0) return set_error(HOM_ERR_INVALID_ARG, "hom_solve: negative refine option");
  if (opts->refine > 0 && (opts->precision != HOM_FP32 || cg || adj || ext))
    return set_error(HOM_ERR_NOT_IMPL, "hom_solve: defect correction is for FP32 forward solves of hom_solve");
  if (opts->scheme != HOM_SCHEME_BASIC && opts->scheme != HOM_SCHEME_EYRE_MILTON)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: unknown scheme %d", opts->scheme);
  if (opts->warm_start) {
    if (cg || adj || ext || opts->refine > 0 || opts->scheme != HOM_SCHEME_BASIC)
      return set_error(HOM_ERR_NOT_IMPL, "hom_solve: a warm start is for the basic scheme of hom_solve without "
                                         "defect correction");
    if (!is_device_ptr(out->eps))
      return set_error(HOM_ERR_INVALID_ARG, "hom_solve: a warm start reads the initial field from device memory "
                                            "at out->eps");
  }
  if (opts->scheme == HOM_SCHEME_EYRE_MILTON &&
      (cg || adj || ext || opts->refine > 0 || opts->green != HOM_GREEN_CONTINUOUS))
    return set_error(HOM_ERR_NOT_IMPL,
                     "hom_solve: the Eyre-Milton scheme is for forward solves of hom_solve with the continuous "
                     "Green operator and no defect correction");
  if (!mat->label || !mat->phase_c32 || !mat->phase_c64)
    return set_error(HOM_ERR_INVALID_ARG, "hom_solve: material not built");
  const int dim = cells[0].dim;
  for (int c = 0; c < ncells; ++c) {
    if (cells[c].dim != dim || (dim != 2 && dim != 3))
      return set_error(HOM_ERR_INVALID_ARG, "hom_solve: every cell must share dim 2 or 3");
    if (!grid_supported(cells[c].n))
      return set_error(HOM_ERR_UNSUPPORTED_SIZE, "hom_solve: cell %d grid %d unsupported", c, cells[c].n);
    if (!(c0[2 * c + 1] > 0.0) || !(c0[2 * c] + 2.0 * c0[2 * c + 1] > 0.0))
      return set_error(HOM_ERR_INVALID_ARG, "hom_solve: reference medium of cell %d is not positive", c);
  }
  if (mat->dim != dim) return set_error(HOM_ERR_INVALID_ARG, "hom_solve: material built for another dimension");
  cudaGetLastError();  // do not report an error left behind by an unrelated earlier call
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // Largest register radix of the generic FFT stages: FP32 kernels are compiled for 15, 27 and 45
  // (opts->max_radix; 0 = 27), FP64 ones for 15.
  auto dispatch = [&](const hom_solve_opts* op, hom_result* res) -> int {
    const int r32 = op->max_radix > 0 ? op->max_radix : 27;
    if (op->precision == HOM_FP32) {
      if (r32 >= 45)
        return dim == 2 ? run_solve<float, 2, 45>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg)
                        : run_solve<float, 3, 45>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg);
      if (r32 <= 15)
        return dim == 2 ? run_solve<float, 2, 15>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg)
                        : run_solve<float, 3, 15>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg);
      return dim == 2 ? run_solve<float, 2, 27>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg)
                      : run_solve<float, 3, 27>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg);
    }
    return dim == 2 ? run_solve<double, 2, 15>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg)
                    : run_solve<double, 3, 15>(cells, ncells, mat, E, L, c0, op, res, st, ext, adj, cg);
  };
  hom_solve_opts o = *opts;
  if (opts->tune && opts->precision == HOM_FP32 && !ext && !adj && !cg && opts->passes == HOM_PASSES_AUTO &&
      opts->max_radix == 0) {
    // Autotuner: the first solve of a batch shape times every candidate plan -- the specialised
    // passes (where every size has one) and the generic passes with register radices up to 15, 27
    // and 45 -- over a few fixed iterations of this very batch, and keeps the fastest for the shape.
    int dev = 0;
    HOM_CUDA_TRY(cudaGetDevice(&dev));
    std::vector<int> ns;
    for (int c = 0; c < ncells; ++c) ns.push_back(cells[c].n);
    std::sort(ns.begin(), ns.end());
    // defect correction and warm starts run on the generic passes: a choice of their own, over their radices
    const bool generic = opts->refine > 0 || opts->warm_start != 0;
    std::string key = "dev" + std::to_string(dev) + " dim" + std::to_string(dim) + " L" + std::to_string(L) +
                      " green" + std::to_string(opts->green) + " scheme" + std::to_string(opts->scheme) +
                      (generic ? " generic n" : " n");
    for (size_t i = 0; i < ns.size(); ++i) {
      size_t j = i;
      while (j + 1 < ns.size() && ns[j + 1] == ns[i]) ++j;
      key += " " + std::to_string(ns[i]) + "x" + std::to_string(j - i + 1);
      i = j;
    }
    TuneChoice choice{};
    if (!find_tuned(key, &choice)) {
      struct Cand { int passes, radix; };
      Cand cands[] = {{HOM_PASSES_AUTO, 27}, {HOM_PASSES_GENERIC, 15}, {HOM_PASSES_GENERIC, 27},
                      {HOM_PASSES_GENERIC, 45}};
      if (generic) cands[0].passes = HOM_PASSES_GENERIC;
      std::vector<double> ms_sigma((size_t)ncells * L * nc_of(dim));
      std::string report;
      double best = 1e300;
      // The time per iteration of a candidate is that of the call as it would run (whatever mix of passes
      // and on-chip solver it takes), from the difference of two fixed budgets: set-up drops out.  A caller
      // waits for the trials, so they are few: 1, 1 and 8 iterations a candidate.
      cudaEvent_t ev[2] = {};
      HOM_CUDA_TRY(cudaEventCreate(&ev[0]));
      if (cudaEventCreate(&ev[1]) != cudaSuccess) {
        cudaEventDestroy(ev[0]);
        return set_error(HOM_ERR_CUDA, "autotuner: event creation failed");
      }
      int tune_rc = HOM_OK, trial_iters = 0;
      auto timed = [&](const Cand& cd, int iters) {
        hom_solve_opts t = *opts;
        t.passes = cd.passes;
        t.max_radix = cd.radix;
        // a trial has no field to start from, and its iterations are those of the plain scheme
        t.warm_start = 0;
        t.refine = 0;
        t.tol = -1.0;  // a fixed number of iterations, no early stop
        t.max_iter = iters - 1;  // max_iter Green-operator applications make one iterate more
        trial_iters += iters;
        t.use_graph = 0;
        t.tune = 0;
        hom_result tr{};
        tr.mean_sigma = ms_sigma.data();
        cudaEventRecord(ev[0], st);
        const int rc = dispatch(&t, &tr);
        cudaEventRecord(ev[1], st);
        if (rc != HOM_OK && rc != HOM_ERR_NOT_CONVERGED && rc != HOM_ERR_DIVERGED) tune_rc = rc;
        float ms = 0.f;
        cudaEventSynchronize(ev[1]);
        cudaEventElapsedTime(&ms, ev[0], ev[1]);
        return (double)ms;
      };
      for (const Cand& cd : cands) {
        timed(cd, 1);  // the first call builds plans and workspace
        const double few = timed(cd, 1), more = timed(cd, 8);
        if (tune_rc != HOM_OK) break;
        const double ms = std::max(0.0, more - few) / 7.0;
        char line[160];
        std::snprintf(line, sizeof(line), "%s%s r%d %.3f ms", report.empty() ? "" : " | ",
                      cd.passes == HOM_PASSES_AUTO ? "specialised" : "generic", cd.radix, ms);
        report += line;
        if (ms < best) {
          best = ms;
          choice = TuneChoice{cd.passes, cd.radix};
        }
      }
      cudaEventDestroy(ev[0]);
      cudaEventDestroy(ev[1]);
      if (tune_rc != HOM_OK) return tune_rc;
      keep_tuned(key, choice, report + " (" + std::to_string(trial_iters) + " trial iterations)");
    }
    o.passes = choice.passes;
    o.max_radix = choice.radix;
  }
  return dispatch(&o, out);
}

}  // namespace hom

extern "C" int hom_solve(const hom_cell* cells, int32_t ncells, const hom_material* mat, const double* E, int32_t L,
                         const double* c0, const hom_solve_opts* opts, hom_result* out, void* stream) {
  NvtxRange nvtx_range_("hom_solve");
  return solve_entry(cells, ncells, mat, E, L, c0, opts, out, stream, nullptr);
}

extern "C" int32_t hom_autotune_report(char* buf, int32_t len) {
  const std::string r = hom::tune_report();
  if (buf && len > 0) {
    const size_t k = std::min<size_t>(r.size(), (size_t)len - 1);
    std::memcpy(buf, r.data(), k);
    buf[k] = 0;
  }
  return (int32_t)r.size();
}

extern "C" int hom_solve_cg(const hom_cell* cells, int32_t ncells, const hom_material* mat, const double* E,
                            int32_t L, const hom_solve_opts* opts, hom_result* out, void* stream) {
  NvtxRange nvtx_range_("hom_solve_cg");
  if (!cells || ncells <= 0) return set_error(HOM_ERR_INVALID_ARG, "hom_solve_cg: null or empty argument");
  std::vector<double> c0(2 * (size_t)ncells, 0.5);  // validated only; the solve uses c0 = identity
  return solve_entry(cells, ncells, mat, E, L, c0.data(), opts, out, stream, nullptr, nullptr, true);
}
