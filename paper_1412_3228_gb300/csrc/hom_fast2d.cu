// Specialised FP32 row and Green passes of the 2D fixed-point and Eyre-Milton schemes (section 2, eqs. 1-a,
// 1-b, 2), with the radices of a few grid sizes fixed at compile time and those of every other read from a plan.
//
// Lane pairs.  Shared memory holds one float4 per (position, pair): (re_A, re_B, im_A, im_B), the
// same position of two complex lines A and B.  Every butterfly, the Green operator and the
// constitutive update then act on both lines with packed FP32x2 instructions (add/sub/mul/fma
// .f32x2), one instruction per pair of values.
//   row pass  : pair c = Mandel component c; line A = real rows y0 + i*(y0+1), line B = rows
//               y0+2 + i*(y0+3).  One CTA handles 4 rows and loops over the active loads.
//   Green pass: pair c = component c; line A = column kx0, line B = column kx0 + 1.
// With the three components side by side, the element stride is 48 bytes, so consecutive
// positions fall on distinct bank quads: the stage accesses are free of bank conflicts.
//
// Transforms are the in-place mixed-radix DIF (natural -> digit-reversed) and DIT (digit-reversed
// -> natural) of hom_common.cuh with the radices as template parameters: every index division is
// by a compile-time constant (plan-read transforms: by multiplication, FastDiv).  The row pass works on x samples at digit-reversed positions and
// reads one-byte labels permuted the same way (label8); the Green pass reads the wave number of each
// position from a table.
//
// State in HBM.  The specialised passes keep the mixed-domain state (eps buffers, tau) tiled by kx
// pairs (tile_index): one Green task reads one contiguous tile with 16-byte asynchronous copies
// straight into its shared-memory layout, and a row task reads 192 contiguous bytes per pair.  The
// Green pass keeps its displacement-like state g as [load][column pair][position][4 complex].
// Both layouts are private to these passes: the initial state and the output fields are written
// by the kernels here.
#define HOM_FILE_ID 2
#include <algorithm>
#include <cstring>
#include <functional>
#include <mutex>
#include <vector>

#include "hom_fast2d.h"
#include "hom_plan.h"
#include "hom_solve_args.cuh"
#include "hom_fastfft.cuh"
#include "hom_em.cuh"
#include "hom_point2d.cuh"

namespace hom {
namespace {

#ifndef HOM_ROW_PREFETCH
#define HOM_ROW_PREFETCH 0  // row pass L2 prefetch: 1 = the next load, 2 = the next task (bit mask)
#endif
#ifndef HOM_GREEN_GPF
#define HOM_GREEN_GPF 1  // Green pass: L2 prefetch of the task's own g (or u_hat) block before its forward FFT
#endif
#ifndef HOM_GREEN_PREFETCH
#define HOM_GREEN_PREFETCH 0  // Green pass: L2 prefetch of the task that starts next
#endif
constexpr int kFastSizes[] = {45, 75, 135, 225, 405, 1215};  // sizes with specialised 2D passes

constexpr int kRowSpare = 2 * NP * kFastRows;  // float4 entries of the row pass's spare landing area
// ------------------------------------------------------------------ row pass
// eps (stored x half-spectra) -> inverse x-DFT -> tau = sigma - c0 : eps -> forward x-DFT -> tau.
// OUT: the final fields eps and sigma of the returned iterate (real, solver output layout).
struct RowShared {
  int al[kMaxLoads], nal;                    // active loads
  float dc[kMaxLoads][2][kFastRows][NP];     // [load][eps row mean, tau row sum][row][comp]
};

// EM (Eyre-Milton scheme): the stored state is u = sigma + c0 : eps.  A pure voxel's tau is then
// W u with the isotropic W = (c - c0)(c + c0)^-1 (a per-phase pair of constants in place of
// (lam - lam0, 2 mu - 2 mu0)); a mixed group first solves eps = (c~ + c0)^-1 u per voxel and takes
// tau = c~ : eps - c0 : eps; the output pass turns u into eps first; the row sums of sigma are
// (tau + u) / 2.
template <bool OUT, bool SRC, bool EM, class PL>
__device__ __forceinline__ void row_body(const PL& pl, const SolveArgs& A, int task, const TaskR& t, const CellDev& c,
                                         const FastPlanDev& fp, float4* s, RowShared& sh) {
  const int N = pl.n;
  const int H = N / 2 + 1;
  const int P = (H + 1) / 2;  // kx pairs holding data
  int* s_al = sh.al;
  int& s_nal = sh.nal;
  auto& s_dc = sh.dc;
  const int it = *A.it_dev;
  if (threadIdx.x == 0) {
    int nal = 0;
    for (int l = 0; l < A.L; ++l) {
      const int cl = t.cell * A.L + l;
      if ((t.load < 0 || l == t.load) && (OUT || A.active[cl])) s_al[nal++] = l;
    }
    s_nal = nal;
  }
  __syncthreads();
  const int nal = s_nal;
  if (nal == 0) return;
  const int y0 = t.row0, nr = t.nrows;
  CellConst<float> cc;
  cell_const(c, cc);
  // OUT: sigma = c~ : eps, i.e. the update with a zero reference medium
  float4* taub = static_cast<float4*>(A.tau);
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  // one-byte labels of the task's rows (transform order) and the twiddle table -> shared memory,
  // behind the first loads
  const int NL = (N + 15) / 16 * 16;  // label row stride (bytes)
  uint8_t* slab = reinterpret_cast<uint8_t*>(s + pl.tile);
  {
    const uint4* src = reinterpret_cast<const uint4*>(A.label8 + c.lp_off + (size_t)y0 * NL);
    for (int i = threadIdx.x; i < nr * NL / 16; i += kT) cp16(slab + 16 * i, src + i);
  }
  float2* tws = reinterpret_cast<float2*>(s + pl.tile + kFastRows * NL / 16);
  for (int i = threadIdx.x; i < (N + 1) / 2; i += kT) cp16(tws + 2 * i, fp.tw2 + 2 * i);
  float4* spare = s + pl.tile + kFastRows * NL / 16 + (N + 1) / 2;
  float2* sph = reinterpret_cast<float2*>(spare + kRowSpare);
  float2* sinv = sph + c.nph;  // EM: per local phase, (c + c0)^-1 as the pair (coefficient of tr(u) I, of u)
  cp_commit();
  phase_constants<OUT, EM>(A, c, cc, sph, sinv, kT);  // visible after the next barrier
  uint16_t* xpos = reinterpret_cast<uint16_t*>(sinv + c.nph);  // OUT: position of x
  if (OUT)
    for (int i = threadIdx.x; i < N; i += kT) xpos[__ldg(fp.iperm + i)] = (uint16_t)i;

  for (int la = 0; la < nal; ++la) {
    const int l = s_al[la];
    const float4* ein = static_cast<const float4*>(A.eps[OUT ? (A.iters[t.cell * A.L + l] & 1) : (it & 1)]);
    // 1. four half-spectrum rows -> two Hermitian-extended complex lines per component.  Item
    // (p, k) = kx pair p, component k: its four row values (one 16-byte lane pair each) land, by
    // asynchronous copies all in flight at once, in the tile slots of the four line positions
    // they produce (row_slot), and are turned into line values in place below.  Rows beyond the
    // task (r >= nr) are zero-filled by the copy itself.
    for (int f = threadIdx.x; f < P * NP; f += kT) {
      const int p = f / NP, k = f - p * NP;
      const float4* src = ein + tile_index(c, N, l, p, y0) + k;
#pragma unroll
      for (int r = 0; r < kFastRows; ++r)
        cp16z(row_slot_p<NP>(pl, s, spare, p, k, r), src + (size_t)(r < nr ? r : 0) * NP, r < nr ? 16u : 0u);
    }
    cp_commit();
    // the next active load's rows of every pair (192 contiguous bytes each) -> L2, so that its
    // copies above hit L2 while this load's transforms run
    if ((HOM_ROW_PREFETCH & 1) && la + 1 < nal) {
      const float4* nx = static_cast<const float4*>(A.eps[OUT ? (A.iters[t.cell * A.L + s_al[la + 1]] & 1) : (it & 1)]);
      for (int p = threadIdx.x; p < P; p += kT)
        prefetch_l2(nx + tile_index(c, N, s_al[la + 1], p, y0), (unsigned)(nr * NP * sizeof(float4)));
    }
    cp_wait_all();
    __syncthreads();
    for (int f = threadIdx.x; f < P * NP; f += kT) {
      const int p = f / NP, k = f - p * NP;
      float4 v[kFastRows];
#pragma unroll
      for (int r = 0; r < kFastRows; ++r) v[r] = *row_slot_p<NP>(pl, s, spare, p, k, r);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int kx = 2 * p + h;
        if (kx >= H) break;
        // row r at kx: (re, im) = lane h of v[r]
        const float2 q0 = h ? make_float2(v[0].y, v[0].w) : make_float2(v[0].x, v[0].z);
        const float2 q1 = h ? make_float2(v[1].y, v[1].w) : make_float2(v[1].x, v[1].z);
        const float2 q2 = h ? make_float2(v[2].y, v[2].w) : make_float2(v[2].x, v[2].z);
        const float2 q3 = h ? make_float2(v[3].y, v[3].w) : make_float2(v[3].x, v[3].z);
        // A + iB at kx and conj(A) + i conj(B) at n - kx, for (A, B) = (row 0, row 1) and (row 2, row 3)
        s[pl.at(kx) + k] = make_float4(q0.x - q1.y, q2.x - q3.y, q0.y + q1.x, q2.y + q3.x);
        if (kx > 0) {
          if (2 * kx != N)  // the Nyquist column of an even grid is its own partner (real rows: q.y = 0)
            s[pl.at(N - kx) + k] = make_float4(q0.x + q1.y, q2.x + q3.y, q1.x - q0.y, q3.x - q2.y);
        } else {
          s_dc[la][0][0][k] = q0.x;
          s_dc[la][0][1][k] = q1.x;
          s_dc[la][0][2][k] = q2.x;
          s_dc[la][0][3][k] = q3.x;
        }
      }
    }
    __syncthreads();
    fft_dif<NP, false, kT>(pl, s, tws);  // inverse: eps at digit-reversed positions

    // 2. constitutive update: lanes (x, y, z, w) of a float4 are rows (0, 2, 1, 3).  A one-byte
    // label is the local phase index of a pure voxel, or kLabel8Mixed (full label read from the
    // material, which also covers any voxel whose phase is not in the cell's list).
    auto labels = [&](int pos, uint32_t (&lab)[kFastRows]) {
#pragma unroll
      for (int r = 0; r < kFastRows; ++r) lab[r] = r < nr ? (uint32_t)slab[r * NL + pos] : 0u;
    };
    if constexpr (OUT) {
      // strains first (EM: from the states u), then stresses, each in place in the tile and out from there
      float* field[2] = {static_cast<float*>(A.out_eps), static_cast<float*>(A.out_sig)};
      const size_t base = c.fld_off + (size_t)l * NP * c.nv + (size_t)y0 * N;
      for (int ph = 0; ph < 2; ++ph) {
        if (ph == 1 || EM) {
          for (int pos = threadIdx.x; pos < N; pos += kT) {
            const int at = pl.at(pos);
            uint32_t lab[kFastRows];
            labels(pos, lab);
            float4 e[NP], o[NP];
#pragma unroll
            for (int k = 0; k < NP; ++k) e[k] = s[at + k];
            if (ph == 0) tau_point<true, false, true>(A, c, fp, sph, sinv, cc, nr, y0, l, pos, lab, e, o);
            else tau_point<true, false, false>(A, c, fp, sph, sinv, cc, nr, y0, l, pos, lab, e, o);
#pragma unroll
            for (int k = 0; k < NP; ++k) s[at + k] = ph == 0 ? e[k] : o[k];
          }
          __syncthreads();
        }
        if (field[ph]) store_rows<NP, kT>(pl, s, xpos, field[ph] + base, c.nv, nr);
        __syncthreads();  // the tile is rewritten by the next phase or the next load's fill
      }
      continue;
    }
    for (int pos = threadIdx.x; pos < N; pos += kT) {
      const int at = pl.at(pos);
      uint32_t lab[kFastRows];
      labels(pos, lab);
      float4 e[NP], o[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) e[k] = s[at + k];
      tau_point<OUT, SRC, EM>(A, c, fp, sph, sinv, cc, nr, y0, l, pos, lab, e, o);
#pragma unroll
      for (int k = 0; k < NP; ++k) s[at + k] = o[k];
    }
    __syncthreads();
    fft_dit<NP, true, kT>(pl, s, tws);  // forward: natural order

    // 3. split the two real rows of each line; store the half spectra of tau, pair by pair
    for (int f = threadIdx.x; f < P * NP; f += kT) {
      const int p = f / NP, k = f - p * NP;
      float4 w[kFastRows];  // rows 0..3 at (kx = 2p, 2p + 1): (re, re, im, im)
#pragma unroll
      for (int r = 0; r < kFastRows; ++r) w[r] = z4;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int kx = 2 * p + h;
        if (kx >= H) break;
        const float4 Z = s[pl.at(kx) + k];
        const float4 Zm = s[pl.at(kx == 0 ? 0 : N - kx) + k];
        // (Z[k] + conj Z[n-k]) / 2 -> first row of a line, (Z[k] - conj Z[n-k]) / 2i -> second row
        const float2 o0 = make_float2(0.5f * (Z.x + Zm.x), 0.5f * (Z.z - Zm.z));
        const float2 o1 = make_float2(0.5f * (Z.z + Zm.z), 0.5f * (Zm.x - Z.x));
        const float2 o2 = make_float2(0.5f * (Z.y + Zm.y), 0.5f * (Z.w - Zm.w));
        const float2 o3 = make_float2(0.5f * (Z.w + Zm.w), 0.5f * (Zm.y - Z.y));
        if (h == 0) {
          w[0].x = o0.x; w[0].z = o0.y; w[1].x = o1.x; w[1].z = o1.y;
          w[2].x = o2.x; w[2].z = o2.y; w[3].x = o3.x; w[3].z = o3.y;
          if (kx == 0) {
            s_dc[la][1][0][k] = o0.x;
            s_dc[la][1][1][k] = o1.x;
            s_dc[la][1][2][k] = o2.x;
            s_dc[la][1][3][k] = o3.x;
          }
        } else {
          w[0].y = o0.x; w[0].w = o0.y; w[1].y = o1.x; w[1].w = o1.y;
          w[2].y = o2.x; w[2].w = o2.y; w[3].y = o3.x; w[3].w = o3.y;
        }
      }
      const size_t b = tile_index(c, N, l, p, y0) + k;
#pragma unroll
      for (int r = 0; r < kFastRows; ++r)
        if (r < nr) taub[b + (size_t)r * NP] = w[r];
    }
    __syncthreads();
  }
  if (OUT) {
    if (threadIdx.x == 0)
      atomicAdd(A.bytes + HOM_K_OUTPUT,
                (unsigned long long)((size_t)nal * nr * NP * (H * sizeof(float2) + 2 * (size_t)N * sizeof(float)) +
                                     (size_t)nr * N * 4));
    return;
  }
  // sum of sigma over the task's rows per load and component (see the generic row pass):
  //   sum_x sigma = sum_x tau + c0 : (n * row mean of eps), rows combined in FP64
  if (threadIdx.x < nal * NP) {
    const int la = threadIdx.x / NP, k = threadIdx.x - la * NP;
    double acc = 0.0;
    for (int r = 0; r < nr; ++r) {
      if (EM) {  // sigma = (tau + u) / 2
        acc += 0.5 * ((double)s_dc[la][1][r][k] + (double)N * (double)s_dc[la][0][r][k]);
        continue;
      }
      const double tr = (double)s_dc[la][0][r][0] + (double)s_dc[la][0][r][1];
      const double se = (double)N * (2.0 * c.mu0 * (double)s_dc[la][0][r][k] + (k < 2 ? c.lam0 * tr : 0.0));
      acc += (double)s_dc[la][1][r][k] + se;
    }
    A.partR[((size_t)task * A.L + s_al[la]) * NP + k] = acc;
  }
  if (threadIdx.x == 0)
    atomicAdd(A.bytes + HOM_K_ROW,
              (unsigned long long)(2 * (size_t)nr * nal * NP * H * sizeof(float2) + (size_t)nr * N));
}

// L2 prefetch of the first active load of row task `task` (every pair's rows, 16 * 3 * nrows
// contiguous bytes each), issued while the CTA still works on its current task.
template <bool OUT>
__device__ __forceinline__ void prefetch_row_task(const SolveArgs& A, int task) {
  const TaskR t = A.tR[task];
  const CellDev c = A.cells[t.cell];
  int l = -1;
  for (int q = 0; q < A.L && l < 0; ++q)
    if (OUT || A.active[t.cell * A.L + q]) l = q;
  if (l < 0) return;
  const float4* e = static_cast<const float4*>(A.eps[OUT ? (A.iters[t.cell * A.L + l] & 1) : (*A.it_dev & 1)]);
  const int P = (c.n / 2 + 2) / 2;
  for (int p = threadIdx.x; p < P; p += kT)
    prefetch_l2(e + tile_index(c, c.n, l, p, t.row0), (unsigned)(t.nrows * NP * sizeof(float4)));
}

// One CTA per task.  `ahead` is the number of CTAs resident on the device at once: task b + ahead
// is about the one that starts when this CTA ends, so CTA b prefetches its first load into L2.
// RUN: radices up to RUN read from the plan (any size; see k_row_r2d); 0: compiled ones.
template <bool OUT, bool SRC, bool EM, int RUN>
__device__ __forceinline__ void row_task(const SolveArgs& A, int ntasks, int ahead) {
  HOM_DBG_POISON();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RowShared sh;
  float4* s = reinterpret_cast<float4*>(smem_raw);
  const int task = blockIdx.x;
  if ((HOM_ROW_PREFETCH & 2) && task + ahead < ntasks) prefetch_row_task<OUT>(A, task + ahead);
  const TaskR t = A.tR[task];
  const CellDev c = A.cells[t.cell];
  // debug builds: the task's rows lie in the cell (the CTA skips a bad task as a whole)
  if (!HOM_CHECK(A, t.row0 >= 0 && t.nrows >= 1 && t.nrows <= kFastRows && t.row0 + t.nrows <= c.nrows &&
                        t.load < A.L, (size_t)task))
    return;
  const FastPlanDev& fp = A.fplans[c.fplan];
  if constexpr (RUN > 0) {
    __shared__ RunPlan sp;
    row_body<OUT, SRC, EM>(RunN<NP, RUN>(stage_plan(fp.run, sp, kT)), A, task, t, c, fp, s, sh);
  } else {
    switch (c.n) {
      case 45: row_body<OUT, SRC, EM>(FixedN<45, NP>(), A, task, t, c, fp, s, sh); break;
      case 75: row_body<OUT, SRC, EM>(FixedN<75, NP>(), A, task, t, c, fp, s, sh); break;
      case 135: row_body<OUT, SRC, EM>(FixedN<135, NP>(), A, task, t, c, fp, s, sh); break;
      case 225: row_body<OUT, SRC, EM>(FixedN<225, NP>(), A, task, t, c, fp, s, sh); break;
      case 405: row_body<OUT, SRC, EM>(FixedN<405, NP>(), A, task, t, c, fp, s, sh); break;
      case 1215: row_body<OUT, SRC, EM>(FixedN<1215, NP>(), A, task, t, c, fp, s, sh); break;
      default: break;
    }
  }
}
template <bool OUT, bool SRC, bool EM = false>
__global__ void __launch_bounds__(kT, 3) k_row_f2d(SolveArgs A, int ntasks, int ahead) {
  row_task<OUT, SRC, EM, 0>(A, ntasks, ahead);
}
// The same pass with radices read from a plan, for batches that hold a size without compiled ones.  Radices
// up to 16 (lane pairs) take 128 registers, two CTAs per SM; batches whose plans stay at 9 and below run the
// 80-register variant, three CTAs per SM.  Measured against the generic row pass, which keeps two real rows
// per complex line and scalar arithmetic: 2 cells of 512^2, 3 loads: 72 us generic, 55 us with 128
// registers, 39 us with 80; 143^2: 43 us generic, 16 us (one load per task).
template <bool OUT, bool SRC, bool EM, int MAXR>
__global__ void __launch_bounds__(kT, MAXR > 9 ? 2 : 3) k_row_r2d(SolveArgs A, int ntasks, int ahead) {
  row_task<OUT, SRC, EM, MAXR>(A, ntasks, ahead);
}

// eps = E: the stored x-spectrum holds E at kx = 0 of every row (lane A of pair 0), zero elsewhere.
// EM: u = 2 c0 : E instead, and its 1/N_v-scaled spectrum at k = 0 in the Green pass's private state
// (pair 0, position 0; the rest is cleared by the caller).
template <bool EM = false>
__global__ void k_init_f2d(SolveArgs A, int ncells) {
  for (int cell = blockIdx.y; cell < ncells; cell += gridDim.y) {
    const CellDev c = A.cells[cell];
    const long long items = (long long)A.L * c.n * NP;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < items; i += (long long)gridDim.x * blockDim.x) {
      const int k = (int)(i % NP);
      const long long r = i / NP;
      const int y = (int)(r % c.n);
      const int l = (int)(r / c.n);
      const double* El = A.E + ((size_t)cell * A.L + l) * NP;
      double v = El[k];
      if (EM) {
        v = 2.0 * (2.0 * c.mu0 * El[k] + (k < 2 ? c.lam0 * (El[0] + El[1]) : 0.0));
        if (y == 0) {  // u_hat(0): component k of lane A at position 0, (re, im) in float2 slot k
          float2* ub = reinterpret_cast<float2*>(static_cast<float4*>(A.g) + (c.g_off + (size_t)l * (c.Hp / 2) * c.n * 6) / 2);
          ub[k] = make_float2((float)v, 0.f);
        }
      }
      static_cast<float4*>(A.eps[0])[tile_index(c, c.n, l, 0, y) + k] = make_float4((float)v, 0.f, 0.f, 0.f);
    }
  }
}

// ------------------------------------------------------------------ Green pass
// Eyre-Milton scheme: the positions of one thread, lane by lane; the private state is u_hat of the
// current iterate, [position][6 complex] = (kx0 components 0..2, kx0+1 components 0..2) as three
// float4, in place of g.  Returns the three compensated sums.
template <class PL>
__device__ __forceinline__ void green_em(const PL& pl, const SolveArgs& A, int kx0, bool hasB, const CellDev& c, const float* sx,
                                         const FastPlanDev& fp, float4* s, float4* ub, const double* Eld,
                                         Acc<float> (&acc)[3]) {
  const GreenPairEm gp(A, c, fp, kx0, Eld);
  float2* u2 = reinterpret_cast<float2*>(ub);  // [position][lane A comps 0..2, lane B comps 0..2]
  // one (position, lane) per item: lane h reads and writes its own floats of the lane pairs
  for (int i = threadIdx.x; i < 2 * pl.n; i += kT) {
    const int pos = i >> 1, h = i & 1;
    if (h && !hasB) continue;
    gp.point(reinterpret_cast<float*>(s + pl.at(pos)), h, sx[pos], pos == 0, u2 + 6 * pos + 3 * h, u2 + 6 * pos + 3 * h, acc);
  }
  if (!hasB) {  // the missing lane B of the last pair stays zero
    float* sf = reinterpret_cast<float*>(s);
    for (int i = threadIdx.x; i < pl.tile; i += kT) {
      sf[4 * i + 1] = 0.f;
      sf[4 * i + 3] = 0.f;
    }
  }
}

// Piece `i` of a tile that bulk copies move: the whole tile (contiguous in HBM and in shared memory), or,
// padded, the positions between two paddings.
template <class PL>
__device__ __forceinline__ int tile_pieces(const PL& pl) {
  if constexpr (PL::fixed) return 1;
  else return pl.p.pad ? pl.n / pl.p.r[0] : 1;
}
template <class PL>
__device__ __forceinline__ int piece_len(const PL& pl, int pieces) { return pl.n / pieces * NP; }

// The finished tile (natural order after the inverse transform) -> the next eps buffer.
template <class PL>
__device__ __forceinline__ void green_store(const PL& pl, const float4* s, float4* out) {
  fence_proxy_async();  // this thread's tile writes, visible to the bulk copy
  __syncthreads();
  const int pieces = tile_pieces(pl), len = piece_len(pl, pieces);
  for (int i = threadIdx.x; i < pieces; i += kT) bulk_store(out + i * len, s + i * (len + 1), (unsigned)(len * sizeof(float4)));
  if (threadIdx.x < pieces) bulk_store_wait_read();  // the CTA keeps its shared memory until the copies have read it
}

// Positions per thread of a fixed-size Green task.
template <class PL> __host__ __device__ constexpr int green_npos() {
  if constexpr (PL::fixed) return (PL::n + kT - 1) / kT;
  else return 1;
}

// tau (mixed domain) -> forward y-DFT -> Gamma0 and the residual on J (eq. 2) -> inverse y-DFT -> eps.
template <bool EM, class PL>
__device__ __forceinline__ void green_body(const PL& pl, const SolveArgs& A, int task, const TaskL& t, const CellDev& c,
                                           const FastPlanDev& fp, float4* s) {
  const int N = pl.n, H = N / 2 + 1;
  const int cl = t.cell * A.L + t.load;
  if (!A.active[cl]) return;
  const int it = *A.it_dev;
  const int Hp = c.Hp, kx0 = t.kx0;
  const bool hasB = kx0 + 1 < H;
  // this task's tile (pair kx0 / 2 of its load): n rows x 3 components, contiguous
  const size_t tb = tile_index(c, N, t.load, kx0 / 2, 0);
  const float4* in = static_cast<const float4*>(A.tau) + tb;
  float4* out = static_cast<float4*>(A.eps[(it + 1) & 1]) + tb;
  const float2 z2 = make_float2(0.f, 0.f);
  // g of this column pair, [position][4 complex] = (kx0 d0, kx0 d1, kx0+1 d0, kx0+1 d1)
  float4* gb = static_cast<float4*>(A.g) +
               (c.g_off + ((size_t)t.load * (Hp / 2) + (size_t)(kx0 / 2)) * N * 4) / 2;
  // tile, twiddles and the wave numbers of the positions -> shared memory
  float2* tws = reinterpret_cast<float2*>(s + pl.tile);  // scalar twiddles: 3 CTAs per SM fit
  float* sx = reinterpret_cast<float*>(s + pl.tile + (N + 1) / 2);
  for (int i = threadIdx.x; i < (N + 1) / 2; i += kT) cp16(tws + 2 * i, fp.tw2 + 2 * i);
  // the tile (N NP float4, contiguous in HBM) by bulk copies
  __shared__ __align__(8) unsigned long long tile_bar;
  const int pieces = tile_pieces(pl), len = piece_len(pl, pieces);
  fence_proxy_async();  // earlier generic writes to this shared memory are ordered before the copies'
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_init(&tile_bar, 1);
    mbar_expect(&tile_bar, (unsigned)(N * NP * sizeof(float4)));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < pieces; i += kT)
    bulk_load(s + i * (len + 1), in + i * len, (unsigned)(len * sizeof(float4)), &tile_bar);
  for (int i = threadIdx.x; i < (N + 3) / 4; i += kT) cp16(sx + 4 * i, fp.xipos + 4 * i);
  cp_commit();
  cp_wait_all();
  // bounded wait (a copy of 60 KB lands in microseconds); running out is recorded, never a hang
  if (!mbar_wait(&tile_bar, 0, 1 << 22) && A.dbg) atomicCAS(A.dbg, 0u, 0xFFFFFFFFu);
  __syncthreads();
  if (threadIdx.x == 0) mbar_inval(&tile_bar);
  __syncthreads();
#if HOM_GREEN_GPF
  // the private state of this column pair (contiguous: N positions x 2 or 3 float4) -> L2, so that
  // its reads after the transform hit L2
  if (threadIdx.x < 32) {
    const size_t per = EM ? 3 : 2;
    const char* gsrc = reinterpret_cast<const char*>(static_cast<const float4*>(A.g) +
                                                     (c.g_off + ((size_t)t.load * (Hp / 2) + (size_t)(kx0 / 2)) * N * 2 * per) / 2);
    const unsigned bytes = (unsigned)(N * per * sizeof(float4));
    constexpr unsigned kPiece = 4096;
    for (unsigned o = threadIdx.x * kPiece; o < bytes; o += 32 * kPiece) prefetch_l2(gsrc + o, min(kPiece, bytes - o));
  }
#endif
  fft_dif<NP, true, kT>(pl, s, tws);  // forward: bin ky at position perm(ky)

  if constexpr (EM) {
    float4* ub = static_cast<float4*>(A.g) + (c.g_off + ((size_t)t.load * (Hp / 2) + (size_t)(kx0 / 2)) * N * 6) / 2;
    Acc<float> acc[3];
    green_em(pl, A, kx0, hasB, c, sx, fp, s, ub, A.E + (size_t)cl * NP, acc);
    double tot[3];
    block_sum<float, 3, kT>(acc, tot);  // contains the barrier before the inverse transform
    if (threadIdx.x == 0) {
      A.partC[2 * (size_t)task] = tot[0];
      A.partC[2 * (size_t)task + 1] = tot[1];
      A.partE[task] = tot[2];
    }
    fft_dit<NP, false, kT>(pl, s, tws);  // inverse: natural order
    green_store(pl, s, out);
    if (threadIdx.x == 0) {
      const int ntk = hasB ? 2 : 1;
      atomicAdd(A.bytes + HOM_K_GREEN, (unsigned long long)(4 * (size_t)N * ntk * NP * sizeof(float2)));
    }
    return;
  }

  GreenPair gp(A, c, fp, kx0, cl);
  // g of every position of this thread, loaded at once where their number is known
  constexpr int NPOS = green_npos<PL>();
  float4 gr[NPOS][2];
  auto load_g = [&](int pos, float4(&r)[2]) {
    if (pos < N) {
      r[0] = gb[2 * pos];
      r[1] = gb[2 * pos + 1];
    }
  };
  if constexpr (PL::fixed) {
#pragma unroll
    for (int i = 0; i < NPOS; ++i) load_g(threadIdx.x + i * kT, gr[i]);
  }
  auto point = [&](int pos, const float4(&gin)[2]) {
    gp.point(s + pl.at(pos), sx[pos], pos == 0, gin, gb + 2 * pos);
  };
  if constexpr (PL::fixed) {
#pragma unroll
    for (int i = 0; i < NPOS; ++i) {
      const int pos = threadIdx.x + i * kT;
      if (pos < N) point(pos, gr[i]);
    }
  } else {
    float4 nx[2];  // g of the thread's next position, loaded while this one is processed
    load_g(threadIdx.x, nx);
    for (int pos = threadIdx.x; pos < N; pos += kT) {
      gr[0][0] = nx[0];
      gr[0][1] = nx[1];
      load_g(pos + kT, nx);
      point(pos, gr[0]);
    }
  }
  {
    Acc<float> vv[2];
    gp.sums(vv);
    double tot[2];
    block_sum<float, 2, kT>(vv, tot);  // contains the barrier before the inverse transform
    if (threadIdx.x == 0) {
      A.partC[2 * (size_t)task] = tot[0];
      A.partC[2 * (size_t)task + 1] = tot[1];
    }
  }
  fft_dit<NP, false, kT>(pl, s, tws);  // inverse: natural order
  green_store(pl, s, out);
  if (threadIdx.x == 0) {
    const int ntk = hasB ? 2 : 1;
    atomicAdd(A.bytes + HOM_K_GREEN,
              (unsigned long long)(2 * (size_t)N * ntk * NP * sizeof(float2) + 2 * (size_t)N * ntk * 2 * sizeof(float2)));
  }
}

// L2 prefetch of Green task `task`'s tau tile and g block (contiguous, in 4 KB pieces).
__device__ __forceinline__ void prefetch_green_task(const SolveArgs& A, int task) {
  const TaskL t = A.tC[task];
  if (!A.active[t.cell * A.L + t.load]) return;
  const CellDev c = A.cells[t.cell];
  const char* tau = reinterpret_cast<const char*>(static_cast<const float4*>(A.tau) + tile_index(c, c.n, t.load, t.kx0 / 2, 0));
  const char* g = reinterpret_cast<const char*>(static_cast<const float4*>(A.g) +
                                                (c.g_off + ((size_t)t.load * (c.Hp / 2) + (size_t)(t.kx0 / 2)) * c.n * 4) / 2);
  const unsigned bt = (unsigned)c.n * NP * sizeof(float4), bg = (unsigned)c.n * 2 * sizeof(float4);  // basic scheme's g
  constexpr unsigned kPiece = 4096;
  const unsigned nt = (bt + kPiece - 1) / kPiece, ng = (bg + kPiece - 1) / kPiece;
  for (unsigned i = threadIdx.x; i < nt + ng; i += kT) {
    const bool on_t = i < nt;
    const unsigned o = (on_t ? i : i - nt) * kPiece, b = on_t ? bt : bg;
    prefetch_l2((on_t ? tau : g) + o, min(kPiece, b - o));
  }
}

// One CTA per task; CTA b prefetches task b + ahead into L2 (see k_row_f2d).
template <bool EM, int RUN>
__device__ __forceinline__ void green_task(const SolveArgs& A, int ntasks, int ahead) {
  HOM_DBG_POISON();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* s = reinterpret_cast<float4*>(smem_raw);
  const int task = blockIdx.x;
  if (HOM_GREEN_PREFETCH && task + ahead < ntasks) prefetch_green_task(A, task + ahead);
  const TaskL t = A.tC[task];
  const CellDev c = A.cells[t.cell];
  // debug builds: an even kx pair start inside the half spectrum, a valid load
  if (!HOM_CHECK(A, t.kx0 >= 0 && (t.kx0 & 1) == 0 && t.kx0 < c.H && t.load >= 0 && t.load < A.L, (size_t)task))
    return;
  const FastPlanDev& fp = A.fplans[c.fplan];
  if constexpr (RUN > 0) {
    __shared__ RunPlan sp;
    green_body<EM>(RunN<NP, RUN>(stage_plan(fp.run, sp, kT)), A, task, t, c, fp, s);
  } else {
    switch (c.n) {
      case 45: green_body<EM>(FixedN<45, NP>(), A, task, t, c, fp, s); break;
      case 75: green_body<EM>(FixedN<75, NP>(), A, task, t, c, fp, s); break;
      case 135: green_body<EM>(FixedN<135, NP>(), A, task, t, c, fp, s); break;
      case 225: green_body<EM>(FixedN<225, NP>(), A, task, t, c, fp, s); break;
      case 405: green_body<EM>(FixedN<405, NP>(), A, task, t, c, fp, s); break;
      case 1215: green_body<EM>(FixedN<1215, NP>(), A, task, t, c, fp, s); break;
      default: break;
    }
  }
}
template <bool EM = false>
__global__ void __launch_bounds__(kT, 3) k_green_f2d(SolveArgs A, int ntasks, int ahead) {
  green_task<EM, 0>(A, ntasks, ahead);
}
// Radices read from a plan (see k_row_r2d): 2 cells of 512^2, 3 loads: 103 us generic, 45 us with 128
// registers, 33 us with 80; 143^2: 42 us generic, 14 us.
template <bool EM, int MAXR>
__global__ void __launch_bounds__(kT, MAXR > 9 ? 2 : 3) k_green_r2d(SolveArgs A, int ntasks, int ahead) {
  green_task<EM, MAXR>(A, ntasks, ahead);
}

// ------------------------------------------------------------------ labels in transform order
__global__ void k_permute_labels(SolveArgs A, int ncells) {
  const int ci = blockIdx.y;
  if (ci >= ncells) return;
  const CellDev c = A.cells[ci];
  if (c.fplan < 0) return;
  const FastPlanDev fp = A.fplans[c.fplan];
  const long long nv = c.nv;  // rows x n (rows are y in 2D, z n + y in 3D)
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
    const long long y = i / c.n;
    const int pos = (int)(i - y * c.n);
    const uint32_t lab = A.label[c.vox_off + y * c.n + fp.iperm[pos]];
    const int nl = (c.n + 15) / 16 * 16;
    // local index of a pure voxel's phase in the cell's list (not found: the full-label path)
    uint32_t loc = kLabel8Mixed;
    if (!(lab & HOM_MIXED_BIT))
      for (int j = 0; j < c.nph; ++j)
        if ((uint32_t)A.cell_phases[c.ph_off + j] == lab) {
          loc = (uint32_t)j;
          break;
        }
    const_cast<uint8_t*>(A.label8)[c.lp_off + y * nl + pos] = (uint8_t)loc;
  }
}

// ------------------------------------------------------------------ host side
struct FastCacheEntry {
  int dev, n;
  bool run;
  FastPlanDev p;
  void* mem;
};
std::mutex g_fast_mu;
std::vector<FastCacheEntry> g_fast_cache;

std::vector<int> radices_of(int n) {
  switch (n) {
    case 45: return {Radix<45>::r0, Radix<45>::r1};
    case 75: return {Radix<75>::r0, Radix<75>::r1};
    case 135: return {Radix<135>::r0, Radix<135>::r1};
    case 225: return {Radix<225>::r0, Radix<225>::r1};
    case 405: return {Radix<405>::r0, Radix<405>::r1, Radix<405>::r2};
    case 1215: return {Radix<1215>::r0, Radix<1215>::r1, Radix<1215>::r2};
    case 27: return {Radix<27>::r0, Radix<27>::r1};
    case 81: return {Radix<81>::r0, Radix<81>::r1};
    case 243: return {Radix<243>::r0, Radix<243>::r1, Radix<243>::r2};
    default: return {};
  }
}

}  // namespace

bool fast2d_size(int n) {
  for (int k : kFastSizes)
    if (k == n) return true;
  return false;
}

namespace {
// Radices (DIT order) of the run-time plans: the fewest stages of radices up to 16, then the smallest
// largest radix; even radices first (their stage is padded, and the spans that follow are then multiples
// of 8 or 16 where the size allows, which keeps neighbouring butterflies on distinct banks).
std::vector<int> run_radices(int n) {
  static const int kR[] = {16, 15, 13, 11, 9, 8, 7, 5, 4, 3, 2};
  std::vector<int> best, cur;
  std::function<void(int)> search = [&](int rem) {
    if (rem == 1) {
      auto key = [](const std::vector<int>& v) { return std::make_pair(v.size(), *std::max_element(v.begin(), v.end())); };
      if (best.empty() || key(cur) < key(best)) best = cur;
      return;
    }
    if ((int)cur.size() >= kMaxRunStages || (!best.empty() && cur.size() + 1 > best.size())) return;
    for (int r : kR) {
      if (rem % r != 0 || (!cur.empty() && r > cur.back())) continue;
      cur.push_back(r);
      search(rem / r);
      cur.pop_back();
    }
  };
  search(n);
  std::stable_sort(best.begin(), best.end(), [](int a, int b) { return (a & 1) < (b & 1); });
  return best;
}
void fill_run_plan(const HostPlan& hp, RunPlan& r) {
  r.n = hp.n;
  r.m = (int)hp.radix.size();
  r.pad = (hp.radix[0] & 1) ? 0 : 1;
  int off = 0;
  for (int st = 0; st < r.m; ++st) {
    r.r[st] = hp.radix[st];
    r.L[st] = hp.span[st];
    r.tw[st] = off;
    if (st > 0) off += r.L[st] * (r.r[st] - 1);
    r.d_nb[st] = make_fastdiv(r.n / r.r[st]);
    r.d_L[st] = make_fastdiv(r.L[st]);
  }
  r.d_r0 = make_fastdiv(r.r[0]);
}
}  // namespace

void run_plan_shape(int n, int* largest, int* stages) {
  struct Shape { int n, largest, stages; };
  static std::vector<Shape> known;  // every size asked for once
  std::lock_guard<std::mutex> lk(g_fast_mu);
  auto it = std::find_if(known.begin(), known.end(), [&](const Shape& s) { return s.n == n; });
  if (it == known.end()) {
    const std::vector<int> r = run_radices(n);
    known.push_back({n, r.empty() ? 0 : *std::max_element(r.begin(), r.end()), (int)r.size()});
    it = known.end() - 1;
  }
  *largest = it->largest;
  *stages = it->stages;
}

bool run2d_size(int n) {  // the row pass's tile, twiddles and labels of 4 rows on chip, a few phases
  return grid_supported(n) && fast2d_smem_row(n, 64) <= 200 * 1024;
}

int fast2d_plan_host(int n, bool run, std::vector<unsigned char>& h, FastPlanDev* out) {
  HostPlan hp;
  const std::vector<int> radix = run ? run_radices(n) : radices_of(n);
  if (radix.empty() || !build_host_plan_radices(n, radix, hp))
    return set_error(HOM_ERR_UNSUPPORTED_SIZE, "no specialised plan for n = %d", n);
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t b_ip = up((size_t)n * 2), b_xp = up((size_t)n * 4), b_xn = up((size_t)n * 4), b_tw = up((size_t)n * 8 + 8);
  h.assign(b_ip + b_xp + b_xn + b_tw, 0);
  // per-stage twiddle tables (stages with span L > 1): entry (q - 1) L + j = w^(j q n / (L R))
  float* tw = reinterpret_cast<float*>(h.data() + b_ip + b_xp + b_xn);
  {
    size_t e = 0;
    for (size_t st = 1; st < hp.radix.size(); ++st) {
      const int R = hp.radix[st], L = hp.span[st], TS = n / (L * R);
      for (int q = 1; q < R; ++q)
        for (int j = 0; j < L; ++j, ++e) {
          const int t = (j * q * TS) % n;
          tw[2 * e] = (float)hp.tw[2 * t];
          tw[2 * e + 1] = (float)hp.tw[2 * t + 1];
        }
    }
  }
  uint16_t* ip = reinterpret_cast<uint16_t*>(h.data());
  for (int k = 0; k < n; ++k) ip[hp.perm[k]] = (uint16_t)k;
  float* xp = reinterpret_cast<float*>(h.data() + b_ip);
  float* xn = reinterpret_cast<float*>(h.data() + b_ip + b_xp);
  for (int p = 0; p < n; ++p) xp[p] = (float)hp.xi[ip[p]];
  for (int k = 0; k < n; ++k) xn[k] = (float)hp.xi[k];
  // table pointers as byte offsets from the start of the tables (fast2d_plan_rebase adds the base)
  FastPlanDev p{};
  p.iperm = reinterpret_cast<const uint16_t*>(size_t(0));
  p.xipos = reinterpret_cast<const float*>(b_ip);
  p.xinat = reinterpret_cast<const float*>(b_ip + b_xp);
  p.tw2 = reinterpret_cast<const float2*>(b_ip + b_xp + b_xn);
  p.n = n;
  fill_run_plan(hp, p.run);
  *out = p;
  return HOM_OK;
}

void fast2d_plan_rebase(FastPlanDev& p, const unsigned char* base) {
  auto at = [&](const void* off) { return base + reinterpret_cast<size_t>(off); };
  p.iperm = reinterpret_cast<const uint16_t*>(at(p.iperm));
  p.xipos = reinterpret_cast<const float*>(at(p.xipos));
  p.xinat = reinterpret_cast<const float*>(at(p.xinat));
  p.tw2 = reinterpret_cast<const float2*>(at(p.tw2));
}

int fast2d_plan(int n, bool run, FastPlanDev* out) {
  int dev = 0;
  HOM_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_fast_mu);
  for (const auto& e : g_fast_cache)
    if (e.dev == dev && e.n == n && e.run == run) {
      *out = e.p;
      return HOM_OK;
    }
  std::vector<unsigned char> h;
  FastPlanDev p{};
  int rc = fast2d_plan_host(n, run, h, &p);
  if (rc != HOM_OK) return rc;
  void* mem = nullptr;
  HOM_CUDA_TRY(cudaMalloc(&mem, h.size()));
  HOM_CUDA_TRY(cudaMemcpy(mem, h.data(), h.size(), cudaMemcpyHostToDevice));
  fast2d_plan_rebase(p, static_cast<const unsigned char*>(mem));
  g_fast_cache.push_back({dev, n, run, p, mem});
  *out = p;
  return HOM_OK;
}

void fast2d_release() {
  std::lock_guard<std::mutex> lk(g_fast_mu);
  for (auto& e : g_fast_cache) {
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(e.dev);
    cudaFree(e.mem);
    cudaSetDevice(cur);
  }
  g_fast_cache.clear();
}

// row: tile | one-byte labels of 4 rows | twiddles | spare landing slots | per-phase update constants
// Green: tile | twiddles | wave numbers
// (even sizes: the tile with its padding, at most one float4 for every two positions)
namespace {
size_t tile_bytes(int n) { return ((size_t)n * NP + ((n & 1) ? 0 : n / 2)) * sizeof(float4); }
}  // namespace
size_t fast2d_smem_row(int nmax, int nphase_cell) {
  const size_t labels = (size_t)kFastRows * ((nmax + 15) / 16 * 16);
  return tile_bytes(nmax) + labels + ((size_t)nmax + 1) / 2 * 16 + (size_t)kRowSpare * sizeof(float4) +
         ((size_t)nphase_cell * 16 + 15) / 16 * 16;  // two float2 per phase (the second for the Eyre-Milton scheme)
}
size_t fast2d_smem_green(int nmax) {
  return tile_bytes(nmax) + ((size_t)nmax + 1) / 2 * 16 + ((size_t)nmax + 3) / 4 * 16;
}

namespace {
template <typename K>
int launch_tasks(K kernel, const SolveArgs& A, unsigned ntasks, size_t smem, cudaStream_t st) {
  int rc = opt_in(kernel, smem);
  if (rc != HOM_OK) return rc;
  kernel<<<ntasks, kT, smem, st>>>(A, (int)ntasks, resident_ctas(kernel, kT, smem));
  return HOM_OK;
}
}  // namespace

// `run`: 0 for compiled radices, else the largest radix of the batch's plans.
#define HOM_LAUNCH_ROW(OUT, SRC, EM)                                                                             \
  (run == 0 ? launch_tasks(k_row_f2d<OUT, SRC, EM>, A, ntasks, smem, st)                                         \
            : run <= 9 ? launch_tasks(k_row_r2d<OUT, SRC, EM, 9>, A, ntasks, smem, st)                           \
                       : launch_tasks(k_row_r2d<OUT, SRC, EM, 16>, A, ntasks, smem, st))
int fast2d_row(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st) {
  if (A.scheme == HOM_SCHEME_EYRE_MILTON) return HOM_LAUNCH_ROW(false, false, true);
  if (A.src) return HOM_LAUNCH_ROW(false, true, false);  // adjoint solve: the constitutive step takes the source term
  return HOM_LAUNCH_ROW(false, false, false);
}

int fast2d_out(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st) {
  // (`smem` with room for the x positions)
  if (A.scheme == HOM_SCHEME_EYRE_MILTON) return HOM_LAUNCH_ROW(true, false, true);
  return HOM_LAUNCH_ROW(true, false, false);
}
#undef HOM_LAUNCH_ROW

int fast2d_init(const SolveArgs& A, int ncells, cudaStream_t st) {
  dim3 grid(64, (unsigned)std::min(ncells, 65535));
  if (A.scheme == HOM_SCHEME_EYRE_MILTON) k_init_f2d<true><<<grid, 256, 0, st>>>(A, ncells);
  else k_init_f2d<false><<<grid, 256, 0, st>>>(A, ncells);
  return HOM_OK;
}

namespace {
template <bool EM>
int launch_green(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st) {
  if (run == 0) return launch_tasks(k_green_f2d<EM>, A, ntasks, smem, st);
  return run <= 9 ? launch_tasks(k_green_r2d<EM, 9>, A, ntasks, smem, st) : launch_tasks(k_green_r2d<EM, 16>, A, ntasks, smem, st);
}
}  // namespace
int fast2d_green(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st) {
  return A.scheme == HOM_SCHEME_EYRE_MILTON ? launch_green<true>(A, ntasks, smem, run, st)
                                            : launch_green<false>(A, ntasks, smem, run, st);
}

int fast2d_permute_labels(const SolveArgs& A, int ncells, long long max_nv, cudaStream_t st) {
  if (ncells > 65535) return set_error(HOM_ERR_UNSUPPORTED_SIZE, "too many cells for the label permutation");
  const unsigned gx = (unsigned)std::min<long long>((max_nv + 255) / 256, 1024);
  k_permute_labels<<<dim3(gx, (unsigned)ncells), 256, 0, st>>>(A, ncells);
  HOM_CUDA_TRY(cudaGetLastError());
  return HOM_OK;
}

}  // namespace hom
