// On-chip solver of small 2D grids (FP32, section 2, eqs. 1-a, 1-b, 2, or the Eyre-Milton scheme): one
// thread-block cluster runs a (cell, load) pair from its initial state to its stopping point.
//
// Why.  The passes of hom_fast2d.cu take three launches per iteration, and on a small grid each is a chain
// of a few short stages: at 45^2 (one cell, three loads) an iteration took 33 us for about 2 us of work.
// Here the half-spectrum state stays in the shared memory of the cluster's CTAs.  CTA r owns a block of
// row groups (4 real rows each) and a block of kx pairs; both kinds of tile have the layout of the passes
// (n positions of three float4 lane pairs):
//   rows    : pull the four rows of every kx pair of the group from the CTAs that own the pairs (distributed
//             shared memory), inverse x-DFT, constitutive update, forward x-DFT, push the rows of tau back;
//   columns : forward y-DFT, Green operator and residual, inverse y-DFT, in place;
//   control : the FP64 partial sums go to rank 0, whose first warp applies the stopping rule while the
//             others start the next rows; the flag comes back with the barrier after the pull.
// Three cluster barriers an iteration, no launch and no trip through HBM.  The Green step's private state
// (g, or u_hat of the Eyre-Milton scheme) has two buffers used in turn, in shared memory where they fit (n up
// to about 190, Eyre-Milton 170) and in the workspace otherwise: when iterate `it` passes, its own spectrum is
// rebuilt from the state it was made with, and its rows are left where the output pass reads them.  The steps are
// those of the passes, so the iterates are too.
//
// Measured, 40 iterations, 3 loads (whole call): 45^2, one cell: 1.35 ms in passes, 0.69 ms here; 143^2, two
// cells: 1.7 ms in passes, 1.11 ms.
#define HOM_FILE_ID 4
#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "hom_control.cuh"
#include "hom_fast2d.h"
#include "hom_point2d.cuh"

namespace hom {
namespace {

namespace cg = cooperative_groups;

constexpr int kTR = 256;         // threads per CTA
constexpr int kMaxCluster = 8;   // portable cluster size
constexpr int kSums = 6;         // per-rank totals: three stress sums, three residual sums
constexpr size_t kResSmem = 200 * 1024;  // dynamic shared memory a CTA may take

struct ResShape {  // how a pair of grid size n is spread over C CTAs
  int gpc, ppc;    // row groups and kx pairs per CTA
  size_t bytes;    // dynamic shared memory of a CTA, without and
  size_t priv;     // for the Green step's private state
};
__host__ __device__ inline int res_tile(int n, int pad, int r0) { return n * NP + (pad ? n / r0 : 0); }
ResShape res_shape(int n, int C, int nph, int tile, bool em) {
  const int G = (n + kFastRows - 1) / kFastRows, P = (n / 2 + 2) / 2;
  ResShape s;
  s.gpc = (G + C - 1) / C;
  s.ppc = (P + C - 1) / C;
  s.bytes = (size_t)(s.gpc + s.ppc) * tile * sizeof(float4) + ((size_t)n + 1) / 2 * 16 + ((size_t)n + 3) / 4 * 16 +
            (size_t)s.gpc * kFastRows * ((n + 15) / 16 * 16) + (size_t)s.gpc * 2 * kFastRows * NP * sizeof(float) + 2 * NP * sizeof(double) +
            ((size_t)nph * 16 + 15) / 16 * 16 + (size_t)kMaxCluster * kSums * sizeof(double) + 64;
  s.priv = 2 * (size_t)s.ppc * n * (em ? 3 : 2) * sizeof(float4);
  return s;
}

template <bool EM>
__global__ void __launch_bounds__(kTR, 2) k_resident2d(SolveArgs A, const int* list, int priv_on_chip) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RunPlan sp;
  __shared__ double s_mine[kSums];
  __shared__ int s_stop;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  HOM_DBG_POISON();
  const int pair = list[blockIdx.x / C];
  // debug builds: a pair of the batch (every CTA of the cluster finds the same and leaves before the first
  // cluster barrier, here and below)
  if (!HOM_CHECK(A, pair >= 0 && pair < A.npairs, (size_t)pair)) return;
  const PairDev pr = A.pairs[pair];
  const CellDev c = A.cells[pr.cell];
  const FastPlanDev& fp = A.fplans[c.fplan];
  if (threadIdx.x == 0) s_stop = 0;
  const RunN<NP, 16> pl(stage_plan(fp.run, sp, kTR));
  const int N = pl.n, tile = pl.tile, H = N / 2 + 1, P = (H + 1) / 2, G = (N + kFastRows - 1) / kFastRows;
  const int NL = (N + 15) / 16 * 16;
  const int gpc = (G + C - 1) / C, ppc = (P + C - 1) / C;
  const int g0 = min(rank * gpc, G), ng = min(gpc, G - g0), p0 = min(rank * ppc, P), np = min(ppc, P - p0);
  const int l = pr.load;

  // shared memory: row tiles | column tiles | twiddles | wave numbers | labels | row sums | phase constants
  float4* rows = reinterpret_cast<float4*>(smem_raw);
  float4* cols = rows + (size_t)gpc * tile;
  float2* tws = reinterpret_cast<float2*>(cols + (size_t)ppc * tile);
  float* sx = reinterpret_cast<float*>(reinterpret_cast<float4*>(tws) + (N + 1) / 2);
  uint8_t* slab = reinterpret_cast<uint8_t*>(reinterpret_cast<float4*>(sx) + (N + 3) / 4);
  double* s_part = reinterpret_cast<double*>(slab + (size_t)gpc * kFastRows * NL);  // [rank][kSums], filled by every rank
  double* s_rs = s_part + kMaxCluster * kSums;                                      // [eps, tau][component]
  float* s_dc = reinterpret_cast<float*>(s_rs + 2 * NP);                            // [group][eps, tau][row][component]
  float2* sph = reinterpret_cast<float2*>(s_dc + (size_t)gpc * 2 * kFastRows * NP);
  float2* sinv = sph + c.nph;
  constexpr int GP = EM ? 3 : 2;  // float4 per position of the Green step's private state
  float4* s_priv = reinterpret_cast<float4*>(sph + 2 * c.nph);  // [buffer][pair][position][GP]

  // debug builds: the arrays above end within the launch's dynamic shared memory, every pair's tile and
  // private state within the workspace (2 complex elements a float4), the grid within the labels, every
  // position within its tile, every kx pair with an owner
  if (!HOM_CHECK(A, reinterpret_cast<unsigned char*>(s_priv + (priv_on_chip ? 2 * (size_t)ppc * N * GP : 0)) <=
                        smem_raw + dynamic_smem(), pair) ||
      !HOM_CHECK(A, 2 * tile_index(c, N, l, P - 1, N) <= A.n_ws, pair) ||
      !HOM_CHECK(A, c.g_off + ((size_t)l * (c.Hp / 2) + P) * N * 2 * GP <= A.n_g, pair) ||
      !HOM_CHECK(A, (size_t)(c.vox_off + c.nv) <= A.n_lab, pair) || !HOM_CHECK(A, pl.at(N - 1) + NP <= tile, pair) ||
      !HOM_CHECK(A, P <= ppc * C && G <= gpc * C, pair))
    return;

  CellConst<float> cc;
  cell_const(c, cc);
  phase_constants<false, EM>(A, c, cc, sph, sinv, kTR);
  for (int i = threadIdx.x; i < (N + 1) / 2; i += kTR) cp16(tws + 2 * i, fp.tw2 + 2 * i);
  for (int i = threadIdx.x; i < (N + 3) / 4; i += kTR) cp16(sx + 4 * i, fp.xipos + 4 * i);
  const int myrows = max(0, min(ng * kFastRows, N - g0 * kFastRows));
  {
    const uint4* src = reinterpret_cast<const uint4*>(A.label8 + c.lp_off + (size_t)g0 * kFastRows * NL);
    for (int i = threadIdx.x; i < myrows * NL / 16; i += kTR) cp16(slab + 16 * i, src + i);
  }
  // the initial state of the owned pairs
  const float4* e0 = static_cast<const float4*>(A.eps[0]);
  for (int i = threadIdx.x; i < np * N * NP; i += kTR) {
    const int pp = i / (N * NP), r = i - pp * (N * NP), y = r / NP, k = r - y * NP;
    cp16(cols + (size_t)pp * tile + pl.at(y) + k, e0 + tile_index(c, N, l, p0 + pp, y) + k);
  }
  cp_commit();
  cp_wait_all();
  // the Green step's private state of an owned pair: iterate `it` was made with buffer it & 1 (in the
  // workspace: g's own array, then the pair's tile of the tau array, which these pairs do not use)
  auto priv_ws = [&](int pp, int which) -> float4* {
    const int p = p0 + pp;
    return which ? static_cast<float4*>(A.tau) + tile_index(c, N, l, p, 0)
                 : static_cast<float4*>(A.g) + (c.g_off + ((size_t)l * (c.Hp / 2) + p) * N * 2 * GP) / 2;
  };
  auto priv = [&](int pp, int which) -> float4* {
    return priv_on_chip ? s_priv + (size_t)(which * ppc + pp) * N * GP : priv_ws(pp, which);
  };
  if (priv_on_chip)
    for (int i = threadIdx.x; i < np * N * GP; i += kTR) {
      const int pp = i / (N * GP), r = i - pp * (N * GP);
      priv(pp, 0)[r] = priv_ws(pp, 0)[r];
    }
  const double* Eld = A.E + (size_t)pair * NP;
  const int nrl = ng * NP, ncl = np * NP;  // owned lines of lane pairs
  cluster.sync();

  int it = 0;
  for (;; ++it) {
    // stopping rule of the last iterate: rank 0's first warp, beside the pull below
    if (it > 0 && rank == 0 && threadIdx.x < 32) {
      double sum = 0.0;
      if (threadIdx.x < kSums)
        for (int r = 0; r < C; ++r) sum += s_part[r * kSums + threadIdx.x];
      const int still = control_pair<NP>(A, pair, (double)c.nv, sum, it - 1);
      if (threadIdx.x == 0 && !still)
        for (int r = 0; r < C; ++r) *cluster.map_shared_rank(&s_stop, r) = 1;
    }
    // rows: four half-spectrum rows -> two Hermitian-extended complex lines per component (see k_row_f2d)
    for (int f = threadIdx.x; f < ng * P * NP; f += kTR) {
      const int gl = f / (P * NP), q = f - gl * (P * NP), p = q / NP, k = q - p * NP;
      const int owner = p / ppc, y0 = (g0 + gl) * kFastRows;
      const float4* src = cluster.map_shared_rank(cols, owner) + (size_t)(p - owner * ppc) * tile + k;
      float4 v[kFastRows];
#pragma unroll
      for (int r = 0; r < kFastRows; ++r)
        v[r] = y0 + r < N ? src[pl.at(y0 + r)] : make_float4(0.f, 0.f, 0.f, 0.f);
      float4* s = rows + (size_t)gl * tile + k;
      float* dc = s_dc + (size_t)gl * 2 * kFastRows * NP + k;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int kx = 2 * p + h;
        if (kx >= H) break;
        const float2 q0 = h ? make_float2(v[0].y, v[0].w) : make_float2(v[0].x, v[0].z);
        const float2 q1 = h ? make_float2(v[1].y, v[1].w) : make_float2(v[1].x, v[1].z);
        const float2 q2 = h ? make_float2(v[2].y, v[2].w) : make_float2(v[2].x, v[2].z);
        const float2 q3 = h ? make_float2(v[3].y, v[3].w) : make_float2(v[3].x, v[3].z);
        s[pl.at(kx)] = make_float4(q0.x - q1.y, q2.x - q3.y, q0.y + q1.x, q2.y + q3.x);
        if (kx > 0) {
          if (2 * kx != N) s[pl.at(N - kx)] = make_float4(q0.x + q1.y, q2.x + q3.y, q1.x - q0.y, q3.x - q2.y);
        } else {
          dc[0] = q0.x;
          dc[NP] = q1.x;
          dc[2 * NP] = q2.x;
          dc[3 * NP] = q3.x;
        }
      }
    }
    cg::cluster_group::arrival_token tok = cluster.barrier_arrive();  // the columns may be overwritten once all have read
    __syncthreads();
    for (int st = sp.m - 1; st >= 0; --st) stage_any<NP, false, false, NP, kTR, 16, true>(rows, tws, sp, st, nrl, tile);
    for (int i = threadIdx.x; i < ng * N; i += kTR) {
      const int gl = i / N, pos = i - gl * N, y0 = (g0 + gl) * kFastRows, nr = min(kFastRows, N - y0);
      float4* s = rows + (size_t)gl * tile + pl.at(pos);
      uint32_t lab[kFastRows];
#pragma unroll
      for (int r = 0; r < kFastRows; ++r) lab[r] = r < nr ? (uint32_t)slab[(size_t)(gl * kFastRows + r) * NL + pos] : 0u;
      float4 e[NP], o[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) e[k] = s[k];
      tau_point<false, false, EM>(A, c, fp, sph, sinv, cc, nr, y0, l, pos, lab, e, o);
#pragma unroll
      for (int k = 0; k < NP; ++k) s[k] = o[k];
    }
    __syncthreads();
    for (int st = 0; st < sp.m; ++st) stage_any<NP, true, true, NP, kTR, 16, true>(rows, tws, sp, st, nrl, tile);
    cluster.barrier_wait(std::move(tok));
    if (s_stop) break;
    // split the two real rows of each line and push the half spectra of tau to the owners of their columns
    for (int f = threadIdx.x; f < ng * P * NP; f += kTR) {
      const int gl = f / (P * NP), q = f - gl * (P * NP), p = q / NP, k = q - p * NP;
      const int owner = p / ppc, y0 = (g0 + gl) * kFastRows;
      const float4* s = rows + (size_t)gl * tile + k;
      float* dc = s_dc + (size_t)gl * 2 * kFastRows * NP + kFastRows * NP + k;
      float4 w[kFastRows];
#pragma unroll
      for (int r = 0; r < kFastRows; ++r) w[r] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int kx = 2 * p + h;
        if (kx >= H) break;
        const float4 Z = s[pl.at(kx)];
        const float4 Zm = s[pl.at(kx == 0 ? 0 : N - kx)];
        const float2 o0 = make_float2(0.5f * (Z.x + Zm.x), 0.5f * (Z.z - Zm.z));
        const float2 o1 = make_float2(0.5f * (Z.z + Zm.z), 0.5f * (Zm.x - Z.x));
        const float2 o2 = make_float2(0.5f * (Z.y + Zm.y), 0.5f * (Z.w - Zm.w));
        const float2 o3 = make_float2(0.5f * (Z.w + Zm.w), 0.5f * (Zm.y - Z.y));
        if (h == 0) {
          w[0].x = o0.x; w[0].z = o0.y; w[1].x = o1.x; w[1].z = o1.y;
          w[2].x = o2.x; w[2].z = o2.y; w[3].x = o3.x; w[3].z = o3.y;
          if (kx == 0) {
            dc[0] = o0.x;
            dc[NP] = o1.x;
            dc[2 * NP] = o2.x;
            dc[3 * NP] = o3.x;
          }
        } else {
          w[0].y = o0.x; w[0].w = o0.y; w[1].y = o1.x; w[1].w = o1.y;
          w[2].y = o2.x; w[2].w = o2.y; w[3].y = o3.x; w[3].w = o3.y;
        }
      }
      float4* dst = cluster.map_shared_rank(cols, owner) + (size_t)(p - owner * ppc) * tile + k;
#pragma unroll
      for (int r = 0; r < kFastRows; ++r)
        if (y0 + r < N) dst[pl.at(y0 + r)] = w[r];
    }
    cluster.sync();
    // sum of sigma over the owned rows (see the row pass), FP64: warp q sums row values q = (eps or tau,
    // component) over the rows, and c0 is applied to the sums
    if (threadIdx.x < 2 * NP * 32) {
      const int q = threadIdx.x >> 5, lane = threadIdx.x & 31, which = q / NP, k = q - which * NP;
      double x = 0.0;
      for (int r = lane; r < myrows; r += 32)
        x += (double)s_dc[((size_t)(r / kFastRows) * 2 + which) * kFastRows * NP + (r % kFastRows) * NP + k];
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) s_rs[q] = x;
    }
    // columns
    for (int st = sp.m - 1; st >= 0; --st) stage_any<NP, true, false, NP, kTR, 16, true>(cols, tws, sp, st, ncl, tile);
    Acc<float> acc[EM ? 3 : 2];
    if constexpr (EM) {
      GreenPairEm gp(A, c, fp, 0, Eld);
      for (int i = threadIdx.x; i < np * 2 * N; i += kTR) {
        const int pp = i / (2 * N), q = i - pp * (2 * N), pos = q >> 1, h = q & 1, kx0 = 2 * (p0 + pp);
        float* T = reinterpret_cast<float*>(cols + (size_t)pp * tile + pl.at(pos));
        if (h && kx0 + 1 >= H) {  // the missing lane B of the last pair stays zero
#pragma unroll
          for (int k = 0; k < NP; ++k) T[4 * k + 1] = T[4 * k + 3] = 0.f;
          continue;
        }
        gp.set_pair(N, fp, kx0);
        const float2* uin = reinterpret_cast<const float2*>(priv(pp, it & 1)) + 6 * pos + 3 * h;
        float2* uout = reinterpret_cast<float2*>(priv(pp, (it + 1) & 1)) + 6 * pos + 3 * h;
        gp.point(T, h, sx[pos], pos == 0, uin, uout, acc);
      }
    } else {
      GreenPair gp(A, c, fp, 0, pair);
      for (int i = threadIdx.x; i < np * N; i += kTR) {
        const int pp = i / N, pos = i - pp * N;
        gp.set_pair(N, fp, 2 * (p0 + pp));
        const float4* gin = priv(pp, it & 1) + 2 * pos;
        const float4 g[2] = {gin[0], gin[1]};
        gp.point(cols + (size_t)pp * tile + pl.at(pos), sx[pos], pos == 0, g, priv(pp, (it + 1) & 1) + 2 * pos);
      }
      gp.sums(acc);
    }
    double tot[EM ? 3 : 2];
    block_sum<float, EM ? 3 : 2, kTR>(acc, tot);  // contains the barrier before the inverse transform
    if (threadIdx.x == 0) {
#pragma unroll
      for (int q = 0; q < 3; ++q) s_mine[NP + q] = q < (EM ? 3 : 2) ? tot[q] : 0.0;
    }
    if (threadIdx.x >= 32 && threadIdx.x < 32 + NP) {
      const int k = threadIdx.x - 32;
      const double tau = s_rs[NP + k], u = s_rs[k], tr = s_rs[0] + s_rs[1];
      s_mine[k] = EM ? 0.5 * (tau + (double)N * u)
                     : tau + (double)N * (2.0 * c.mu0 * u + (k < 2 ? c.lam0 * tr : 0.0));
    }
    for (int st = 0; st < sp.m; ++st) stage_any<NP, false, true, NP, kTR, 16, true>(cols, tws, sp, st, ncl, tile);
    if (threadIdx.x < kSums) cluster.map_shared_rank(s_part, 0)[rank * kSums + threadIdx.x] = s_mine[threadIdx.x];
    cluster.sync();
  }

  // iterate it - 1 is the one returned: its spectrum from the state it was made with, inverse y-DFT, and its
  // rows to the eps buffer the output pass reads
  const int ret = it - 1;
  for (int pp = 0; pp < np; ++pp) {
    const int p = p0 + pp;
    const float4* g = priv(pp, ret & 1);
    if constexpr (EM) {
      const bool hasB = 2 * p + 1 < H;
      for (int i = threadIdx.x; i < 2 * N; i += kTR) {
        const int pos = i >> 1, h = i & 1;
        float* T = reinterpret_cast<float*>(cols + (size_t)pp * tile + pl.at(pos));
        const float2* u = reinterpret_cast<const float2*>(g) + 6 * pos + 3 * h;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          const float2 x = h && !hasB ? make_float2(0.f, 0.f) : u[k];
          T[4 * k + h] = x.x;
          T[4 * k + 2 + h] = x.y;
        }
      }
    } else {
      const GreenPair gp(A, c, fp, 2 * p, pair);
      for (int pos = threadIdx.x; pos < N; pos += kTR)
        gp.spectrum(cols + (size_t)pp * tile + pl.at(pos), sx[pos], pos == 0, g[2 * pos], g[2 * pos + 1]);
    }
  }
  __syncthreads();
  for (int st = 0; st < sp.m; ++st) stage_any<NP, false, true, NP, kTR, 16, true>(cols, tws, sp, st, ncl, tile);
  float4* out = static_cast<float4*>(A.eps[ret & 1]);
  for (int i = threadIdx.x; i < np * N * NP; i += kTR) {
    const int pp = i / (N * NP), r = i - pp * (N * NP), y = r / NP, k = r - y * NP;
    out[tile_index(c, N, l, p0 + pp, y) + k] = cols[(size_t)pp * tile + pl.at(y) + k];
  }
  cluster.sync();  // no CTA leaves while another may still write to its shared memory
}


// Which batches run on chip: those whose every grid fits a cluster (n up to about 235), and whose clusters are
// estimated faster than the passes.  A cluster's iteration is a chain of short stages whatever else runs, so
// further waves of clusters soon lose to the passes, which fill the chip (64 random-disk cells, 39 of their 64
// grids eligible: 8.4 ms in passes, 11.2 ms with the small grids on chip first), and small grids beside large
// ones ride along in the passes' launches (the 2D sweep: 28.9 ms, 30.1 ms): a batch goes on chip as a whole or
// not at all.
//
// The estimates, in us an iteration, follow measurements at n = 15 to 243, 1 to 48 pairs, both schemes:
//   on chip: 8 + (0.007 + 0.0045 m) g n per wave of clusters, g row groups a CTA, m stages of the transform; 1.28
//            times that for the Eyre-Milton scheme; cluster sizes run one after another.  105: 15.2, 150: 25 (three
//            stages), 165: 24, 195: 32, 208: 34, 225: 37, 243: 43; Eyre-Milton 165: 31, 195: 41, 225: 49.
//   passes : 16 + 16 per wave of their CTAs with radices from a plan (three an SM up to radix 9, else two):
//            105 to 243: 30, 46 and 62 for one to three waves; 16 + 0.06 n per wave with compiled ones (135: 22 and
//            33, 225: 28 and 45); 1.08 times that for the Eyre-Milton scheme.  These are a graph's; the
//            host loop takes 5 more, and half of that is added for either, since a graph gives the loop's results bit
//            for bit.
// They cross near n = 210 (Eyre-Milton 180) for batches of one wave of passes, and below 225, which has compiled
// radices; with two or three waves of passes most sizes that fit gain on chip (208, 12 pairs: 34 against 64),
// unless their clusters take two waves too (152 SMs place about 15 clusters of 8 CTAs that fill an SM each:
// 225, 16 pairs: 75 against 49; 165: 48 against 61).
struct ResGroup {  // pairs of one cluster size
  std::vector<int> pairs;
  size_t bytes = 0, full = 0;  // dynamic shared memory without and with the private state on chip
  double us = 0.0;             // an iteration of the slowest
};
double on_chip_us(const ResShape& sh, int n, int stages, bool em) {
  return (em ? 1.28 : 1.0) * (8.0 + (0.007 + 0.0045 * stages) * sh.gpc * n);
}
double passes_us(const std::vector<int>& sizes, int L, int run, bool em, int sms) {
  long long tasks = 0;
  int nmax = 0;
  for (int n : sizes) {
    tasks += (long long)L * ((n / 2 + 2) / 2);
    nmax = std::max(nmax, n);
  }
  const long long slots = (long long)sms * (run > 9 ? 2 : 3), waves = (tasks + slots - 1) / slots;
  return (em ? 1.08 : 1.0) * (16.0 + (run ? 16.0 : 0.06 * nmax) * (double)waves) + 2.5;
}
// Clusters of `kernel` on the device at once, cached for the last few (device, kernel, size, shared memory) asked;
// 0 where it can place none.
template <typename K>
int active_clusters(K kernel, const cudaLaunchConfig_t& cfg) {
  struct Last { const void* k = nullptr; int dev = -1; unsigned size = 0; size_t smem = 0; int val = 0; };
  static thread_local Last last[8];
  static thread_local int next = 0;
  const void* kp = reinterpret_cast<const void*>(kernel);
  const unsigned size = cfg.attrs[0].val.clusterDim.x;
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  for (const Last& e : last)
    if (e.k == kp && e.dev == dev && e.size == size && e.smem == cfg.dynamicSmemBytes) return e.val;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  last[next] = Last{kp, dev, size, cfg.dynamicSmemBytes, n};
  next = (next + 1) & 7;
  return n;
}

using ResKernel = void (*)(SolveArgs, const int*, int);
ResKernel res_kernel(bool em) { return em ? k_resident2d<true> : k_resident2d<false>; }
struct ResLaunch {  // one launch: the pairs of one cluster size
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr = {};
  int priv_on_chip = 0;
};
// The launches of a batch that runs on chip (clusters of 2^q CTAs), or false: it runs in passes.  Within the rule
// above, a grid is spread until a CTA holds about four row groups or the chip is full.
bool res_launches(const std::vector<int>& sizes, const std::vector<int>& stages, int L, int run, int nphase_cell, bool em,
                  ResGroup (&by_size)[4], ResLaunch (&launch)[4]) {
  const int sms = sm_count(), pairs = (int)sizes.size() * L;
  std::vector<int> least(sizes.size(), 0);
  int ctas = 0;
  if (pairs > sms) return false;
  for (size_t i = 0; i < sizes.size(); ++i) {
    const int n = sizes[i];
    const int tile = res_tile(n, !(n & 1), 2);  // an upper bound for any first radix
    for (int C = 1; C <= kMaxCluster && !least[i]; C *= 2)
      if (res_shape(n, C, nphase_cell, tile, em).bytes <= kResSmem) least[i] = C;
    ctas += least[i] * L;
    if (!least[i] || ctas > sms) return false;
  }
  for (size_t i = 0; i < sizes.size(); ++i) {
    const int n = sizes[i], G = (n + kFastRows - 1) / kFastRows;
    int C = least[i];
    while (C < kMaxCluster && (ctas + C * L) <= sms && pairs * C * 2 <= sms && (G + C - 1) / C > 4) {
      ctas += C * L;
      C *= 2;
    }
    ResGroup& g = by_size[C == 1 ? 0 : C == 2 ? 1 : C == 4 ? 2 : 3];
    for (int l = 0; l < L; ++l) g.pairs.push_back((int)i * L + l);
    const ResShape sh = res_shape(n, C, nphase_cell, res_tile(n, !(n & 1), 2), em);
    g.bytes = std::max(g.bytes, sh.bytes);
    g.full = std::max(g.full, sh.bytes + sh.priv);
    g.us = std::max(g.us, on_chip_us(sh, n, stages[i], em));
  }
  const ResKernel kernel = res_kernel(em);
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  double chip_us = 0.0;
  for (int q = 3; q >= 0; --q) {
    const ResGroup& g = by_size[q];
    if (g.pairs.empty()) continue;
    ResLaunch& l = launch[q];
    l.priv_on_chip = g.full <= kResSmem;
    l.attr.id = cudaLaunchAttributeClusterDimension;
    l.attr.val.clusterDim.x = 1u << q;
    l.attr.val.clusterDim.y = l.attr.val.clusterDim.z = 1;
    l.cfg.gridDim = dim3((unsigned)g.pairs.size() << q);
    l.cfg.blockDim = dim3(kTR);
    l.cfg.dynamicSmemBytes = l.priv_on_chip ? g.full : g.bytes;
    l.cfg.attrs = &l.attr;
    l.cfg.numAttrs = 1;
    // a device (or a slice of one) that cannot place such a cluster leaves the batch to the passes
    const int clusters = active_clusters(kernel, l.cfg);
    if (clusters < 1) return false;
    chip_us += g.us * (double)(((int)g.pairs.size() + clusters - 1) / clusters);
  }
  return chip_us <= passes_us(sizes, L, run, em, sms);
}

}  // namespace

bool resident2d_takes(const std::vector<int>& sizes, const std::vector<int>& stages, int L, int run, int nphase_cell, bool em) {
  ResGroup by_size[4];
  ResLaunch launch[4];
  return res_launches(sizes, stages, L, run, nphase_cell, em, by_size, launch);
}

int resident2d_solve(const SolveArgs& A, const std::vector<CellDev>& cells, const std::vector<FastPlanDev>& plans, int L,
                     int run, int* list, int nphase_cell, cudaStream_t st, int* count) {
  *count = 0;
  std::vector<int> sizes, stages, all;
  for (const CellDev& c : cells) {
    sizes.push_back(c.n);
    stages.push_back(plans[c.fplan].run.m);
  }
  const bool em = A.scheme == HOM_SCHEME_EYRE_MILTON;
  ResGroup by_size[4];
  ResLaunch launch[4];
  if (!res_launches(sizes, stages, L, run, nphase_cell, em, by_size, launch)) return HOM_OK;
  for (int q = 3; q >= 0; --q) all.insert(all.end(), by_size[q].pairs.begin(), by_size[q].pairs.end());
  HOM_CUDA_TRY(cudaMemcpyAsync(list, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  const int* at = list;
  for (int q = 3; q >= 0; --q) {
    if (by_size[q].pairs.empty()) continue;
    launch[q].cfg.stream = st;
    HOM_CUDA_TRY(cudaLaunchKernelEx(&launch[q].cfg, res_kernel(em), A, at, launch[q].priv_on_chip));
    at += by_size[q].pairs.size();
  }
  HOM_CUDA_TRY(cudaStreamSynchronize(st));  // the list's host copy goes out of scope
  *count = (int)all.size();
  return HOM_OK;
}

}  // namespace hom
