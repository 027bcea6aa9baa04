// FP32 lane-pair passes of the fixed-point and Eyre-Milton schemes (section 2, eqs. 1-a, 1-b, 2), 2D and 3D,
// with radices compiled in for a few sizes and read from a plan for every other, and the on-chip solver of
// small 2D grids.  They compute what the generic passes of hom_solver.cu compute, on the same task lists and
// partial sums; see hom_fast2d.cu for the data layouts.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "hom_common.cuh"

namespace hom {

struct SolveArgs;

// Stages of a transform whose length is known at run time only (RunN in hom_fastfft.cuh), DIT order.
constexpr int kMaxRunStages = 5;
struct RunPlan {
  int n, m;              // length, stages
  int pad;               // 1: one float4 of padding after every r[0] positions (even r[0])
  int r[kMaxRunStages], L[kMaxRunStages];  // radix and span of each stage
  int tw[kMaxRunStages];                   // offset of its twiddle table
  FastDiv d_nb[kMaxRunStages], d_L[kMaxRunStages], d_r0;
};

// Device tables of one grid size n, in the digit order of its radices (compiled in or of `run`).
struct FastPlanDev {
  const uint16_t* iperm;  // iperm[pos]: index held at position pos after a DIF transform
  const float* xipos;     // 2 pi a(iperm[pos]): wave number of the bin at position pos
  const float* xinat;     // 2 pi a(k) in natural order
  const float2* tw2;      // the stages' twiddle tables, (cos, -sin) pairs
  int n;
  RunPlan run;            // the same transform for the run-time-size passes
};

constexpr int kFastRows = 4;  // real rows per row-pass task (two complex lines, one lane pair)
constexpr int kFastCols = 2;  // kx columns per Green-pass task (one lane pair)

// True if n has specialised 2D / 3D passes with its radices compiled in, and if it fits the passes
// whose radices are chosen at run time (every supported size up to what a tile can hold on chip).
bool fast2d_size(int n);
bool fast3d_size(int n);
bool run2d_size(int n);
bool run3d_size(int n);
// Largest radix and number of stages of the plan-read transform of size n.
void run_plan_shape(int n, int* largest, int* stages);
// Device tables of size n (built and uploaded on first use, kept until hom_release).  `run`: for the
// passes with run-time radices, whose digit order differs from the compiled ones'.
int fast2d_plan(int n, bool run, FastPlanDev* out);
// The same tables built on the host only (no device allocation): `h` receives them and `out` their
// layout, with byte offsets from the start of `h` in place of the table pointers; after `h` is
// copied to device memory at `base`, fast2d_plan_rebase turns the offsets into device pointers.
int fast2d_plan_host(int n, bool run, std::vector<unsigned char>& h, FastPlanDev* out);
void fast2d_plan_rebase(FastPlanDev& p, const unsigned char* base);
// Dynamic shared memory of the row and Green passes for the largest grid size n of a call.
size_t fast2d_smem_row(int nmax, int nphase_cell);
size_t fast2d_smem_green(int nmax);
// Launches (one CTA per task); `smem` from fast2d_smem_row / fast2d_smem_green; `run`: 0 for
// compiled radices, else the largest radix of the batch's plans.
int fast2d_row(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st);
int fast2d_green(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st);
// Output pass (final eps and sigma fields) and the initial state eps = E, in the tiled layout of
// the specialised passes (see hom_fast2d.cu).
int fast2d_out(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st);
int fast2d_init(const SolveArgs& A, int ncells, cudaStream_t st);
// label8[lp_off + y nl + pos] = index, in the cell's list of pure phases, of the phase of
// label[vox_off + y n + iperm[pos]] (255 for a mixed voxel; nl = n rounded up to 16).
int fast2d_permute_labels(const SolveArgs& A, int ncells, long long max_nv, cudaStream_t st);
void fast2d_release();

// On-chip solver of batches of small grids (hom_resident2d.cu): where every pair of the batch fits and it is the
// faster way, runs all of them to their stopping points and leaves them inactive, their iterates where the output pass reads them.
// `run` as above; `list` holds room for every pair; *count receives the number of pairs taken, all or none.
struct CellDev;
int resident2d_solve(const SolveArgs& A, const std::vector<CellDev>& cells, const std::vector<FastPlanDev>& plans, int L,
                     int run, int* list, int nphase_cell, cudaStream_t st, int* count);
// Whether it will: the cells' sizes and the stages of their plans.
bool resident2d_takes(const std::vector<int>& sizes, const std::vector<int>& stages, int L, int run, int nphase_cell, bool em);

// Specialised 3D passes (hom_fast3d.cu): row, y forward / inverse, Green (z lines), the initial
// state eps = E and the output pass, on the kx-pair tiled state of those passes.
size_t fast3d_smem_row(int nmax, int nphase_cell);
size_t fast3d_smem_y(int nmax);
size_t fast3d_smem_green(int nmax);
int fast3d_row(const SolveArgs& A, unsigned ntasks, size_t smem, bool out, int run, cudaStream_t st);
int fast3d_ypass(const SolveArgs& A, unsigned ntasks, size_t smem, bool fwd, int run, cudaStream_t st);
int fast3d_green(const SolveArgs& A, unsigned ntasks, size_t smem, int run, cudaStream_t st);
int fast3d_init(const SolveArgs& A, int ncells, cudaStream_t st);

}  // namespace hom
