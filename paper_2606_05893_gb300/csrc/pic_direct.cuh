// pic_direct.cuh -- the direct solver of the scaled 7-point operator: real FFTs
// along the periodic x and y, a tridiagonal solve along z per Fourier mode.
#pragma once

#include <vector>

#include <cuda_runtime.h>

#include "pic_internal.cuh"

namespace pic {

struct SolveCtl;
struct MgLevel;

constexpr int kDirMaxPasses = 8;
constexpr int kDirLines = 16;  // lines an FFT block transforms together (16 float2: one 128-byte row)

// One periodic axis of n points: passes of an in-place decimation-in-frequency
// FFT (radix R on blocks of L points, M = L / R), its outputs left in
// digit-reversed order (pos[f]: where frequency f ends up).
struct AxisPlan {
  int n, npass;
  int pow2;      // every radix one of 2, 4, 8, 16
  int pingpong;  // a radix without an unrolled butterfly: passes alternate between two buffers
  int R[kDirMaxPasses], L[kDirMaxPasses];
  FastDiv dM[kDirMaxPasses];
  const float2* tw;  // [n] exp(-2 pi i m / n)
  const int* pos;    // [n]
};

struct DirectArgs {
  int nx, ny, P;   // cells in x and y, unknown planes
  int C;           // complex columns kept per row of x (nx even: Nyquist packed with the mean)
  int packed;      // nx even
  int plane;       // floats per plane of the spectrum, 2 C ny
  long long rows;  // ny P rows of x
  float norm;      // 1 / (nx ny)
  AxisPlan x, y;
  const int2* col;   // [C] where column c's frequency f and -f end up (columns in the order of the former)
  const float* lam;  // [plane] x and y eigenvalue of every float of a spectral plane
  float* spec;       // [P][ny][C] float2
};

// What the residual kernels need to decide on another pass.
struct DirectLoop {
  double rtol;
  int maxit, max_outer, use_graph;
  cudaGraphConditionalHandle handle;
  double margin2 = 1.0;  // below 1: a residual that meets the tolerance (squared) but not margin2 of it takes one
                         // more pass, unless the tolerance is within SolveCtl::floor2
};
constexpr int kDirParts = 1 << 15;  // blocks of a residual launch (two partial sums each)

struct DirectSolver {
  bool on = false;
  DirectArgs a{};
  void* tables = nullptr;
  size_t smem_x = 0, smem_y = 0, smem_xy = 0;
  bool planes = false;  // whole planes in one block (both axes in one launch each way)
  int zm = 0, zw = 0;  // planes per warp and warps of the tridiagonal kernel
  // nz - 1 unknown planes; on stays false where the sizes do not fit
  cudaError_t init(int nx, int ny, int nz);
  // the same in parts, on memory of the caller's: the plan (false: the sizes do
  // not fit), what it needs, and its placement (the tables are written on s)
  bool plan(int nx, int ny, int nz);
  size_t table_bytes() const;
  size_t spec_bytes() const;
  cudaError_t place(void* tables_mem, void* spec_mem, cudaStream_t s);
  void release();
  // x += A^-1 r: r FP32 (mixed: x is hi + lo) or FP64 (x FP64), unknown view,
  // [k][j][i]. Nothing is done once c->stopped is set, except that a zero
  // right-hand side sets x = 0.
  void apply_mixed(const float* r, float* hi, float* lo, double phi_c, double dphi_dk, const SolveCtl* c,
                   cudaStream_t s) const;
  void apply_fp64(const double* r, double* x, const SolveCtl* c, cudaStream_t s) const;
  // r = b - A x and the decision on another pass (SolveCtl); first: b.b and the
  // tolerance too, later: nothing once c->stopped is set. part: 2 kDirParts doubles.
  void residual_mixed(bool first, const MgLevel& M, const float* hi, const float* lo, const float* f, float* r,
                      float fold_first, float fold_last, double* part, SolveCtl* c, const DirectLoop& d,
                      cudaStream_t s) const;
  void residual_fp64(bool first, const MgLevel& M, const double* x, const double* b, double* r, double* part, SolveCtl* c,
                     const DirectLoop& d, cudaStream_t s) const;
};

}  // namespace pic
