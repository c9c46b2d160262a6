// solver_dev.cuh -- what the Poisson solver's translation units share: launches
// with programmatic dependent edges, the grid-wide sum that finishes in its own
// kernel, the 7-point neighbour sums and the error-free sum of two floats.
#pragma once

#include <utility>

#include <cuda_runtime.h>

#include "pic_internal.cuh"
#include "pic_solver.cuh"

namespace pic {

// Programmatic dependent launch: each solver kernel may be launched while its
// predecessor drains (it waits here until the predecessor has completed and its
// writes are visible), and lets its own successor launch as soon as all of its
// blocks are running. Hides most of the launch gap between the many short
// multigrid kernels. A no-op for kernels launched without the attribute.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

extern bool g_pdl;  // cleared when a graph with programmatic edges cannot be built

template <class K>
struct PdlLaunch {
  K k;
  dim3 g, b;
  size_t smem;
  cudaStream_t s;
  template <class... A>
  void operator()(A&&... a) const {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = g_pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, k, std::forward<A>(a)...);
  }
};
#define SOLVER_LAUNCH(grid, block, smem, stream, ...) \
  (::pic::count_kernel()), ::pic::PdlLaunch<decltype(&__VA_ARGS__)>{&__VA_ARGS__, dim3(grid), dim3(block), (size_t)(smem), stream}

// Level geometry with 32-bit indices (a level holds far fewer than 2^31 unknowns).
struct Lv {
  int nx, ny, nz, pl, nu;
};
inline Lv lv_of(const MgLevel& L) { return Lv{L.nx, L.ny, L.nz, L.nx * L.ny, (int)L.nu}; }

template <class T>
__device__ __forceinline__ T nb_sum(const Lv& L, const T* __restrict__ x, int u, int i, int j, int k) {
  // k: unknown plane index 0..nz-2
  const int row = u - i;
  const int im = i == 0 ? L.nx - 1 : i - 1, ip = i == L.nx - 1 ? 0 : i + 1;
  const int rm = j == 0 ? (L.ny - 1) * L.nx : -L.nx;
  const int rp = j == L.ny - 1 ? -(L.ny - 1) * L.nx : L.nx;
  T s = x[row + im] + x[row + ip] + x[u + rm] + x[u + rp];
  if (k > 0) s += x[u - L.pl];
  if (k < L.nz - 2) s += x[u + L.pl];
  return s;
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bv = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bv)), __fsub_rn(b, bv));
}

// sum of the six neighbours of u as s + e (s rounded, e the accumulated exact errors)
__device__ __forceinline__ void nb_sum_ff(const Lv& L, const float* __restrict__ x, int u, int i, int j, int k, float& s,
                                          float& e) {
  const int row = u - i;
  const int im = i == 0 ? L.nx - 1 : i - 1, ip = i == L.nx - 1 ? 0 : i + 1;
  const int rm = j == 0 ? (L.ny - 1) * L.nx : -L.nx;
  const int rp = j == L.ny - 1 ? -(L.ny - 1) * L.nx : L.nx;
  float t;
  s = x[row + im];
  e = 0.f;
  two_sum(s, x[row + ip], s, t);
  e = __fadd_rn(e, t);
  two_sum(s, x[u + rm], s, t);
  e = __fadd_rn(e, t);
  two_sum(s, x[u + rp], s, t);
  e = __fadd_rn(e, t);
  if (k > 0) {
    two_sum(s, x[u - L.pl], s, t);
    e = __fadd_rn(e, t);
  }
  if (k < L.nz - 2) {
    two_sum(s, x[u + L.pl], s, t);
    e = __fadd_rn(e, t);
  }
}

template <class V>
__device__ __forceinline__ V warp_sum(V d) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
  return d;
}

// Grid-wide sum without a second launch: each block stores its partial in
// part[block], then the last block to arrive (a ticket counter) adds all
// partials in a fixed order (fixed thread assignment and tree, so the total is
// reproducible) and resets the ticket. Returns true in thread 0 of that block
// only, with the total in *tot. Every thread of every block must call it.
// Per-thread and warp sums stay in V (FP32 for the FP32 solve: FP64 is a narrow
// pipe on GB300); warp totals and everything above them are FP64.
template <class V>
__device__ __forceinline__ bool grid_total(V v, double* part, unsigned* ticket, double* tot) {
  __shared__ double sm[32];
  __shared__ int s_last;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int nthr = blockDim.x * blockDim.y;
  const int nw = nthr >> 5;
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  const V w = warp_sum(v);
  if ((tid & 31) == 0) sm[tid >> 5] = (double)w;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int k = 0; k < nw; ++k) s += sm[k];
    part[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == nb - 1u ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  // four independent partial sums per thread keep several loads in flight
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  unsigned i = tid;
  for (; i + 3u * nthr < nb; i += 4u * nthr) {
    s0 += __ldcg(part + i);
    s1 += __ldcg(part + i + nthr);
    s2 += __ldcg(part + i + 2u * nthr);
    s3 += __ldcg(part + i + 3u * nthr);
  }
  for (; i < nb; i += nthr) s0 += __ldcg(part + i);
  double s = warp_sum((s0 + s1) + (s2 + s3));
  __syncthreads();
  if ((tid & 31) == 0) sm[tid >> 5] = s;
  __syncthreads();
  if (tid != 0) return false;
  double t = 0.0;
  for (int k = 0; k < nw; ++k) t += sm[k];
  *tot = t;
  *ticket = 0u;
  return true;
}

}  // namespace pic
