// k_direct.cu -- direct solve of A d = r for the scaled 7-point operator of
// Eq. (1) on the node grid (periodic x, y; Dirichlet planes in z), in FP32.
//
// A is the sum of two periodic second differences and one Dirichlet one, so the
// discrete Fourier modes of x and y decouple it into one tridiagonal system per
// mode, (2 + lx + ly) u_k - u_(k-1) - u_(k+1) = f_k. Five launches:
//   k_dir_xf  real FFT of every row (two rows packed as one complex line)
//   k_dir_y   complex FFT of every column of a plane
//   k_dir_z   tridiagonal solve of every mode, the planes split over warps
//   k_dir_y, k_dir_xi  the inverse transforms; the last adds d to the potential
// (planes of about 32 x 32 points: three, k_dir_xyf and k_dir_xyi transform both axes)
// The solve is one pass of iterative refinement: the caller forms r = b - A x in
// float-float (mixed) or FP64, and repeats until the residual meets its tolerance.
// FP32 rounding leaves 1e-6 to 1e-3 of the residual per pass (the most for modes
// that are smooth in all three directions), so a warm-started mixed solve to 1e-8
// takes one pass and an FP64 one to 1e-13 two or three.
//
// What bounds the kernels: every pass over a vector of the unknowns is one read
// and one write of L2 (up to 128x128x256) or HBM; the butterflies are far below
// the FP32 rate. A block holds 16 lines of an axis with the line index innermost
// in shared memory, so every butterfly access of a half warp is one contiguous
// 128-byte row whatever the radix (rows of 17 float2 in x, where the loads
// transpose). What is left is latency: a tile is loaded by asynchronous copies,
// all in flight at once, and the last kernel loads what it adds to in batches
// before it stores (256x256x512: k_dir_xi 281 -> 170 us, with wider blocks 148, with
// the columns ordered by their place in the tile 123; k_dir_z with its pivots in
// shared memory, two blocks an SM instead of one, 108 -> 71). Spectra stay in the
// order the passes leave them in (digit reversed): the tridiagonal kernel only
// needs each column's eigenvalue.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "dev_mem.cuh"
#include "pic_direct.cuh"
#include "pic_internal.cuh"
#include "pic_solver.cuh"
#include "solver_dev.cuh"

namespace pic {

namespace {

constexpr int kFftThreads = 256;  // most threads of an FFT block: x tiles above 128 points (k_dir_xi 170 -> 148 us
                                  // at 256x256x512); the others 128 (y tiles with 256: 55 -> 65 us)
constexpr int kLpX = kDirLines + 1;  // row pitch (float2) of the x tiles
constexpr int kLpY = kDirLines;

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a w (forward) or a conj(w) (inverse)
template <bool INV>
__device__ __forceinline__ float2 ctw(float2 a, float2 w) {
  return INV ? make_float2(fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -a.x * w.y))
             : make_float2(fmaf(a.x, w.x, -a.y * w.y), fmaf(a.y, w.x, a.x * w.y));
}
// -i a (forward) or i a (inverse)
template <bool INV>
__device__ __forceinline__ float2 crot(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// cos(2 pi m / 16), m = 0..4
__device__ __forceinline__ constexpr float cos16(int m) {
  return m == 0 ? 1.f : (m == 1 ? 0.923879532511286756f : (m == 2 ? 0.707106781186547524f : (m == 3 ? 0.382683432365089772f : 0.f)));
}

// Power-of-two DFT, natural order in and out: halves of even and odd index.
template <int R, bool INV>
struct Dft {
  static __device__ __forceinline__ void run(float2 (&v)[R]) {
    float2 e[R / 2], o[R / 2];
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    Dft<R / 2, INV>::run(e);
    Dft<R / 2, INV>::run(o);
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      const int m = k * (16 / R);  // exp(-2 pi i m / 16), m < 8
      float2 t = o[k];
      if (m == 4) t = crot<INV>(t);
      else if (m > 0) {
        const float c = m < 4 ? cos16(m) : -cos16(8 - m), s = m < 4 ? cos16(4 - m) : cos16(m - 4);
        t = ctw<INV>(t, make_float2(c, -s));
      }
      v[k] = cadd(e[k], t);
      v[k + R / 2] = csub(e[k], t);
    }
  }
};
template <bool INV>
struct Dft<1, INV> {
  static __device__ __forceinline__ void run(float2 (&)[1]) {}
};

// DFT of an odd prime length: x_s +- x_(R-s) pair up, so each output pair (k, R - k) takes
// (R - 1) / 2 real products of each kind. w[m] = exp(-2 pi i m / R).
template <int R, bool INV>
__device__ __forceinline__ void dft_odd(float2 (&v)[R], const float2* w, int step) {
  constexpr int H = (R - 1) / 2;
  float2 a[H], b[H];
  float c[H], s[H];
  float2 y0 = v[0];
#pragma unroll
  for (int q = 0; q < H; ++q) {
    a[q] = cadd(v[q + 1], v[R - 1 - q]);
    b[q] = csub(v[q + 1], v[R - 1 - q]);
    const float2 t = w[(q + 1) * step];
    c[q] = t.x;
    s[q] = -t.y;
    y0 = cadd(y0, a[q]);
  }
  const float2 x0 = v[0];
  v[0] = y0;
#pragma unroll
  for (int k = 1; k <= H; ++k) {
    float2 re = x0, im = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < H; ++q) {
      const int m = (k * (q + 1)) % R;  // 1..R - 1, R being prime
      const float cm = m <= H ? c[m - 1] : c[R - m - 1];
      const float sm = m <= H ? s[m - 1] : -s[R - m - 1];
      re = make_float2(fmaf(cm, a[q].x, re.x), fmaf(cm, a[q].y, re.y));
      im = make_float2(fmaf(sm, b[q].x, im.x), fmaf(sm, b[q].y, im.y));
    }
    const float2 t = crot<INV>(im);
    v[k] = cadd(re, t);
    v[R - k] = csub(re, t);
  }
}

// One pass over the tiles (one after the other in memory): butterflies of radix R
// on blocks of L points.
template <int R, bool INV, int LP>
__device__ __forceinline__ void fft_pass(float2* Z, const float2* tw, int n, int L, const FastDiv& dM, int tiles) {
  const int M = dM.d, nb = n / R, step = n / L, st = M * LP;
  for (int t = threadIdx.x; t < tiles * nb * kDirLines; t += blockDim.x) {
    const int l = t & (kDirLines - 1);
    int b = t / kDirLines;
    float2* z = Z;
    if (tiles > 1) {
      const int tile = (int)((unsigned)b / (unsigned)nb);
      b -= tile * nb;
      z += tile * n * LP;
    }
    const int s = fdiv(b, dM), j = b - s * M;
    z += (s * L + j) * LP + l;
    const int jw = j * step;
    float2 v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      v[q] = z[q * st];
      if (INV && q > 0) v[q] = ctw<true>(v[q], tw[q * jw]);
    }
    if constexpr ((R & (R - 1)) == 0) Dft<R, INV>::run(v);
    else dft_odd<R, INV>(v, tw, n / R);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (!INV && q > 0) v[q] = ctw<false>(v[q], tw[q * jw]);
      z[q * st] = v[q];
    }
  }
}

// A radix without an unrolled butterfly (a prime above 13): one output per
// thread and turn, from Z to Z2.
template <bool INV, int LP>
__device__ void fft_pass_any(const float2* Z, float2* Z2, const float2* tw, int n, int R, int L, const FastDiv& dM) {
  const int M = dM.d, step = n / L, root = n / R;
  for (int t = threadIdx.x; t < n * kDirLines; t += blockDim.x) {
    const int l = t & (kDirLines - 1), e = t / kDirLines;
    const int qs = fdiv(e, dM), j = e - qs * M;  // e = (s R + q) M + j
    const int s = qs / R, q = qs - s * R;
    const float2* z = Z + (s * L + j) * LP + l;
    float2 acc = z[0];
    int idx = 0;
    for (int p = 1; p < R; ++p) {
      idx += q;
      if (idx >= R) idx -= R;
      float2 x = z[p * M * LP];
      if (INV) x = ctw<true>(x, tw[p * j * step]);
      const float2 y = ctw<INV>(x, tw[idx * root]);
      acc = cadd(acc, y);
    }
    if (!INV) acc = ctw<false>(acc, tw[q * j * step]);
    Z2[e * LP + l] = acc;
  }
}

// All passes of an axis on the tile in Z (forward: natural in, digit reversed
// out; inverse: the reverse). Returns the buffer that holds the result.
template <bool INV, int LP, bool POW2>
__device__ __forceinline__ float2* fft_tile(float2* Z, float2* Z2, const float2* tw, const AxisPlan& A, int tiles = 1) {
  for (int p = 0; p < A.npass; ++p) {
    const int q = INV ? A.npass - 1 - p : p;
    const int R = A.R[q], L = A.L[q];
    const FastDiv dM = A.dM[q];
    switch (R) {
      case 2: fft_pass<2, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
      case 4: fft_pass<4, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
      case 8: fft_pass<8, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
      case 16: fft_pass<16, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
      default:
        if constexpr (!POW2) {
          switch (R) {
            case 3: fft_pass<3, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
            case 5: fft_pass<5, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
            case 7: fft_pass<7, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
            case 11: fft_pass<11, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
            case 13: fft_pass<13, INV, LP>(Z, tw, A.n, L, dM, tiles); break;
            default: {
              fft_pass_any<INV, LP>(Z, Z2, tw, A.n, R, L, dM);
              float2* t = Z;
              Z = Z2;
              Z2 = t;
            }
          }
        }
    }
    __syncthreads();
  }
  return Z;
}

// Global to shared memory without a register in between, so that a thread has
// its whole share of the tile in flight at once.
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(BYTES)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void load_tw(float2* tw, const AxisPlan& A) {
  for (int m = threadIdx.x; m < A.n; m += blockDim.x) tw[m] = __ldg(A.tw + m);
}

// Rows 2q and 2q + 1 as real and imaginary part; scale applied in FP64 to FP64 input.
template <class T>
__device__ __forceinline__ float scaled(T v, double scale) {
  if constexpr (sizeof(T) == 8) return (float)(v * scale);
  else return v;
}

// The spectra A, B of the two rows packed in line l of a tile, at column c:
// A = (Z_f + conj Z_-f) / 2, B = (Z_f - conj Z_-f) / 2i; column 0 holds the mean and,
// for an even n, the Nyquist coefficient. And back: Z_f = A + i B, Z_-f = conj A + i conj B.
__device__ __forceinline__ void rows_from_line(const DirectArgs& a, const float2* Z, int l, int c, float2& A, float2& B) {
  const int2 at = __ldg(a.col + c);
  if (c == 0) {
    const float2 z0 = Z[l];
    const float2 zh = a.packed ? Z[at.y * kLpX + l] : make_float2(0.f, 0.f);
    A = make_float2(z0.x, zh.x);
    B = make_float2(z0.y, zh.y);
  } else {
    const float2 p = Z[at.x * kLpX + l], m = Z[at.y * kLpX + l];
    A = make_float2(0.5f * (p.x + m.x), 0.5f * (p.y - m.y));
    B = make_float2(0.5f * (p.y + m.y), 0.5f * (m.x - p.x));
  }
}
__device__ __forceinline__ void line_from_rows(const DirectArgs& a, float2* Z, int l, int c, float2 A, float2 B) {
  const int2 at = __ldg(a.col + c);
  if (c == 0) {
    Z[l] = make_float2(A.x, B.x);
    if (a.packed) Z[at.y * kLpX + l] = make_float2(A.y, B.y);
  } else {
    Z[at.x * kLpX + l] = make_float2(A.x - B.y, A.y + B.x);
    Z[at.y * kLpX + l] = make_float2(A.x + B.y, B.x - A.y);
  }
}

template <class T, bool POW2>
__global__ void __launch_bounds__(kFftThreads, 3) k_dir_xf(DirectArgs a, const T* __restrict__ in, const SolveCtl* c) {
  pdl_enter();
  if (c->stopped) return;
  extern __shared__ __align__(16) float2 sm[];
  const int n = a.nx;
  float2* tw = sm;
  float2* Z = sm + n;
  load_tw(tw, a.x);
  const long long row0 = 2ll * kDirLines * blockIdx.x;
  const double scale = sizeof(T) == 8 ? c->scale : 1.0;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int l = w; l < kDirLines; l += (int)blockDim.x / 32) {
    const long long r = row0 + 2 * l;
    const T* pa = in + r * n;
    const bool va = r < a.rows, vb = r + 1 < a.rows;
    if constexpr (sizeof(T) == 4) {
      if (vb) {
        for (int i = lane; i < n; i += 32) {
          copy_async<4>(&Z[i * kLpX + l].x, pa + i);
          copy_async<4>(&Z[i * kLpX + l].y, pa + n + i);
        }
        continue;
      }
    }
#pragma unroll 8
    for (int i = lane; i < n; i += 32)
      Z[i * kLpX + l] = make_float2(va ? scaled(pa[i], scale) : 0.f, vb ? scaled(pa[n + i], scale) : 0.f);
  }
  if constexpr (sizeof(T) == 4) copy_async_wait();
  __syncthreads();
  Z = fft_tile<false, kLpX, POW2>(Z, Z + n * kLpX, tw, a.x);
  float2* out = reinterpret_cast<float2*>(a.spec);
  for (int l = w; l < kDirLines; l += (int)blockDim.x / 32) {
    const long long r = row0 + 2 * l;
    if (r >= a.rows) break;
    const bool vb = r + 1 < a.rows;
    for (int f = lane; f < a.C; f += 32) {
      float2 A, B;
      rows_from_line(a, Z, l, f, A, B);
      out[r * a.C + f] = A;
      if (vb) out[(r + 1) * a.C + f] = B;
    }
  }
}

// Column 0 of an even nx carries the mean and the Nyquist coefficient of every
// row as one complex number: after (before) the y transform its frequencies g
// and -g are combined into the two coefficients' own spectra (and back).
template <bool INV>
__device__ __forceinline__ void split_packed(float2* Z, const AxisPlan& A) {
  for (int g = 1 + threadIdx.x; 2 * g < A.n; g += blockDim.x) {
    float2 &p = Z[__ldg(A.pos + g) * kLpY], &m = Z[__ldg(A.pos + A.n - g) * kLpY];
    const float2 u = p, v = m;
    if (!INV) {
      p = make_float2(0.5f * (u.x + v.x), 0.5f * (u.y - v.y));
      m = make_float2(0.5f * (u.y + v.y), 0.5f * (v.x - u.x));
    } else {  // p = u + i v, m = conj(u) + i conj(v)
      p = make_float2(u.x - v.y, u.y + v.x);
      m = make_float2(u.x + v.y, v.x - u.y);
    }
  }
}

template <bool INV, bool POW2>
__global__ void __launch_bounds__(kFftThreads, 3) k_dir_y(DirectArgs a, const SolveCtl* c) {
  pdl_enter();
  if (c->stopped) return;
  extern __shared__ __align__(16) float2 sm[];
  const int n = a.ny;
  float2* tw = sm;
  float2* Z = sm + n;
  load_tw(tw, a.y);
  const int col0 = blockIdx.x * kDirLines, l = threadIdx.x & (kDirLines - 1);
  const bool in = col0 + l < a.C;
  float2* g = reinterpret_cast<float2*>(a.spec) + (long long)blockIdx.y * n * a.C + col0 + l;
  for (int y = threadIdx.x / kDirLines; y < n; y += (int)blockDim.x / kDirLines) {
    if (in) copy_async<8>(&Z[y * kLpY + l], g + (long long)y * a.C);
    else Z[y * kLpY + l] = make_float2(0.f, 0.f);
  }
  copy_async_wait();
  __syncthreads();
  const bool split = a.packed && col0 == 0;
  if (INV && split) {
    split_packed<true>(Z, a.y);
    __syncthreads();
  }
  Z = fft_tile<INV, kLpY, POW2>(Z, Z + n * kLpY, tw, a.y);
  if (!INV && split) {
    split_packed<false>(Z, a.y);
    __syncthreads();
  }
  if (!in) return;
#pragma unroll 8
  for (int y = threadIdx.x / kDirLines; y < n; y += (int)blockDim.x / kDirLines) g[(long long)y * a.C] = Z[y * kLpY + l];
}

// What the last inverse transform does with d (already normalised): mixed,
// (hi, lo) += d renormalised; FP64, x += d / scale. Loads and stores are apart,
// so that a thread's loads are all in flight before its first store.
struct AddMixed {
  float *hi, *lo;
  double phi_c, dphi_dk;
  using Val = float2;
  __device__ __forceinline__ Val load(long long u) const { return make_float2(hi[u], lo[u]); }
  __device__ __forceinline__ void store(long long u, Val v, float d, double) const {
    float s, e;
    two_sum(v.x, d, s, e);
    e = __fadd_rn(e, v.y);
    const float h2 = __fadd_rn(s, e);
    hi[u] = h2;
    lo[u] = __fsub_rn(e, __fsub_rn(h2, s));
  }
  __device__ __forceinline__ void zero(long long u, int k) const {  // phi = 0: hi + lo = -vac
    const double v = -(phi_c + dphi_dk * (double)(k + 1));
    const float vh = (float)v;
    hi[u] = vh;
    lo[u] = (float)(v - (double)vh);
  }
};
struct Add64 {
  double* x;
  using Val = double;
  __device__ __forceinline__ Val load(long long u) const { return x[u]; }
  __device__ __forceinline__ void store(long long u, Val v, float d, double inv_scale) const {
    x[u] = v + (double)d * inv_scale;
  }
  __device__ __forceinline__ void zero(long long u, int) const { x[u] = 0.0; }
};

// Rows r and r + 1 (if vb) of the potential plus line l of a transformed tile.
template <class Add>
__device__ __forceinline__ void add_rows(const Add& add, const float2* Z, int l, long long r, bool vb, int n, int lane,
                                         float norm, double inv_scale) {
  constexpr int B = 4;  // points of both rows a thread loads before it stores any
  for (int i0 = lane; i0 < n; i0 += 32 * B) {
    typename Add::Val xa[B] = {}, xb[B] = {};
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const int i = i0 + 32 * q;
      if (i >= n) break;
      xa[q] = add.load(r * n + i);
      if (vb) xb[q] = add.load((r + 1) * n + i);
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const int i = i0 + 32 * q;
      if (i >= n) break;
      const float2 d = Z[i * kLpX + l];
      add.store(r * n + i, xa[q], d.x * norm, inv_scale);
      if (vb) add.store((r + 1) * n + i, xb[q], d.y * norm, inv_scale);
    }
  }
}

template <class Add, bool POW2>
__global__ void __launch_bounds__(kFftThreads, 3) k_dir_xi(DirectArgs a, Add add, const SolveCtl* c) {
  pdl_enter();
  const long long row0 = 2ll * kDirLines * blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = a.nx;
  if (c->stopped) {
    if (c->bb != 0.0) return;
    for (long long r = row0 + w; r < row0 + 2 * kDirLines && r < a.rows; r += (int)blockDim.x / 32)  // b = 0: x = 0
      for (int i = lane; i < n; i += 32) add.zero(r * n + i, (int)(r / a.ny));
    return;
  }
  extern __shared__ __align__(16) float2 sm[];
  float2* tw = sm;
  float2* Z = sm + n;
  load_tw(tw, a.x);
  const float2* spec = reinterpret_cast<const float2*>(a.spec);
  for (int l = w; l < kDirLines; l += (int)blockDim.x / 32) {
    const long long r = row0 + 2 * l;
    const bool va = r < a.rows, vb = r + 1 < a.rows;
#pragma unroll 4
    for (int f = lane; f < a.C; f += 32) {
      const float2 A = va ? spec[r * a.C + f] : make_float2(0.f, 0.f);
      const float2 B = vb ? spec[(r + 1) * a.C + f] : make_float2(0.f, 0.f);
      line_from_rows(a, Z, l, f, A, B);
    }
  }
  __syncthreads();
  Z = fft_tile<true, kLpX, POW2>(Z, Z + n * kLpX, tw, a.x);
  const double inv_scale = c->inv_scale;
  for (int l = w; l < kDirLines; l += (int)blockDim.x / 32) {
    const long long r = row0 + 2 * l;
    const bool va = r < a.rows, vb = r + 1 < a.rows;
    if (!va) break;
    add_rows(add, Z, l, r, vb, n, lane, a.norm, inv_scale);
  }
}

// Whole planes in one block, x and y transforms after one another in shared
// memory: two launches fewer per pass where a plane is small (measured with
// separate launches and fused, a whole pass of steps at 32x32x64: 3025 and 2948 us
// mixed, 4270 and 4053 FP64). Rows pair up within a plane, so ny is even.
template <class T, bool POW2>
__global__ void __launch_bounds__(kFftThreads, 3) k_dir_xyf(DirectArgs a, const T* __restrict__ in, const SolveCtl* c) {
  pdl_enter();
  if (c->stopped) return;
  extern __shared__ __align__(16) float2 sm[];
  const int n = a.nx, m = a.ny, pairs = m / 2, tx = (pairs + kDirLines - 1) / kDirLines;
  const int ty = (a.C + kDirLines - 1) / kDirLines;
  float2 *twx = sm, *twy = sm + n, *Z = twy + m, *S = Z + tx * n * kLpX;
  load_tw(twx, a.x);
  load_tw(twy, a.y);
  const double scale = sizeof(T) == 8 ? c->scale : 1.0;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const T* plane = in + (long long)blockIdx.x * n * m;
  for (int q = w; q < tx * kDirLines; q += nw) {
    const T* pa = plane + (long long)(2 * q) * n;
    float2* z = Z + (q / kDirLines) * n * kLpX + (q & (kDirLines - 1));
    const bool v = q < pairs;
#pragma unroll 4
    for (int i = lane; i < n; i += 32) z[i * kLpX] = v ? make_float2(scaled(pa[i], scale), scaled(pa[n + i], scale)) : make_float2(0.f, 0.f);
  }
  __syncthreads();
  fft_tile<false, kLpX, POW2>(Z, nullptr, twx, a.x, tx);
  for (int q = w; q < pairs; q += nw)
    for (int f = lane; f < ty * kDirLines; f += 32) {
      float2 A = make_float2(0.f, 0.f), B = A;
      if (f < a.C) rows_from_line(a, Z + (q / kDirLines) * n * kLpX, q & (kDirLines - 1), f, A, B);
      float2* o = S + ((f / kDirLines) * m + 2 * q) * kLpY + (f & (kDirLines - 1));
      o[0] = A;
      o[kLpY] = B;
    }
  __syncthreads();
  fft_tile<false, kLpY, POW2>(S, nullptr, twy, a.y, ty);
  if (a.packed) {
    split_packed<false>(S, a.y);
    __syncthreads();
  }
  float2* out = reinterpret_cast<float2*>(a.spec) + (long long)blockIdx.x * m * a.C;
  for (int u = threadIdx.x; u < m * a.C; u += blockDim.x) {
    const int y = (int)((unsigned)u / (unsigned)a.C), f = u - y * a.C;
    out[u] = S[((f / kDirLines) * m + y) * kLpY + (f & (kDirLines - 1))];
  }
}

template <class Add, bool POW2>
__global__ void __launch_bounds__(kFftThreads, 3) k_dir_xyi(DirectArgs a, Add add, const SolveCtl* c) {
  pdl_enter();
  const int n = a.nx, m = a.ny, pairs = m / 2, tx = (pairs + kDirLines - 1) / kDirLines;
  const int ty = (a.C + kDirLines - 1) / kDirLines;
  if (c->stopped) {
    if (c->bb != 0.0) return;
    for (int u = threadIdx.x; u < n * m; u += blockDim.x) add.zero((long long)blockIdx.x * n * m + u, blockIdx.x);  // b = 0: x = 0
    return;
  }
  extern __shared__ __align__(16) float2 sm[];
  float2 *twx = sm, *twy = sm + n, *Z = twy + m, *S = Z + tx * n * kLpX;
  load_tw(twx, a.x);
  load_tw(twy, a.y);
  const float2* spec = reinterpret_cast<const float2*>(a.spec) + (long long)blockIdx.x * m * a.C;
#pragma unroll 4
  for (int u = threadIdx.x; u < m * a.C; u += blockDim.x) {
    const int y = (int)((unsigned)u / (unsigned)a.C), f = u - y * a.C;
    S[((f / kDirLines) * m + y) * kLpY + (f & (kDirLines - 1))] = spec[u];
  }
  __syncthreads();
  if (a.packed) {
    split_packed<true>(S, a.y);
    __syncthreads();
  }
  fft_tile<true, kLpY, POW2>(S, nullptr, twy, a.y, ty);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int q = w; q < pairs; q += nw)
    for (int f = lane; f < a.C; f += 32) {
      const float2* o = S + ((f / kDirLines) * m + 2 * q) * kLpY + (f & (kDirLines - 1));
      line_from_rows(a, Z + (q / kDirLines) * n * kLpX, q & (kDirLines - 1), f, o[0], o[kLpY]);
    }
  __syncthreads();
  fft_tile<true, kLpX, POW2>(Z, nullptr, twx, a.x, tx);
  const double inv_scale = c->inv_scale;
  for (int q = w; q < pairs; q += nw)
    add_rows(add, Z + (q / kDirLines) * n * kLpX, q & (kDirLines - 1), (long long)blockIdx.x * m + 2 * q, true, n, lane, a.norm,
             inv_scale);
}

// Tridiagonal systems (2 + lambda) u_k - u_(k-1) - u_(k+1) = f_k, zero beyond
// both ends, one per float column of the spectrum (lane = column). Warp w of the
// block takes planes [w M, (w + 1) M): it eliminates its chunk with zero outer
// neighbours (pivots 1 / (2 + lambda - pivot), the same for every chunk, formed
// as 1 / (1 + s), s = lambda + s pivot, which does not cancel for small lambda);
// the chunks' first and last values then satisfy a recurrence that warp 0 solves
// along the chunks, and each warp adds the response to its two outer neighbours.
// Planes stay in registers in between, so the spectrum is read and written once.
template <int M, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS) k_dir_z(DirectArgs a, const SolveCtl* c) {
  pdl_enter();
  if (c->stopped) return;
  extern __shared__ float zs[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  float* sF = zs + lane;         // [W][32] first value of the chunk
  float* sE = sF + 32 * W;       // last value with zero neighbours, then the left neighbour's value
  float* sD = sE + 32 * W;       // response of the first value to the right neighbour
  float* sV = sD + 32 * W;
  float* sC = sV + 32 * W;       // [M][32] the pivots and, after them, their product
  const int col = blockIdx.x * 32 + lane;
  const bool in = col < a.plane;
  const int k0 = w * M, len = min(M, a.P - k0);
  float* g = a.spec + (long long)k0 * a.plane + col;
  float y[M];
  // reloaded at each use: registers then hold the planes alone
  auto cp = [&](int k) -> float { return *(volatile float*)(sC + 32 * k); };
#pragma unroll
  for (int k = 0; k < M; ++k) y[k] = in && k < len ? g[(long long)k * a.plane] : 0.f;
  if (w == 0) {
    const float lam = in ? __ldg(a.lam + col) : 1.f;
    float s = lam + 1.f, b = 1.f;
    for (int k = 0; k < M; ++k) {
      const float v = 1.f / (1.f + s);
      sC[32 * k] = v;
      s = fmaf(s, v, lam);
      b *= v;
    }
    sC[32 * M] = b;
  }
  __syncthreads();
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    t = cp(k) * (y[k] + t);
    y[k] = k < len ? t : 0.f;
  }
  sE[32 * w] = y[M - 1];
  t = 0.f;
#pragma unroll
  for (int k = M - 1; k >= 0; --k) t = fmaf(cp(k), t, y[k]);
  sF[32 * w] = t;
  __syncthreads();
  if (w == 0) {
    // F = pF + a L + b R, E = pE + b L + a R per chunk (a, b: responses at the near
    // and the far end), L the left chunk's E, R the right chunk's F. With
    // L = u + v F: F = (pF + a u + b R) / (1 - a v), and u, v of the next chunk.
    const int last = a.P - (W - 1) * M;  // planes of the last chunk
    const float alast = cp(last - 1), afull = cp(M - 1), b = cp(M);
    float u = 0.f, v = 0.f;
    for (int q = 0; q < W; ++q) {
      const float aq = q == W - 1 ? alast : afull, bq = q == W - 1 ? 0.f : b;
      const float inv = 1.f / fmaf(-aq, v, 1.f);
      const float F = fmaf(aq, u, sF[32 * q]) * inv, D = bq * inv, pE = sE[32 * q];
      sF[32 * q] = F;
      sD[32 * q] = D;
      sE[32 * q] = u;
      sV[32 * q] = v;
      u = fmaf(bq, fmaf(v, F, u), pE);
      v = fmaf(bq * v, D, aq);
    }
    float R = 0.f;
    for (int q = W - 1; q >= 0; --q) {
      R = fmaf(sD[32 * q], R, sF[32 * q]);
      sF[32 * q] = R;
      sE[32 * q] = fmaf(sV[32 * q], R, sE[32 * q]);
    }
  }
  __syncthreads();
  t = sE[32 * w];  // the left neighbour's value (0 for the first chunk)
  const float right = w + 1 < W ? sF[32 * (w + 1)] : 0.f;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    t *= cp(k);
    y[k] += t;
  }
  y[M - 1] = fmaf(cp(M - 1), right, y[M - 1]);
  t = 0.f;
#pragma unroll
  for (int k = M - 1; k >= 0; --k) {
    t = k < len ? fmaf(cp(k), t, y[k]) : 0.f;
    if (in && k < len) g[(long long)k * a.plane] = t;
  }
}

// ---------------------------------------------------------------------------
// residuals of the refinement
// ---------------------------------------------------------------------------
// Two grid-wide sums at once (as grid_total; partials interleaved).
template <class V>
__device__ __forceinline__ bool grid_total2(V v0, V v1, double* part, unsigned* ticket, double* t0, double* t1) {
  __shared__ double sm0[32], sm1[32];
  __shared__ int s_last;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int nthr = blockDim.x * blockDim.y, nw = nthr >> 5;
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  v0 = warp_sum(v0);
  v1 = warp_sum(v1);
  if ((tid & 31) == 0) {
    sm0[tid >> 5] = (double)v0;
    sm1[tid >> 5] = (double)v1;
  }
  __syncthreads();
  if (tid == 0) {
    double a = 0.0, b = 0.0;
    for (int k = 0; k < nw; ++k) {
      a += sm0[k];
      b += sm1[k];
    }
    const unsigned at = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    reinterpret_cast<double2*>(part)[at] = make_double2(a, b);
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == nb - 1u ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  double a = 0.0, b = 0.0;
#pragma unroll 4
  for (unsigned i = tid; i < nb; i += nthr) {
    const double2 p = __ldcg(reinterpret_cast<const double2*>(part) + i);
    a += p.x;
    b += p.y;
  }
  a = warp_sum(a);
  b = warp_sum(b);
  __syncthreads();
  if ((tid & 31) == 0) {
    sm0[tid >> 5] = a;
    sm1[tid >> 5] = b;
  }
  __syncthreads();
  if (tid != 0) return false;
  a = b = 0.0;
  for (int k = 0; k < nw; ++k) {
    a += sm0[k];
    b += sm1[k];
  }
  *t0 = a;
  *t1 = b;
  *ticket = 0u;
  return true;
}

// The refinement's decision from r.r: another pass or stop; the power of two
// that brings r to unit size for the FP32 pass of an FP64 residual, from the
// exponents alone, and no relative residual (the host forms it): two square roots
// and two divisions by one thread were on every solve's critical path (1.1 us a residual).
__device__ __forceinline__ void fin_pass(const DirectLoop& d, SolveCtl* c, double rr, long long n) {
  c->rr_true = rr;
  const bool small = c->bb == 0.0 || rr <= c->tol2;
  bool enough = small;
  if (d.margin2 < 1.0 && small && c->it_total > 0 && !c->margin_used && rr > d.margin2 * c->tol2 && c->tol2 > c->floor2) {
    c->margin_used = 1;
    enough = false;
  }
  const bool done = enough || !(rr == rr) || c->it_total >= d.maxit || c->outer >= d.max_outer;
  c->converged = small ? 1 : 0;
  c->more = done ? 0 : 1;
  c->stopped = done ? 1 : 0;
  const int ex = rr > 0.0 && rr < INFINITY ? max(-900, min(900, (ilogb((double)n) - ilogb(rr)) >> 1)) : 0;
  c->scale = scalbn(1.0, ex);
  c->inv_scale = scalbn(1.0, -ex);
  if (d.use_graph) cudaGraphSetConditional(d.handle, done ? 0u : 1u);
}
// first: the solve begins (b.b sets the tolerance); later: one pass has run
__device__ __forceinline__ void fin_first(const DirectLoop& d, SolveCtl* c, double rr, double bb, long long n) {
  c->bb = bb;
  c->tol2 = d.rtol * d.rtol * bb;
  c->maxit = d.maxit;
  c->it_total = 0;
  c->outer = 0;
  fin_pass(d, c, rr, n);
}
__device__ __forceinline__ void fin_next(const DirectLoop& d, SolveCtl* c, double rr, long long n) {
  c->it_total += 1;
  c->outer += 1;
  fin_pass(d, c, rr, n);
}

template <class T, int V>
struct VecOf;
template <>
struct VecOf<float, 1> {
  using type = float;
};
template <>
struct VecOf<float, 4> {
  using type = float4;
};
template <>
struct VecOf<double, 1> {
  using type = double;
};
template <>
struct VecOf<double, 2> {
  using type = double2;
};
template <int V, class T>
__device__ __forceinline__ void vload(T (&v)[V], const T* p) {
  using U = typename VecOf<T, V>::type;
  const U u = *reinterpret_cast<const U*>(p);
#pragma unroll
  for (int e = 0; e < V; ++e) v[e] = reinterpret_cast<const T*>(&u)[e];
}
template <int V, class T>
__device__ __forceinline__ void vstore(T* p, const T (&v)[V]) {
  using U = typename VecOf<T, V>::type;
  U u;
#pragma unroll
  for (int e = 0; e < V; ++e) reinterpret_cast<T*>(&u)[e] = v[e];
  *reinterpret_cast<U*>(p) = u;
}

// The residual kernels give a thread V neighbouring points of a row and march it
// through kc planes: a plane is loaded once as the upper neighbour and kept in
// registers as the centre and the lower one, so a point costs one load of its
// own plane instead of three.
constexpr int kResThreads = 256;  // 8, 16 or 32 lanes along x, the rest along y
struct ResGeom {
  Lv L;
  int kc;         // planes per block
  long long n;    // unknowns
};

// r = fl32(f - A (hi + lo)) in float-float (the transformations of the header
// comment of the MIXED solver), r.r and, FIRST, b.b with the folded electrode
// terms. V = 4 where rows are whole float4s.
template <int V, bool FIRST>
__global__ void __launch_bounds__(kResThreads) k_dir_resid_ff(ResGeom G, const float* __restrict__ hi,
                                                              const float* __restrict__ lo, const float* __restrict__ f,
                                                              float* __restrict__ r, float fold_first, float fold_last,
                                                              double* part, SolveCtl* c, DirectLoop d) {
  pdl_enter();
  if (!FIRST && c->stopped) return;
  const Lv& L = G.L;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) * V, j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = blockIdx.z * G.kc, kend = min(k0 + G.kc, L.nz - 1);
  float rr = 0.f, bb = 0.f;
  if (i < L.nx && j < L.ny) {
    const int row = j * L.nx;
    const int left = row + (i == 0 ? L.nx - 1 : i - 1), right = row + (i + V == L.nx ? 0 : i + V);
    const int down = (j == 0 ? L.ny - 1 : j - 1) * L.nx + i, up = (j == L.ny - 1 ? 0 : j + 1) * L.nx + i;
    const long long at0 = (long long)k0 * L.pl;
    float hm[V] = {}, hc[V], hp[V], lm[V] = {}, lc[V], lp[V];
    vload<V>(hc, hi + at0 + row + i);
    vload<V>(lc, lo + at0 + row + i);
    if (k0 > 0) {
      vload<V>(hm, hi + at0 - L.pl + row + i);
      vload<V>(lm, lo + at0 - L.pl + row + i);
    }
    for (int k = k0; k < kend; ++k) {
      const float *H = hi + (long long)k * L.pl, *O = lo + (long long)k * L.pl;
      float hy0[V], hy1[V], ly0[V], ly1[V], fv[V], rv[V];
      if (k < L.nz - 2) {
        vload<V>(hp, H + L.pl + row + i);
        vload<V>(lp, O + L.pl + row + i);
      } else {
#pragma unroll
        for (int e = 0; e < V; ++e) hp[e] = lp[e] = 0.f;
      }
      vload<V>(hy0, H + down);
      vload<V>(hy1, H + up);
      vload<V>(ly0, O + down);
      vload<V>(ly1, O + up);
      vload<V>(fv, f + (long long)k * L.pl + row + i);
      const float hl = H[left], hr = H[right], ol = O[left], orr = O[right];
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const float xl = e == 0 ? hl : hc[e > 0 ? e - 1 : 0], xr = e == V - 1 ? hr : hc[e < V - 1 ? e + 1 : 0];
        float s = xl, er = 0.f, t;
        two_sum(s, xr, s, t);
        er = __fadd_rn(er, t);
        two_sum(s, hy0[e], s, t);
        er = __fadd_rn(er, t);
        two_sum(s, hy1[e], s, t);
        er = __fadd_rn(er, t);
        two_sum(s, hm[e], s, t);
        er = __fadd_rn(er, t);
        two_sum(s, hp[e], s, t);
        er = __fadd_rn(er, t);
        const float p6 = __fmul_rn(6.f, hc[e]), e6 = __fmaf_rn(6.f, hc[e], -p6);
        float a1, ea, r1, e1;
        two_sum(p6, -s, a1, ea);
        const float zl = e == 0 ? ol : lc[e > 0 ? e - 1 : 0], zr = e == V - 1 ? orr : lc[e < V - 1 ? e + 1 : 0];
        const float nl = ((((zl + zr) + ly0[e]) + ly1[e]) + lm[e]) + lp[e];
        const float alo = __fsub_rn(__fmul_rn(6.f, lc[e]), nl);
        two_sum(fv[e], -a1, r1, e1);
        rv[e] = __fadd_rn(r1, __fsub_rn(__fadd_rn(__fsub_rn(__fsub_rn(e1, ea), e6), er), alo));
        rr += rv[e] * rv[e];
        if (FIRST) {
          float bv = fv[e];
          if (k == 0) bv += fold_first;
          if (k == L.nz - 2) bv += fold_last;
          bb += bv * bv;
        }
      }
      vstore<V>(r + (long long)k * L.pl + row + i, rv);
#pragma unroll
      for (int e = 0; e < V; ++e) {
        hm[e] = hc[e];
        hc[e] = hp[e];
        lm[e] = lc[e];
        lc[e] = lp[e];
      }
    }
  }
  double t0, t1;
  if constexpr (FIRST) {
    if (grid_total2(rr, bb, part, &c->ticket, &t0, &t1)) fin_first(d, c, t0, t1, G.n);
  } else {
    if (grid_total(rr, part, &c->ticket, &t0)) fin_next(d, c, t0, G.n);
  }
}

// r = b - A x in FP64, r.r and, FIRST, b.b
template <int V, bool FIRST>
__global__ void __launch_bounds__(kResThreads) k_dir_resid64(ResGeom G, const double* __restrict__ x,
                                                             const double* __restrict__ b, double* __restrict__ r,
                                                             double* part, SolveCtl* c, DirectLoop d) {
  pdl_enter();
  if (!FIRST && c->stopped) return;
  const Lv& L = G.L;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) * V, j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = blockIdx.z * G.kc, kend = min(k0 + G.kc, L.nz - 1);
  double rr = 0.0, bb = 0.0;
  if (i < L.nx && j < L.ny) {
    const int row = j * L.nx;
    const int left = row + (i == 0 ? L.nx - 1 : i - 1), right = row + (i + V == L.nx ? 0 : i + V);
    const int down = (j == 0 ? L.ny - 1 : j - 1) * L.nx + i, up = (j == L.ny - 1 ? 0 : j + 1) * L.nx + i;
    double xm[V] = {}, xc[V], xp[V];
    vload<V>(xc, x + (long long)k0 * L.pl + row + i);
    if (k0 > 0) vload<V>(xm, x + (long long)(k0 - 1) * L.pl + row + i);
    for (int k = k0; k < kend; ++k) {
      const double* X = x + (long long)k * L.pl;
      double y0[V], y1[V], bv[V], rv[V];
      if (k < L.nz - 2) {
        vload<V>(xp, X + L.pl + row + i);
      } else {
#pragma unroll
        for (int e = 0; e < V; ++e) xp[e] = 0.0;
      }
      vload<V>(y0, X + down);
      vload<V>(y1, X + up);
      vload<V>(bv, b + (long long)k * L.pl + row + i);
      const double xl0 = X[left], xr0 = X[right];
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const double xl = e == 0 ? xl0 : xc[e > 0 ? e - 1 : 0], xr = e == V - 1 ? xr0 : xc[e < V - 1 ? e + 1 : 0];
        const double s = ((((xl + xr) + y0[e]) + y1[e]) + xm[e]) + xp[e];
        rv[e] = bv[e] - (6.0 * xc[e] - s);
        rr += rv[e] * rv[e];
        if (FIRST) bb += bv[e] * bv[e];
        xm[e] = xc[e];
      }
#pragma unroll
      for (int e = 0; e < V; ++e) xc[e] = xp[e];
      vstore<V>(r + (long long)k * L.pl + row + i, rv);
    }
  }
  double t0, t1;
  if constexpr (FIRST) {
    if (grid_total2(rr, bb, part, &c->ticket, &t0, &t1)) fin_first(d, c, t0, t1, G.n);
  } else {
    if (grid_total(rr, part, &c->ticket, &t0)) fin_next(d, c, t0, G.n);
  }
}

// radices of n points, powers of two first; false where a factor or the count is out of range
bool axis_plan(int n, AxisPlan& A) {
  A.n = n;
  A.npass = 0;
  A.pow2 = 1;
  A.pingpong = 0;
  std::vector<int> R;
  int m = n, p2 = 0;
  while (m % 2 == 0) {
    m /= 2;
    ++p2;
  }
  while (p2 > 0) {  // 16 x 8, 8 x 8, 8 x 4 ...: as few passes as radices up to 16 allow, evenly
    const int passes = (p2 + 3) / 4, b = (p2 + passes - 1) / passes;
    R.push_back(1 << b);
    p2 -= b;
  }
  for (int p = 3; m > 1; p += 2)
    while (m % p == 0) {
      R.push_back(p);
      m /= p;
      A.pow2 = 0;
      if (p > 13) A.pingpong = 1;
    }
  if ((int)R.size() > kDirMaxPasses) return false;
  int L = n;
  for (int r : R) {
    A.R[A.npass] = r;
    A.L[A.npass] = L;
    A.dM[A.npass] = make_fastdiv(L / r);
    ++A.npass;
    L /= r;
  }
  return true;
}

// frequency that the forward passes leave at position p
__device__ __forceinline__ int axis_freq(const AxisPlan& A, int p) {
  int freq = 0, mul = 1;
  for (int q = 0; q < A.npass; ++q) {
    const int M = A.dM[q].d, d = fdiv(p, A.dM[q]);
    freq += mul * d;
    p -= d * M;
    mul *= A.R[q];
  }
  return freq;
}
__device__ __forceinline__ double axis_lambda(int n, int f) {  // 2 - 2 cos(2 pi f / n), without cancellation
  const double s = sinpi((double)f / n);
  return 4.0 * s * s;
}

// Twiddles, positions, columns and eigenvalues of a plan, formed in FP64 and
// rounded once. Columns of x (frequencies 0..C - 1) are ordered by position: the
// lanes that gather (k_dir_xf) or scatter (k_dir_xi) them then walk runs of
// neighbouring rows of the tile, where frequency order jumps by a whole radix
// and meets the same bank 8 (128 points) or 16 times (256).
__global__ void k_dir_tables(DirectArgs a) {
  const int t = (int)gtid(), n = (int)gstride();
  extern __shared__ int sh[];  // frequency of every position of x, its inverse, frequency of every column
  int *freqx = sh, *posx = sh + a.nx, *colf = posx + a.nx;
  for (int p = threadIdx.x; p < a.nx; p += blockDim.x) {
    const int f = axis_freq(a.x, p);
    freqx[p] = f;
    posx[f] = p;
  }
  __syncthreads();
  for (int p = threadIdx.x; p < a.nx; p += blockDim.x) {
    if (freqx[p] >= a.C) continue;
    int c = 0;
    for (int q = 0; q < p; ++q) c += freqx[q] < a.C ? 1 : 0;
    colf[c] = freqx[p];
  }
  __syncthreads();
#pragma unroll
  for (int axis = 0; axis < 2; ++axis) {
    const AxisPlan& A = axis == 0 ? a.x : a.y;
    for (int m = t; m < A.n; m += n) {
      double s, c;
      sincospi(2.0 * m / A.n, &s, &c);
      const_cast<float2*>(A.tw)[m] = make_float2((float)c, (float)-s);
      const_cast<int*>(A.pos)[axis_freq(A, m)] = m;
    }
  }
  for (int c = t; c < a.C; c += n) {
    const int f = colf[c];
    const_cast<int2*>(a.col)[c] = make_int2(posx[f], posx[f > 0 ? a.nx - f : (a.packed ? a.nx / 2 : 0)]);
  }
  for (int u = t; u < a.plane / 2; u += n) {
    const int p = u / a.C, q = colf[u - p * a.C];
    const int g = axis_freq(a.y, p);
    const double ly = axis_lambda(a.ny, g);
    double l0 = axis_lambda(a.nx, q), l1 = l0;
    if (q == 0 && a.packed) {
      if (g == 0 || 2 * g == a.ny) l1 = 4.0;  // mean and Nyquist coefficient, both real
      else if (2 * g > a.ny) l0 = l1 = 4.0;   // the Nyquist coefficient's spectrum
    }
    float* lam = const_cast<float*>(a.lam);
    lam[2 * u] = (float)(l0 + ly);
    lam[2 * u + 1] = (float)(l1 + ly);
  }
}

size_t fft_smem(const AxisPlan& A, int lp) {
  return sizeof(float2) * ((size_t)A.n + (size_t)A.n * lp * (A.pingpong ? 2 : 1));
}

constexpr size_t kMaxSmem = 227 * 1024;
constexpr size_t kPlaneSmem = 16 * 1024;  // planes of about 32 x 32 points (64 x 64 measured no faster, slower in ensembles)

template <class K>
cudaError_t allow_smem(K k) {
  // the attribute is the kernel's, shared by every solver of the process
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
}

}  // namespace

bool DirectSolver::plan(int nx, int ny, int nz) {
  const int P = nz - 1;
  // planes: 32 warps of 32 (the tridiagonal kernel's block); lines: what fits in shared memory
  if (P < 1 || P > 1024 || !axis_plan(nx, a.x) || !axis_plan(ny, a.y)) return false;
  smem_x = fft_smem(a.x, kLpX);
  smem_y = fft_smem(a.y, kLpY);
  if (smem_x > kMaxSmem || smem_y > kMaxSmem) return false;
  a.nx = nx;
  a.ny = ny;
  a.P = P;
  a.packed = nx % 2 == 0;
  a.C = a.packed ? nx / 2 : (nx + 1) / 2;
  a.plane = 2 * a.C * ny;
  a.rows = (long long)ny * P;
  a.norm = (float)(1.0 / ((double)nx * ny));
  // a whole plane in one block
  const int tx = (ny / 2 + kDirLines - 1) / kDirLines, ty = (a.C + kDirLines - 1) / kDirLines;
  smem_xy = sizeof(float2) * ((size_t)nx + ny + (size_t)tx * nx * kLpX + (size_t)ty * ny * kLpY);
  planes = ny % 2 == 0 && !a.x.pingpong && !a.y.pingpong && smem_xy <= kPlaneSmem;
  zm = P <= 256 ? 16 : 32;
  zw = (P + zm - 1) / zm;
  return true;
}

size_t DirectSolver::table_bytes() const {
  return (sizeof(float2) + sizeof(int)) * (size_t)(a.nx + a.ny) + 8 + sizeof(int2) * (size_t)a.C +
         sizeof(float) * (size_t)a.plane;
}
size_t DirectSolver::spec_bytes() const { return sizeof(float) * (size_t)a.plane * a.P; }

cudaError_t DirectSolver::place(void* tables_mem, void* spec_mem, cudaStream_t s) {
  char* t = (char*)tables_mem;
  a.x.tw = (const float2*)t;
  a.y.tw = a.x.tw + a.nx;
  a.x.pos = (const int*)(a.y.tw + a.ny);
  a.y.pos = a.x.pos + a.nx;
  a.col = (const int2*)(t + (sizeof(float2) * (a.nx + a.ny) + sizeof(int) * (a.nx + a.ny) + 7) / 8 * 8);
  a.lam = (const float*)(a.col + a.C);
  a.spec = (float*)spec_mem;
  cudaError_t e;
  if ((e = allow_smem(k_dir_xf<float, true>)) || (e = allow_smem(k_dir_xf<float, false>)) ||
      (e = allow_smem(k_dir_xf<double, true>)) || (e = allow_smem(k_dir_xf<double, false>)) ||
      (e = allow_smem(k_dir_y<false, true>)) || (e = allow_smem(k_dir_y<false, false>)) ||
      (e = allow_smem(k_dir_y<true, true>)) || (e = allow_smem(k_dir_y<true, false>)) ||
      (e = allow_smem(k_dir_xi<AddMixed, true>)) || (e = allow_smem(k_dir_xi<AddMixed, false>)) ||
      (e = allow_smem(k_dir_xi<Add64, true>)) || (e = allow_smem(k_dir_xi<Add64, false>)))
    return e;
  const int n = std::max(std::max(a.nx, a.ny), a.plane / 2);
  PIC_LAUNCH(std::min((n + 127) / 128, 1024), 128, sizeof(int) * (2 * a.nx + a.C), s, k_dir_tables)(a);
  return cudaGetLastError();
}

cudaError_t DirectSolver::init(int nx, int ny, int nz) {
  on = false;
  if (!plan(nx, ny, nz)) return cudaSuccess;
  cudaError_t e;
  if ((e = dev_malloc(&tables, table_bytes()))) return e;
  if ((e = dev_malloc((void**)&a.spec, spec_bytes()))) return e;
  if ((e = place(tables, a.spec, cudaStreamLegacy))) return e;
  if ((e = cudaStreamSynchronize(cudaStreamLegacy))) return e;
  on = true;
  return cudaSuccess;
}

void DirectSolver::release() {
  dev_free(tables);
  dev_free(a.spec);
  tables = nullptr;
  a.spec = nullptr;
  on = false;
}

namespace {

template <class T, class Add>
void apply(const DirectSolver& D, const T* r, const Add& add, const SolveCtl* c, cudaStream_t s) {
  const DirectArgs& a = D.a;
  const dim3 gx((unsigned)((a.rows + 2 * kDirLines - 1) / (2 * kDirLines)));
  const dim3 gy((a.C + kDirLines - 1) / kDirLines, a.P);
  const dim3 gz((a.plane + 31) / 32);
  const int tx = a.nx > 128 ? kFftThreads : kFftThreads / 2, ty = kFftThreads / 2;
  const size_t zsm = sizeof(float) * 32 * (4 * D.zw + D.zm + 1);
  const auto z = [&]() {
    if (D.zm == 16) SOLVER_LAUNCH(gz, 32 * D.zw, zsm, s, k_dir_z<16, 512, 3>)(a, c);
    else if (D.zw <= 16) SOLVER_LAUNCH(gz, 32 * D.zw, zsm, s, k_dir_z<32, 512, 2>)(a, c);
    else SOLVER_LAUNCH(gz, 32 * D.zw, zsm, s, k_dir_z<32, 1024, 1>)(a, c);
  };
  if (D.planes) {
    const bool pow2 = a.x.pow2 && a.y.pow2;
    if (pow2) SOLVER_LAUNCH(a.P, kFftThreads, D.smem_xy, s, k_dir_xyf<T, true>)(a, r, c);
    else SOLVER_LAUNCH(a.P, kFftThreads, D.smem_xy, s, k_dir_xyf<T, false>)(a, r, c);
    z();
    if (pow2) SOLVER_LAUNCH(a.P, kFftThreads, D.smem_xy, s, k_dir_xyi<Add, true>)(a, add, c);
    else SOLVER_LAUNCH(a.P, kFftThreads, D.smem_xy, s, k_dir_xyi<Add, false>)(a, add, c);
    return;
  }
  if (a.x.pow2) SOLVER_LAUNCH(gx, tx, D.smem_x, s, k_dir_xf<T, true>)(a, r, c);
  else SOLVER_LAUNCH(gx, tx, D.smem_x, s, k_dir_xf<T, false>)(a, r, c);
  if (a.y.pow2) SOLVER_LAUNCH(gy, ty, D.smem_y, s, k_dir_y<false, true>)(a, c);
  else SOLVER_LAUNCH(gy, ty, D.smem_y, s, k_dir_y<false, false>)(a, c);
  z();
  if (a.y.pow2) SOLVER_LAUNCH(gy, ty, D.smem_y, s, k_dir_y<true, true>)(a, c);
  else SOLVER_LAUNCH(gy, ty, D.smem_y, s, k_dir_y<true, false>)(a, c);
  if (a.x.pow2) SOLVER_LAUNCH(gx, tx, D.smem_x, s, k_dir_xi<Add, true>)(a, add, c);
  else SOLVER_LAUNCH(gx, tx, D.smem_x, s, k_dir_xi<Add, false>)(a, add, c);
}

// points per thread: a vector of a row, or one where vectors would leave SMs without a block
int res_vec(const MgLevel& M, int V, bool aligned) {
  return aligned && M.nu >= 2ll * sm_count() * kResThreads * V ? V : 1;
}

// block shape and planes per block of the residual kernels: a few blocks per SM,
// at most 8 planes (longer marches save little: 1 + 2 / kc plane loads per point)
ResGeom res_geom(const MgLevel& M, int V, dim3* grid, dim3* block) {
  ResGeom G{lv_of(M), 1, M.nu};
  const int P = M.nz - 1, vx = M.nx / V;
  const unsigned bx = vx <= 8 ? 8 : (vx <= 16 ? 16 : 32), by = kResThreads / bx;
  const unsigned gx = (vx + bx - 1) / bx, gy = (M.ny + by - 1) / by;
  int kc = 8;
  while (kc > 1 && (long long)gx * gy * ((P + kc - 1) / kc) < 6ll * sm_count()) kc >>= 1;
  // the partial sums of a block are a double2 each
  while ((long long)gx * gy * ((P + kc - 1) / kc) > kDirParts) kc *= 2;
  G.kc = kc;
  *grid = dim3(gx, gy, (unsigned)((P + kc - 1) / kc));
  *block = dim3(bx, by);
  return G;
}

}  // namespace

void DirectSolver::apply_mixed(const float* r, float* hi, float* lo, double phi_c, double dphi_dk, const SolveCtl* c,
                               cudaStream_t s) const {
  apply(*this, r, AddMixed{hi, lo, phi_c, dphi_dk}, c, s);
}

void DirectSolver::apply_fp64(const double* r, double* x, const SolveCtl* c, cudaStream_t s) const {
  apply(*this, r, Add64{x}, c, s);
}

void DirectSolver::residual_mixed(bool first, const MgLevel& M, const float* hi, const float* lo, const float* f, float* r,
                                  float fold_first, float fold_last, double* part, SolveCtl* c, const DirectLoop& d,
                                  cudaStream_t s) const {
  // float4 rows: hi starts one plane into phi32, so its rows are aligned when nx is a multiple of 4
  const bool v4 = res_vec(M, 4, M.nx % 4 == 0) == 4;
  dim3 g, b;
  const ResGeom G = res_geom(M, v4 ? 4 : 1, &g, &b);
  if (v4 && first)
    SOLVER_LAUNCH(g, b, 0, s, k_dir_resid_ff<4, true>)(G, hi, lo, f, r, fold_first, fold_last, part, c, d);
  else if (v4)
    SOLVER_LAUNCH(g, b, 0, s, k_dir_resid_ff<4, false>)(G, hi, lo, f, r, fold_first, fold_last, part, c, d);
  else if (first)
    SOLVER_LAUNCH(g, b, 0, s, k_dir_resid_ff<1, true>)(G, hi, lo, f, r, fold_first, fold_last, part, c, d);
  else
    SOLVER_LAUNCH(g, b, 0, s, k_dir_resid_ff<1, false>)(G, hi, lo, f, r, fold_first, fold_last, part, c, d);
}

void DirectSolver::residual_fp64(bool first, const MgLevel& M, const double* x, const double* b, double* r, double* part,
                                 SolveCtl* c, const DirectLoop& d, cudaStream_t s) const {
  // double2 rows: the caller's own array may start anywhere on a double
  const bool v2 = res_vec(M, 2, M.nx % 2 == 0 && ((uintptr_t)x | (uintptr_t)b | (uintptr_t)r) % 16 == 0) == 2;
  dim3 g, bl;
  const ResGeom G = res_geom(M, v2 ? 2 : 1, &g, &bl);
  if (v2 && first) SOLVER_LAUNCH(g, bl, 0, s, k_dir_resid64<2, true>)(G, x, b, r, part, c, d);
  else if (v2) SOLVER_LAUNCH(g, bl, 0, s, k_dir_resid64<2, false>)(G, x, b, r, part, c, d);
  else if (first) SOLVER_LAUNCH(g, bl, 0, s, k_dir_resid64<1, true>)(G, x, b, r, part, c, d);
  else SOLVER_LAUNCH(g, bl, 0, s, k_dir_resid64<1, false>)(G, x, b, r, part, c, d);
}

}  // namespace pic
