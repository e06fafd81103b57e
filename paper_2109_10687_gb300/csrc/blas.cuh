// Reduction machinery, the per-right-hand-side scalar record and the fused
// BLAS-1 kernels of the BiCGStab iteration (Algorithm 5 of
// arXiv:2109.10687), shared by the single-lattice solver and the ragged
// batch solver.
//
// Reductions: every reducing kernel accumulates per thread in float32 (the
// float64 kernels in float64), combines the threads of a block to at least
// float64 accuracy and lets the last block to finish sum the per-block partials in
// float64 in a fixed order, so results do not depend on scheduling.  Kernels
// run on a grid (blocks, k) with blockIdx.y = k the right-hand side (or, in a
// ragged batch, the lattice); a Seg says where element k of a stacked vector
// lives.
//
// The float32 sums of a block's threads are combined in triple-float (72
// bits): this GPU has two float64 lanes per SM, and a tree of float64 shuffles
// over every warp took more time than the data on vectors of a few MB (a
// 32-lattice batch: alpha's dot product 60 us against 19 us for p's update,
// which moves more bytes; with this form 34 us, omega's 74 -> 27 us, the
// second update 94 -> 53 us).
#pragma once

#include "qcd_internal.cuh"

namespace qcd {

constexpr int RED_THREADS = 256;
constexpr int MAX_RED_OUT = 4;

// The scalars of one right-hand side's BiCGStab iteration, in device memory.
struct Scal {
  double rho0_re, rho0_im;
  double alpha_re, alpha_im;
  double omega_re, omega_im;
  double beta_re, beta_im;
  double rnorm2, bnorm2;
  double tol2;  // stop when rnorm2 < tol2 * bnorm2
  double aux;
  int done;     // 1: converged or failed; no further updates
  int status;   // QCD_OK, QCD_ERR_BREAKDOWN, QCD_ERR_NONFINITE
  int conv;     // 1: converged
  int iters;   // iterations begun (counted by k_alpha)
  int xpend;   // 1: x += alpha z_p of this iteration not yet applied (k_update2 or k_xfinal does it)
};

// Where element k of a stacked vector lives: uniform stacking (element k at
// k n, n entries) or ragged (off[k], len[k] entries; off and len in device
// memory).
struct Seg {
  size_t n;
  const size_t* off = nullptr;
  const size_t* len = nullptr;
  __device__ __forceinline__ size_t at(int k) const { return off ? __ldg(off + k) : (size_t)k * n; }
  __device__ __forceinline__ size_t size(int k) const { return off ? __ldg(len + k) : n; }
};

// ---------------------------------------------------------------------------
// reduction machinery
// ---------------------------------------------------------------------------
// A sum of float32 numbers as three of them, a + b + c: the errors of the
// sums of a are summed in b, those of b in c (the cascaded summation of Ogita,
// Rump and Oishi, "Accurate sum and dot product", 2005, with K = 3).  The error
// is of order 2^-72 of the summands' magnitudes, below float64's 2^-53, which
// two of them (48 bits) would not reach.
struct Sum3 {
  float a, b, c;
  __device__ explicit Sum3(float x) : a(x), b(0.f), c(0.f) {}
  __device__ Sum3(float a_, float b_, float c_) : a(a_), b(b_), c(c_) {}
  __device__ __forceinline__ void add(float x) {
    const df64 s = two_sum(a, x), t = two_sum(b, s.lo);
    a = s.hi;
    b = t.hi;
    c += t.lo;
  }
  __device__ __forceinline__ void add(const Sum3& o) {
    const df64 s = two_sum(a, o.a), t = two_sum(b, o.b), u = two_sum(t.hi, s.lo);
    a = s.hi;
    b = u.hi;
    c += o.c + (t.lo + u.lo);
  }
  __device__ __forceinline__ double total() const { return (double)a + ((double)b + (double)c); }
};

// The sum of sh[0 .. RED_THREADS) by one warp, to float64 accuracy: float32
// entries as Sum3, which falls back to float64 when the sum leaves float32's
// range (or is not finite), float64 entries in float64.  Lane 0's value counts.
__device__ __forceinline__ double warp_tree(double d) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
  return d;
}
template <typename T>
__device__ __forceinline__ double warp_total(const T* sh) {
  const int lane = threadIdx.x & 31;
  if constexpr (sizeof(T) == 4) {
    Sum3 s(sh[lane]);
#pragma unroll
    for (int j = 1; j < RED_THREADS / 32; ++j) s.add(sh[lane + 32 * j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      s.add(Sum3(__shfl_down_sync(0xffffffffu, s.a, o), __shfl_down_sync(0xffffffffu, s.b, o),
                 __shfl_down_sync(0xffffffffu, s.c, o)));
    if (isfinite(__shfl_sync(0xffffffffu, s.a, 0))) return s.total();
  }
  double d = sh[lane];
#pragma unroll
  for (int j = 1; j < RED_THREADS / 32; ++j) d += (double)sh[lane + 32 * j];
  return warp_tree(d);
}

// Blocks of a (blocks, k) grid that take part in a reduction over n elements:
// none would be left without an element
__device__ __forceinline__ int red_blocks(size_t n) {
  const size_t chunks = (n + RED_THREADS - 1) / RED_THREADS;
  return chunks < gridDim.x ? (chunks ? (int)chunks : 1) : (int)gridDim.x;
}

// Sums v[k] over the nb participating blocks (the others must not call).
// Writes this block's partials (times scale); returns true (in every thread)
// in the block that finished last, which then holds the totals in tot[].
// A warp per output.
template <int N, typename T>
__device__ __forceinline__ bool grid_reduce(const T (&v)[N], int nb, double* partials, unsigned* counter,
                                            double (&tot)[N], double scale = 1.0) {
  __shared__ T sh[N][RED_THREADS];
  __shared__ double res[N];
  __shared__ bool is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  if (warp < N) {
    const double s = warp_total(sh[warp]);
    if (lane == 0) {
      partials[blockIdx.x * N + warp] = s * scale;
      __threadfence();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(counter, 1u) == (unsigned)(nb - 1);
  __syncthreads();
  if (!is_last) return false;
  if (warp < N) {
    __threadfence();
    double s = 0.0;
#pragma unroll 4
    for (int i = lane; i < nb; i += 32) s += __ldcg(partials + i * N + warp);
    s = warp_tree(s);
    if (lane == 0) res[warp] = s;
  }
  if (threadIdx.x == 0) *counter = 0;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) tot[k] = res[k];
  return true;
}

// apply(i, load(i)) for this thread's elements i of [0, n) in ascending order,
// nb blocks in the grid's stride; the loads of two elements are issued together
template <typename L, typename A>
__device__ __forceinline__ void strided(size_t n, int nb, L load, A apply) {
  const size_t step = (size_t)nb * blockDim.x;
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (; i + step < n; i += 2 * step) {
    const auto a = load(i);
    const auto b = load(i + step);
    apply(i, a);
    apply(i + step, b);
  }
  if (i < n) apply(i, load(i));
}

// complex (a.x + i a.y) * (b.x + i b.y) for the two complex numbers of a float4
__device__ __forceinline__ float4 caxpy4(float ar, float ai, float4 xv, float4 y) {
  y.x = fmaf(ar, xv.x, fmaf(-ai, xv.y, y.x));
  y.y = fmaf(ar, xv.y, fmaf(ai, xv.x, y.y));
  y.z = fmaf(ar, xv.z, fmaf(-ai, xv.w, y.z));
  y.w = fmaf(ar, xv.w, fmaf(ai, xv.z, y.w));
  return y;
}
__device__ __forceinline__ void cdot_acc(float4 a, float4 b, float& re, float& im) {
  re = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, re))));
  im = fmaf(a.x, b.y, fmaf(-a.y, b.x, fmaf(a.z, b.w, fmaf(-a.w, b.z, im))));
}
__device__ __forceinline__ float norm4(float4 a) { return a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w; }

// kernels of Algorithm 5 (defined in solver.cu): grid (blocks, k), RED_THREADS threads
__global__ void k_init(const float4* __restrict__ b, float4* x, float4* r, float4* p, float4* rt, Seg seg,
                       double tol2, Scal* scal, double* partials, unsigned* counters, int* ctrl);
__global__ void k_alpha(const float4* __restrict__ rt, const float4* __restrict__ q, Seg seg, Scal* scal,
                        double* partials, unsigned* counters, int* ctrl);
__global__ void k_update1(float4* x, float4* r, const float4* __restrict__ z, const float4* __restrict__ q, Seg seg,
                          Scal* scal, double* partials, unsigned* counters, int* ctrl);
__global__ void k_omega(const float4* __restrict__ t, const float4* __restrict__ r, Seg seg, Scal* scal,
                        double* partials, unsigned* counters, int* ctrl);
__global__ void k_update2(float4* x, float4* r, const float4* __restrict__ zp, const float4* __restrict__ z,
                          const float4* __restrict__ t, const float4* __restrict__ rt, Seg seg, Scal* scal,
                          double* partials, unsigned* counters, int* ctrl);
__global__ void k_update_p(float4* p, const float4* __restrict__ r, const float4* __restrict__ q, Seg seg,
                           Scal* scal);
__global__ void k_xfinal(float4* x, const float4* __restrict__ z, Seg seg, const Scal* scal);
__global__ void k_loop_cond(cudaGraphConditionalHandle handle, int* ctrl);

}  // namespace qcd
