// power.cu -- power iteration v <- A v / ||A v||_2 on a handle, in the original
// space (the permuted product of Eq. 1 with x gathered through cperm and y
// scattered through rperm).  Not in the paper: it is the reuse of one matrix
// across many products that the paper's preconditioning analogy (Section 1)
// assumes, and the serving loop's iterative request type.
//
// Norms and the Rayleigh quotient are FP64 two-stage reductions with a fixed
// block split and fixed trees, so the result is deterministic.  The
// normalisation reads the norm from device memory: no host round trip inside
// the loop.  A step is three launches: the product w = A v, the partial sums of
// w.w (and of v.w for the quotient), and one kernel that adds the partials,
// scales w and gathers the next product's x' = v[cperm].
#include <algorithm>

#include "handle.cuh"
#include "launch.cuh"

namespace maxe {
namespace {

constexpr int kDotThreads = 256;
constexpr int kDotBlocks = 512;

// Sums in FP64 are kept to one warp: an SM has two FP64 lanes, so a tree over
// eight warps, each adding all eight warps' sums, took half of dot_partial's 6 us.

// Sum over a warp (a fixed tree), valid in every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// Sum of the block's values ws[0 .. kDotThreads), by one whole warp.
__device__ __forceinline__ double block_sum(const double* ws) {
  const int lane = threadIdx.x & 31;
  double t = ws[lane];
#pragma unroll
  for (int k = 1; k < kDotThreads / 32; ++k) t += ws[lane + 32 * k];
  return warp_sum(t);
}

// Sum of np <= kDotBlocks partials, by one whole warp: four running sums a lane,
// the loads of all in flight together.
__device__ __forceinline__ double sum_parts(const double* __restrict__ part, int np) {
  const int lane = threadIdx.x & 31;
  double v[kDotBlocks / 32];
#pragma unroll
  for (int k = 0; k < kDotBlocks / 32; ++k) v[k] = lane + 32 * k < np ? part[lane + 32 * k] : 0.0;
  double a[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
  for (int k = 4; k < kDotBlocks / 32; ++k)
    if (32 * k < np) a[k % 4] += v[k];
  return warp_sum((a[0] + a[1]) + (a[2] + a[3]));
}

// part_aa[b] = sum of a[i]^2, part_ab[b] = sum of a[i] * b[Qb ? Qb[i] : i] over
// block b's slice (either may be null).  Four elements of a thread are in
// flight at a time: at the served sizes the kernel is one or two rounds of
// load latency, not bandwidth.
template <typename T>
__global__ void __launch_bounds__(kDotThreads) dot_partial(const T* __restrict__ a, const T* __restrict__ b,
                                                           const int32_t* __restrict__ Qb, int64_t n,
                                                           double* __restrict__ part_aa,
                                                           double* __restrict__ part_ab) {
  start_next();
  after_previous();
  __shared__ double waa[kDotThreads], wab[kDotThreads];
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = blockIdx.x * per, hi = std::min<int64_t>(n, lo + per);
  double aa = 0.0, ab = 0.0;
  for (int64_t i0 = lo + threadIdx.x; i0 < hi; i0 += 4 * kDotThreads) {
    T x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = i0 + u * kDotThreads;
      x[u] = i < hi ? a[i] : T(0);
      y[u] = part_ab && i < hi ? b[Qb ? static_cast<int64_t>(Qb[i]) : i] : T(0);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (part_aa) aa = fma(static_cast<double>(x[u]), static_cast<double>(x[u]), aa);
      if (part_ab) ab = fma(static_cast<double>(x[u]), static_cast<double>(y[u]), ab);
    }
  }
  waa[threadIdx.x] = aa;
  wab[threadIdx.x] = ab;
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp == 0 && part_aa) {
    const double t = block_sum(waa);
    if (threadIdx.x == 0) part_aa[blockIdx.x] = t;
  }
  if (warp == 1 && part_ab) {
    const double t = block_sum(wab);
    if (threadIdx.x == 32) part_ab[blockIdx.x] = t;
  }
}

// One warp: *out = the sum of the partials.
__global__ void __launch_bounds__(32) dot_final(const double* __restrict__ part, int nparts,
                                                double* __restrict__ out) {
  start_next();
  after_previous();
  const double t = sum_parts(part, nparts);
  if (threadIdx.x == 0) *out = t;
}

constexpr int kScaleItems = 4;  // elements per thread

// With s = the sum of part_ww (every block adds the same partials in the same
// order, so no block waits for another): out[j] = w[Q ? Q[j] : j] / sqrt(s)
// and v[j] = w[j] / sqrt(s) (out or v may be null).  Block 0 also writes s to
// *nrm2 and the sum of part_vw to *vw (either may be null).  The square root
// and the division are done once per block: in FP64, with two FMA lanes per SM,
// one of each per element took 12 us of a 300 k vector's step.
template <typename T>
__global__ void __launch_bounds__(kDotThreads) scale_gather(const int32_t* __restrict__ Q, const T* __restrict__ w,
                                                            const double* __restrict__ part_ww,
                                                            const double* __restrict__ part_vw, int np, int64_t n,
                                                            T* __restrict__ out, T* __restrict__ v,
                                                            double* __restrict__ nrm2, double* __restrict__ vw) {
  start_next();
  after_previous();
  __shared__ double inv_s;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * (kDotThreads * kScaleItems) + threadIdx.x;
  T g[kScaleItems], own[kScaleItems];
#pragma unroll
  for (int u = 0; u < kScaleItems; ++u) {  // the loads fly while the partials are added
    const int64_t i = i0 + u * kDotThreads;
    g[u] = out && i < n ? w[Q ? static_cast<int64_t>(Q[i]) : i] : T(0);
    own[u] = v && i < n ? w[i] : T(0);
  }
  const int warp = threadIdx.x >> 5;
  if (warp == 0) {
    const double s = sum_parts(part_ww, np);
    if (threadIdx.x == 0) {
      inv_s = 1.0 / sqrt(s);
      if (blockIdx.x == 0 && nrm2) *nrm2 = s;
    }
  }
  if (warp == 1 && blockIdx.x == 0 && vw) {
    const double q = sum_parts(part_vw, np);
    if (threadIdx.x == 32) *vw = q;
  }
  __syncthreads();
  const double inv = inv_s;
#pragma unroll
  for (int u = 0; u < kScaleItems; ++u) {
    const int64_t i = i0 + u * kDotThreads;
    if (i < n) {
      if (out) out[i] = static_cast<T>(static_cast<double>(g[u]) * inv);
      if (v) v[i] = static_cast<T>(static_cast<double>(own[u]) * inv);
    }
  }
}

int dot_blocks(int64_t n) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kDotBlocks, ceil_div(n, 4 * kDotThreads))));
}

unsigned scale_blocks(int64_t n) {
  return static_cast<unsigned>(std::max<int64_t>(1, ceil_div(n, kDotThreads * kScaleItems)));
}

// The products of an iteration are never staged tiles, so that its history does not
// move with what the autotuner picked: the quotient of a matrix without a dominant
// eigenvalue moves by 1e-6 with the order of its FP32 sums, as with any change of
// rounding.  A large permuted stencil pays for it (4096 x 4096, FP32: a product takes
// 660 us here and 377 us by tiles).
constexpr int kProduct = -2;

// hist_host (nullable): the Rayleigh quotient v^T A v of the iterate after
// every step, taken from the product that starts the next step (no extra
// products); the last one is lambda.
template <typename T>
maxe_status run(const maxe_handle* h, const T* v0, int32_t steps, T* v, double* lambda_host, double* hist_host,
                cudaStream_t st) {
  const int64_t n = h->rows;
  const Allocator al = allocator_on(h, st);
  ScratchSet scratch(al);
  T* w = scratch.get<T>(static_cast<size_t>(n));
  T* xp = h->cperm ? scratch.get<T>(static_cast<size_t>(n)) : nullptr;
  double* part = scratch.get<double>(2 * kDotBlocks + 1 + (hist_host ? std::max(steps, 1) : 0));
  if (!w || (h->cperm && !xp) || !part) return MAXE_ERR_OOM;
  double* part_vw = part + kDotBlocks;
  double* lam = part_vw + kDotBlocks;
  double* hist = hist_host ? lam + 1 : nullptr;
  MAXE_CUDA_TRY(cudaMemcpyAsync(v, v0, sizeof(T) * n, cudaMemcpyDeviceToDevice, st));
  if (xp) MAXE_TRY(launch_gather(h->cperm, n, sizeof(T), 1, v0, 1, xp, 1, st));
  const int nb = dot_blocks(n);
  const T* x = xp ? xp : v;  // the product's x': v itself on a matrix whose columns were not permuted
  for (int32_t s = 0; s < steps; ++s) {
    MAXE_TRY(spmm_launch(h, 1, x, 1, w, 1, h->rperm, st, kProduct));
    const bool quotient = hist && s > 0;  // v = the iterate after step s
    MAXE_CUDA_TRY(launch_after(dot_partial<T>, nb, kDotThreads, 0, st, w, v, nullptr, n, part,
                               quotient ? part_vw : nullptr));
    const bool need_v = !xp || hist || s + 1 == steps;  // v besides the gathered x'
    MAXE_CUDA_TRY(launch_after(scale_gather<T>, scale_blocks(n), kDotThreads, 0, st, h->cperm, w, part, part_vw, nb, n,
                               xp, need_v ? v : nullptr, nullptr, quotient ? hist + s - 1 : nullptr));
    MAXE_CUDA_TRY(cudaGetLastError());
  }
  MAXE_TRY(spmm_launch(h, 1, x, 1, w, 1, h->rperm, st, kProduct));
  MAXE_CUDA_TRY(launch_after(dot_partial<T>, nb, kDotThreads, 0, st, v, w, nullptr, n, nullptr, part_vw));
  MAXE_CUDA_TRY(launch_after(dot_final, 1, 32, 0, st, part_vw, nb, lam));
  MAXE_CUDA_TRY(cudaMemcpyAsync(lambda_host, lam, sizeof(double), cudaMemcpyDeviceToHost, st));
  if (hist && steps > 0) {
    if (steps > 1)
      MAXE_CUDA_TRY(cudaMemcpyAsync(hist_host, hist, sizeof(double) * (steps - 1), cudaMemcpyDeviceToHost, st));
    MAXE_CUDA_TRY(cudaMemcpyAsync(hist_host + steps - 1, lam, sizeof(double), cudaMemcpyDeviceToHost, st));
  }
  MAXE_CUDA_TRY(cudaStreamSynchronize(st));
  return MAXE_OK;
}

template <typename T>
maxe_status norm_gather(const int32_t* Q, int64_t n, const T* w, T* u, double* scratch, cudaStream_t st) {
  const int nb = dot_blocks(n);
  MAXE_CUDA_TRY(launch_after(dot_partial<T>, nb, kDotThreads, 0, st, w, nullptr, nullptr, n, scratch, nullptr));
  MAXE_CUDA_TRY(launch_after(scale_gather<T>, scale_blocks(n), kDotThreads, 0, st, Q, w, scratch, nullptr, nb, n, u,
                             nullptr, scratch + kDotBlocks, nullptr));
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

template <typename T>
maxe_status dot_gather(const int32_t* Q, int64_t n, const T* u, const T* w, double* scratch, double* out,
                       cudaStream_t st) {
  const int nb = dot_blocks(n);
  MAXE_CUDA_TRY(launch_after(dot_partial<T>, nb, kDotThreads, 0, st, u, w, Q, n, nullptr, scratch));
  MAXE_CUDA_TRY(launch_after(dot_final, 1, 32, 0, st, scratch, nb, out));
  return MAXE_OK;
}

}  // namespace

maxe_status power_iteration_run(const maxe_handle* h, const void* v0, int32_t steps, void* v_out,
                                double* lambda_host, double* hist_host, cudaStream_t st) {
  if (h->dtype == MAXE_F64)
    return run<double>(h, static_cast<const double*>(v0), steps, static_cast<double*>(v_out), lambda_host, hist_host,
                       st);
  return run<float>(h, static_cast<const float*>(v0), steps, static_cast<float*>(v_out), lambda_host, hist_host, st);
}

}  // namespace maxe

extern "C" {

maxe_status maxe_vec_norm_gather(const int32_t* Q, int32_t n, int32_t elem_bytes, const void* w, void* u,
                                 double* scratch, void* stream) {
  using namespace maxe;
  if (n < 0 || (elem_bytes != 4 && elem_bytes != 8) || (n > 0 && (!w || !u || !scratch))) return MAXE_ERR_INVALID;
  if (n == 0) return MAXE_OK;
  cudaStream_t st = as_stream(stream);
  if (elem_bytes == 8)
    return norm_gather(Q, n, static_cast<const double*>(w), static_cast<double*>(u), scratch, st);
  return norm_gather(Q, n, static_cast<const float*>(w), static_cast<float*>(u), scratch, st);
}

maxe_status maxe_vec_dot_gather(const int32_t* Q, int32_t n, int32_t elem_bytes, const void* u, const void* w,
                                double* scratch, double* out, void* stream) {
  using namespace maxe;
  if (n < 0 || (elem_bytes != 4 && elem_bytes != 8) || !out || (n > 0 && (!w || !u || !scratch)))
    return MAXE_ERR_INVALID;
  cudaStream_t st = as_stream(stream);
  if (n == 0) {
    MAXE_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(double), st));
    return MAXE_OK;
  }
  if (elem_bytes == 8)
    return dot_gather(Q, n, static_cast<const double*>(u), static_cast<const double*>(w), scratch, out, st);
  return dot_gather(Q, n, static_cast<const float*>(u), static_cast<const float*>(w), scratch, out, st);
}

}  // extern "C"
