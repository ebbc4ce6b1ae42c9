// fe_reduce.cuh -- deterministic CTA and grid reductions, and the CG scalars finished in them.
#pragma once
#include "fe_cgcore.h"

#define RED_BLOCKS 608  // 4 CTAs per SM on 152 SMs; fixed, so reductions are reproducible
#define RED_THREADS 256
#define RED_SLOTS 8
#define RED_U 4  // elements per thread whose loads are issued together in the reduction loops

__device__ __forceinline__ dw dw_shfl_down(dw v, int off) {
  return {__shfl_down_sync(0xffffffffu, v.h, off), __shfl_down_sync(0xffffffffu, v.l, off)};
}

// CTA-wide double-word sum in a fixed shuffle tree; result valid in thread 0
__device__ __forceinline__ dw block_reduce_dw(dw v, dw* sh /* [32] */) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = dw_add(v, dw_shfl_down(v, off));
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? sh[threadIdx.x] : dw{0.0f, 0.0f};
  if (wid == 0) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = dw_add(v, dw_shfl_down(v, off));
  }
  __syncthreads();
  return v;
}

// CTA-wide binary64 sum in a fixed shuffle tree; result valid in thread 0
__device__ __forceinline__ double block_reduce_f64(double v, double* sh /* [32] */) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
  if (wid == 0) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  }
  __syncthreads();
  return v;
}

// The same for NS values and CTAs of any size up to 256, summed by one warp: an SM takes 19 cycles for a
// warp's binary64 addition, and a tree in every warp has 80 of them per CTA and value where this has 13.
constexpr int SUM_THREADS = 256, SUM_MAX = 3;
template <int NS>
__device__ __forceinline__ void block_sums_f64(double (&v)[NS], double* sh /* [NS * SUM_THREADS] */) {
  static_assert(NS <= SUM_MAX, "shared memory of the callers");
#pragma unroll
  for (int s = 0; s < NS; ++s) sh[s * SUM_THREADS + threadIdx.x] = v[s];
  __syncthreads();
  if (threadIdx.x < 32) {
    const int n = blockDim.x, lanes = min(32, n);
    for (int t = threadIdx.x + 32; t < n; t += 32)
#pragma unroll
      for (int s = 0; s < NS; ++s) v[s] += sh[s * SUM_THREADS + t];
    const unsigned mask = lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const double t = __shfl_down_sync(mask, v[s], off);
        if ((int)threadIdx.x + off < lanes) v[s] += t;
      }
  }
  __syncthreads();
}

// True in the last CTA of the grid to arrive, which then sees everything the others wrote before they
// arrived.  The counter is left at zero.
__device__ __forceinline__ bool last_cta(unsigned* counter) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
    if (last) *counter = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last != 0;
}

// sums of NS slots of nparts partials each, `stride` apart, by one CTA in a fixed order; valid in
// thread 0
template <int NS>
__device__ __forceinline__ void sum_slots(const double* partials, int nparts, int stride,
                                          double (&out)[NS], double* sh) {
  double acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x; b < nparts; b += blockDim.x)
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[s] += __ldcg(partials + (size_t)s * stride + b);
#pragma unroll
  for (int s = 0; s < NS; ++s) out[s] = acc[s];
  block_sums_f64<NS>(out, sh);
}

// alpha = <r,z>/<q,p> from the partials of <q,p>, by one CTA
__device__ __forceinline__ void fin_alpha(const double* partials, int nparts, CgScal* sc, double* hist,
                                          double* sh) {
  double qp[1];
  sum_slots<1>(partials, nparts, 0, qp, sh);
  if (threadIdx.x == 0) {
    sc->qp = qp[0];
    if (!(qp[0] > 0.0) || !isfinite(qp[0]) || !isfinite(sc->rz)) {
      sc->status = FE_ERR_BREAKDOWN;
      sc->done = 1;
    } else {
      sc->alpha = sc->rz / qp[0];
      if (hist) hist[3 * sc->iter + 0] = sc->alpha;
    }
  }
}

// A thread's running sum of double-word terms, normalised after every term: the low part then stays below
// an ulp of the high part and its rounding errors near 2^-48 of the sum each, whatever the number of terms.
// Left unnormalised (8 operations a term instead of 11) the low part grows with the sum of the errors it
// holds: 1.7 times the error at 16 terms, 3 at 108, 6 at 640 (positive terms).
struct DwSum {
  dw v = {0.0f, 0.0f};
  __device__ __forceinline__ void add(dw t) { v = dw_add(v, t); }
  __device__ __forceinline__ double value() const { return dw_to_double(v); }
};

// A thread's running sum of products in a pairing: float vectors in double-word (exact products);
// double vectors in binary64 FMAs on the FP64 pipe, one per product, which costs less than
// converting both factors to double-word
__device__ __forceinline__ dw prod_dw(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ dw prod_dw(double a, double b) {
  return dw_mul(dw_from_double(a), dw_from_double(b));
}
template <class S>
struct Acc;
template <>
struct Acc<float> {
  DwSum v;
  __device__ __forceinline__ void add_prod(float a, float b) { v.add(prod_dw(a, b)); }
  __device__ __forceinline__ double value() const { return v.value(); }
};
template <>
struct Acc<double> {
  double v = 0.0;
  __device__ __forceinline__ void add_prod(double a, double b) { v = fma(a, b, v); }
  __device__ __forceinline__ double value() const { return v; }
};

// Fused CG iteration: the CTA's part of <q,p>; the last CTA forms alpha.
template <class S>
__device__ __forceinline__ void cg_finish_apply(const CgApply& cg, const Acc<S>& acc) {
  __shared__ double sh[SUM_THREADS];
  double v[1] = {acc.value()};
  block_sums_f64<1>(v, sh);
  if (threadIdx.x == 0) cg.partials[blockIdx.x] = v[0];
  if (last_cta(cg.count)) fin_alpha(cg.partials, (int)gridDim.x, cg.sc, cg.hist, sh);
}
