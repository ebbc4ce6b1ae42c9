// fe_cg.cu -- conjugate gradients on cell-wise data (Sec. 3.2, Algorithm "Communication-Free
// (Flexible) PCG") with the Jacobi preconditioner P = D_cell^{-1} S (Sec. 3.3).
//
// Every vector of the iteration is cell-wise: u, p, z primal (continuous), r, q dual.  The only
// inter-element step is the DSS inside the preconditioner; every scalar is a duality pairing of
// one dual and one primal vector (Lemma "Duality Pairing Identity"), so the iterates equal those
// of CG on the assembled system (Theorem "Equivalence of Communication-Free FCG").
//
// One iteration is a fixed launch sequence, captured into a CUDA graph of GRAPH_ITERS iterations:
//   p = z + beta p, q = A p, <q,p> -> alpha (one kernel where the operator takes it, CgApply);
//   u += alpha p, r -= alpha q;
//   w = S r, z = D^{-1} w (0 on Dirichlet nodes) with sum w^2/mult, <r,z> (and <q,z> for FCG) -> beta.
// The scalars of a pairing are finished by the last CTA of its kernel.
// alpha, beta, the residual and the stop flag stay in device memory; every kernel returns at once
// when the flag is set, so the host replays the graph several times between two reads of the flag.
// Convergence (unspecified in the paper): ||G^T r||_2 / ||G^T b||_2 <= rtol over free nodes, with
// ||G^T r||^2 = sum_e (S r)_e^2 / mult_e.
//
// Mixed precision: FP32 PCG with FP64 reliable updates (solve_reliable), or FP64 FCG whose variable
// preconditioner is an FP32 PCG solve (solve_fcg_outer).
#include <cmath>
#include <cstring>
#include <new>

#include "fe_cgcore.h"
#include "fe_vec.cuh"

namespace {

// ---- element-wise kernels -------------------------------------------------------------------
// 1/multiplicity per cell-wise node (0 on Dirichlet nodes).  A slab's bottom / top nodes have a
// copy in the neighbouring slab when nbr_lo / nbr_hi; `mask` holds the FE_DIR_* Dirichlet faces.
__global__ void k_invmult(float* __restrict__ out, long long ncells, int n, int mx, int my, int mz,
                          int mask, int nbr_lo, int nbr_hi) {
  const int n3 = n * n * n, p = n - 1;
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long c = warp; c < ncells; c += nwarps) {
    const int cx = (int)(c % mx), cy = (int)((c / mx) % my), cz = (int)(c / ((long long)mx * my));
    for (int l = lane; l < n3; l += 32) {
      const int i = l % n, j = (l / n) % n, k = l / (n * n);
      const int gx = cx * p + i, gy = cy * p + j, gz = cz * p + k;
      int mult = 1;
      if (gx % p == 0 && gx > 0 && gx < mx * p) mult *= 2;
      if (gy % p == 0 && gy > 0 && gy < my * p) mult *= 2;
      if (gz % p == 0 && ((gz > 0 && gz < mz * p) || (gz == 0 && nbr_lo) || (gz == mz * p && nbr_hi)))
        mult *= 2;
      const bool bnd = ((mask & FE_DIR_XY) && (gx == 0 || gx == mx * p || gy == 0 || gy == my * p)) ||
                       ((mask & FE_DIR_ZLO) && gz == 0) || ((mask & FE_DIR_ZHI) && gz == mz * p);
      out[c * n3 + l] = bnd ? 0.0f : 1.0f / (float)mult;
    }
  }
}

__global__ void k_invdiag(const double* __restrict__ d, const float* __restrict__ invmult,
                          double* __restrict__ inv64, float* __restrict__ inv32, long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const double v = invmult[e] == 0.0f ? 0.0 : 1.0 / d[e];
    inv64[e] = v;
    inv32[e] = (float)v;
  }
}

// r = b - q
__global__ void k_residual(const double* __restrict__ b, const double* __restrict__ q,
                           double* __restrict__ r, long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    r[e] = b[e] - q[e];
}

// largest |v| as the bit pattern of a non-negative double (whose order is the values' order)
__global__ void k_absmax_bits(const double* __restrict__ v, long long n,
                              unsigned long long* __restrict__ out) {
  unsigned long long m = 0;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(v[e]) & 0x7FFFFFFFFFFFFFFFull);
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__global__ void k_scale_vec(const double* src, double* dst, double s, long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    dst[e] = s * src[e];
}

// x += d / s
__global__ void k_correct(double* __restrict__ x, const float* __restrict__ d, double inv_s,
                          long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    x[e] += inv_s * (double)d[e];
}

// Elements per thread whose loads a two-input streaming kernel (<q,p>, the p update) issues
// together: eight FP32 elements keep as many bytes in flight per thread as four FP64 ones.
template <class S>
__host__ __device__ constexpr int stream_u() {
  return sizeof(S) == 4 ? 2 * RED_U : RED_U;
}

// u += alpha p ; r -= alpha q, and the new r also into w (the DSS then works on w in place).
// keep_r = 0 leaves r unwritten: with redistribution the preconditioner overwrites r with
// (S r)/mult before anything reads it, so the store would be dead traffic.  Launched on a
// resident grid (RED_BLOCKS CTAs); each thread issues the loads of RED_U of its grid-stride
// elements before their stores (the arrays are distinct): one element at a time, on a grid of
// 2432 CTAs, the kernel ran at 5.4 of the HBM's 6.7 TB/s.
template <class S, class U>
__global__ void k_update_ur(U* __restrict__ u, S* __restrict__ r, S* __restrict__ w,
                            const S* __restrict__ p, const S* __restrict__ q,
                            const CgScal* __restrict__ sc, long long n, int keep_r) {
  if (*(volatile const int*)&sc->done) return;
  const double a = sc->alpha;
  auto step = [&](long long e, U ue, S pe, S qe, S rq) {
    u[e] = (U)((double)ue + a * (double)pe);
    const S re = (S)((double)rq - a * (double)qe);
    if (keep_r) r[e] = re;
    w[e] = re;
  };
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; e + (RED_U - 1) * stride < n; e += RED_U * stride) {
    U uv[RED_U];
    S pv[RED_U], qv[RED_U], rv[RED_U];
#pragma unroll
    for (int k = 0; k < RED_U; ++k) {
      const long long f = e + k * stride;
      uv[k] = u[f], pv[k] = p[f], qv[k] = q[f], rv[k] = r[f];
    }
#pragma unroll
    for (int k = 0; k < RED_U; ++k) step(e + k * stride, uv[k], pv[k], qv[k], rv[k]);
  }
  for (; e < n; e += stride) step(e, u[e], p[e], q[e], r[e]);
}

template <>
__global__ void k_update_ur<float, float>(float* __restrict__ u, float* __restrict__ r,
                                          float* __restrict__ w, const float* __restrict__ p,
                                          const float* __restrict__ q,
                                          const CgScal* __restrict__ sc, long long n, int keep_r) {
  if (*(volatile const int*)&sc->done) return;
  const float a = (float)sc->alpha;
  auto step = [&](long long e, float ue, float pe, float qe, float rq) {
    u[e] = fmaf(a, pe, ue);
    const float re = fmaf(-a, qe, rq);
    if (keep_r) r[e] = re;
    w[e] = re;
  };
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; e + (RED_U - 1) * stride < n; e += RED_U * stride) {
    float uv[RED_U], pv[RED_U], qv[RED_U], rv[RED_U];
#pragma unroll
    for (int k = 0; k < RED_U; ++k) {
      const long long f = e + k * stride;
      uv[k] = u[f], pv[k] = p[f], qv[k] = q[f], rv[k] = r[f];
    }
#pragma unroll
    for (int k = 0; k < RED_U; ++k) step(e + k * stride, uv[k], pv[k], qv[k], rv[k]);
  }
  for (; e < n; e += stride) step(e, u[e], p[e], q[e], r[e]);
}

// p = z + beta p (stream_u elements' loads in flight per thread, on a resident grid)
template <class S>
__global__ void k_update_p(S* __restrict__ p, const S* __restrict__ z, const CgScal* __restrict__ sc,
                           long long n) {
  if (*(volatile const int*)&sc->done) return;
  const S b = (S)sc->beta;
  constexpr int PU = stream_u<S>();
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; e + (PU - 1) * stride < n; e += PU * stride) {
    S zv[PU], pv[PU];
#pragma unroll
    for (int k = 0; k < PU; ++k) zv[k] = z[e + k * stride], pv[k] = p[e + k * stride];
#pragma unroll
    for (int k = 0; k < PU; ++k) p[e + k * stride] = zv[k] + b * pv[k];
  }
  for (; e < n; e += stride) p[e] = z[e] + b * p[e];
}

// double-word for both: the preconditioner kernel already spends its FP64-pipe share on z = w /
// diag (measured: binary64 FMAs for <r,z> there made it slower, 165 -> 202 us at Q3 64^3)
template <class S>
struct AccDw {
  DwSum v;
  __device__ __forceinline__ void add_prod(S a, S b) { v.add(prod_dw(a, b)); }
  __device__ __forceinline__ double value() const { return v.value(); }
};

// residual norm, convergence test and beta
struct FinBeta {
  double rtol;  // negative: sc->rtol
  int mode, flexible;
  double* hist;
  double keep = 0.0;  // FIN_START: beta / <r,z>
};
// by one CTA; the two divisions and the square root, long on the FP64 pipe, in two warps
__device__ void fin_beta(const double* partials, int nparts, CgScal* sc, const FinBeta& f, double* sh) {
  __shared__ double rel;
  double v[3] = {0.0, 0.0, 0.0};
  if (f.mode == FIN_ITER && f.flexible) {
    sum_slots<3>(partials, nparts, RED_BLOCKS, v, sh);
  } else if (f.mode == FIN_INIT_R || f.mode == FIN_ITER || f.mode == FIN_START) {
    double t[2];
    sum_slots<2>(partials, nparts, RED_BLOCKS, t, sh);
    v[0] = t[0], v[1] = t[1];
  } else {
    double t[1];
    sum_slots<1>(partials, nparts, RED_BLOCKS, t, sh);
    v[0] = t[0];
  }
  if (threadIdx.x == 0) sh[0] = v[0];
  __syncthreads();
  if (threadIdx.x == 32 && f.mode != FIN_INIT_B) rel = fin_rel(sc, sh[0], f.mode);
  const double beta =
      threadIdx.x == 0 && f.mode == FIN_ITER ? fin_new_beta(sc, v[1], v[2], f.flexible) : 0.0;
  __syncthreads();
  if (threadIdx.x != 0) return;
  const int k = sc->iter;
  // the direction the first iteration forms, z + beta p: p was z (beta = 0), or a kept direction
  if (f.mode == FIN_INIT_R) sc->beta = 0.0;
  if (f.mode == FIN_START) sc->beta = f.keep * v[1];
  fin_scalars(sc, v[0], v[1], rel, beta, f.rtol < 0.0 ? sc->rtol : f.rtol, f.mode);
  if (f.hist && f.mode == FIN_ITER) {
    f.hist[3 * k + 2] = sc->relres;
    if (!sc->done) f.hist[3 * k + 1] = sc->beta;
  }
}

// <q, p> (slot 0) and alpha
template <class S>
__global__ void __launch_bounds__(RED_THREADS)
    k_qp(const S* __restrict__ q, const S* __restrict__ p, double* partials, unsigned* count,
         CgScal* sc, long long n, double* hist) {
  if (*(volatile const int*)&sc->done) return;
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  Acc<S> acc;
  const long long STRIDE = (long long)gridDim.x * RED_THREADS;
  constexpr int QU = stream_u<S>();
  long long e = (long long)blockIdx.x * RED_THREADS + threadIdx.x;
  // QU elements' loads in flight before their products join the accumulator, in the same order
  for (; e + (QU - 1) * STRIDE < n; e += QU * STRIDE) {
    S qv[QU], pv[QU];
#pragma unroll
    for (int u = 0; u < QU; ++u) {
      qv[u] = q[e + u * STRIDE];
      pv[u] = p[e + u * STRIDE];
    }
#pragma unroll
    for (int u = 0; u < QU; ++u) acc.add_prod(qv[u], pv[u]);
  }
  for (; e < n; e += STRIDE) acc.add_prod(q[e], p[e]);
  double v[1] = {acc.value()};
  block_sums_f64<1>(v, sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = v[0];
  if (last_cta(count)) fin_alpha(partials, (int)gridDim.x, sc, hist, sh);
}

// z = w * invdiag (when z != null); partials: slot 0 sum w^2 invmult, slot 1 <r,z>, slot 2 <q,z>
// With `redistribute` the dual residual is replaced by its assembled value split evenly over the
// copies, r = (S r) / mult (0 on Dirichlet nodes): the same G^T r and the same pairings with
// continuous vectors, without the cancelling per-copy parts that FP32 cannot hold.  N > 0: w is not
// assembled yet, and every entry gathers its node's copies (dss_gather, n = N).
template <class S, int N>
__global__ void __launch_bounds__(RED_THREADS)
    k_precond(const S* __restrict__ w, S* __restrict__ r, const S* __restrict__ q,
              const S* __restrict__ invdiag, const float* __restrict__ invmult, S* __restrict__ z,
              double* partials, unsigned* count, CgScal* sc, long long n, int check_done, int redistribute,
              const DssGrid grid, const FinBeta fin) {
  if (check_done && *(volatile const int*)&sc->done) return;
  auto assembled = [&](long long f) {
    if constexpr (N > 0)
      return dss_gather<S, N>(w, (int)f, grid);
    else
      return w[f];
  };
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  DwSum a0;
  AccDw<S> a1, a2;
  auto body = [&](long long e, S we, float im, S idg, S rv, S qv) {
    const dw w2 = prod_dw(we, we);
    a0.add({w2.h * im, w2.l * im});  // im: a power of two or zero, exact scaling
    if (z) {
      const S ze = we * idg;
      z[e] = ze;
      S re;
      if (redistribute) {
        re = we * (S)im;
        r[e] = re;
      } else {
        re = rv;
      }
      a1.add_prod(re, ze);
      if (q) a2.add_prod(qv, ze);
    }
  };
  const long long STRIDE = (long long)gridDim.x * RED_THREADS;
  long long e = (long long)blockIdx.x * RED_THREADS + threadIdx.x;
  // RED_U elements' loads in flight before they join the accumulators, in the same order
  for (; e + (RED_U - 1) * STRIDE < n; e += RED_U * STRIDE) {
    S wv[RED_U], idg[RED_U], rv[RED_U], qv[RED_U];
    float im[RED_U];
#pragma unroll
    for (int u = 0; u < RED_U; ++u) {
      const long long f = e + u * STRIDE;
      wv[u] = assembled(f);
      im[u] = invmult[f];
      idg[u] = z ? invdiag[f] : S(0);
      rv[u] = (z && !redistribute) ? r[f] : S(0);
      qv[u] = (z && q) ? q[f] : S(0);
    }
#pragma unroll
    for (int u = 0; u < RED_U; ++u) body(e + u * STRIDE, wv[u], im[u], idg[u], rv[u], qv[u]);
  }
  for (; e < n; e += STRIDE)
    body(e, assembled(e), invmult[e], z ? invdiag[e] : S(0), (z && !redistribute) ? r[e] : S(0),
         (z && q) ? q[e] : S(0));
  // slots 1 and 2 only where they are formed
  if (q) {
    double v[3] = {a0.value(), a1.value(), a2.value()};
    block_sums_f64<3>(v, sh);
    if (threadIdx.x == 0)
      for (int k = 0; k < 3; ++k) partials[k * RED_BLOCKS + blockIdx.x] = v[k];
  } else {
    double v[2] = {a0.value(), a1.value()};
    block_sums_f64<2>(v, sh);
    if (threadIdx.x == 0)
      for (int k = 0; k < (z ? 2 : 1); ++k) partials[k * RED_BLOCKS + blockIdx.x] = v[k];
  }
  if (last_cta(count)) fin_beta(partials, (int)gridDim.x, sc, fin, sh);
}

// Start of an FP32 run on A d = s S(r)/mult, from w = S r in FP64 (assembled: every copy of a node holds
// its value): r32 = s w / mult, z32 = D^{-1} (s w), d32 = 0, and the pairings sum (s w)^2/mult and
// <r32, z32>; p = z where p is given.  The dual residual r is unassembled: the copies of a node hold
// partial integrals that cancel when summed, so near convergence single copies are orders of magnitude
// larger than G^T r.  Rounding them to FP32 would destroy the assembled value; the residual is therefore
// assembled in FP64 first and its value is split evenly over the copies.  G^T r32 = s G^T r, and every
// pairing with a continuous vector is unchanged (Lemma "Duality Pairing Identity").  S r32 is s w
// rounded (exactly where mult is a power of two), so nothing is summed again: the separate passes (right-
// hand side, copy, interface sums, norm, copy, interface sums, preconditioner, two readings of the
// scalars by the host) made an outer step at Q3 32^3 0.15 ms longer than this one kernel (20 us) does.
__global__ void __launch_bounds__(RED_THREADS)
    k_start_run(const double* __restrict__ w, const float* __restrict__ invmult,
                const float* __restrict__ invdiag, double s, float* __restrict__ r,
                float* __restrict__ z, float* __restrict__ d, float* __restrict__ p, double* partials,
                unsigned* count, CgScal* sc, long long n, const FinBeta fin) {
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  DwSum a0;
  Acc<float> a1;
  const long long STRIDE = (long long)gridDim.x * RED_THREADS;
  for (long long e = (long long)blockIdx.x * RED_THREADS + threadIdx.x; e < n; e += RED_U * STRIDE) {
    double wv[RED_U];
    float im[RED_U], dg[RED_U];
#pragma unroll
    for (int u = 0; u < RED_U; ++u) {
      const long long f = e + u * STRIDE;
      if (f < n) wv[u] = w[f], im[u] = invmult[f], dg[u] = invdiag[f];
    }
#pragma unroll
    for (int u = 0; u < RED_U; ++u) {
      const long long f = e + u * STRIDE;
      if (f >= n) continue;
      const float we = (float)(s * wv[u]), ze = we * dg[u], re = we * im[u];
      r[f] = re;
      z[f] = ze;
      d[f] = 0.0f;
      if (p) p[f] = ze;
      const dw w2 = prod_dw(we, we);
      a0.add({w2.h * im[u], w2.l * im[u]});
      a1.add_prod(re, ze);
    }
  }
  double v[2] = {a0.value(), a1.value()};
  block_sums_f64<2>(v, sh);
  if (threadIdx.x == 0)
    for (int k = 0; k < 2; ++k) partials[k * RED_BLOCKS + blockIdx.x] = v[k];
  if (last_cta(count)) fin_beta(partials, (int)gridDim.x, sc, fin, sh);
}

// z = d / s (FP64 primal correction from the FP32 inner solve)
__global__ void k_from_inner(double* __restrict__ z, const float* __restrict__ d, double inv_s,
                             long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    z[e] = inv_s * (double)d[e];
}

// partials: slot 1 <r, z>, slot 2 <q, z> (q may be null)
__global__ void __launch_bounds__(RED_THREADS)
    k_zpairs(const double* __restrict__ r, const double* __restrict__ q,
             const double* __restrict__ z, double* __restrict__ partials, long long n) {
  __shared__ dw sh[32];
  dw a1 = {0.0f, 0.0f}, a2 = {0.0f, 0.0f};
  for (long long e = (long long)blockIdx.x * RED_THREADS + threadIdx.x; e < n;
       e += (long long)RED_BLOCKS * RED_THREADS) {
    const double ze = z[e];
    a1 = dw_add(a1, prod_dw(r[e], ze));
    if (q) a2 = dw_add(a2, prod_dw(q[e], ze));
  }
  a1 = block_reduce_dw(a1, sh);
  if (threadIdx.x == 0) partials[1 * RED_BLOCKS + blockIdx.x] = dw_to_double(a1);
  if (q) {
    a2 = block_reduce_dw(a2, sh);
    if (threadIdx.x == 0) partials[2 * RED_BLOCKS + blockIdx.x] = dw_to_double(a2);
  }
}

// outer FCG scalars: init rz = <r,z>; iteration beta = -<q,z>/<q,p>, rz = <r,z>
__global__ void __launch_bounds__(RED_THREADS)
    k_fin_fcg(const double* __restrict__ partials, CgScal* __restrict__ sc, int init) {
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  double v[2];
  sum_slots<2>(partials + RED_BLOCKS, RED_BLOCKS, RED_BLOCKS, v, sh);
  if (threadIdx.x != 0) return;
  if (!init) sc->beta = -v[1] / sc->qp;
  sc->rz = v[0];
}

unsigned grid_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152LL * 16) b = 152LL * 16;
  return (unsigned)(b < 1 ? 1 : b);
}

// CTAs of the vector kernels of an iteration: four elements per thread at least, at most the resident
// grid (the reductions' order depends on n only)
unsigned red_grid(long long n) {
  const long long b = (n + 4 * RED_THREADS - 1) / (4 * RED_THREADS);
  return (unsigned)(b < 1 ? 1 : b > RED_BLOCKS ? RED_BLOCKS : b);
}

// ---- workspace -------------------------------------------------------------------------------
}  // namespace

static void free_work(CgWork* w, cudaStream_t st) {
  if (!w) return;
  for (int f = 0; f < 2; ++f) {
    if (w->g64[f]) cudaGraphExecDestroy(w->g64[f]);
    if (w->g32[f]) cudaGraphExecDestroy(w->g32[f]);
  }
  void* bufs[] = {w->x, w->r, w->z, w->p, w->q, w->w, w->bs, w->invdiag64, w->partials, w->count, w->hist,
                  w->r32, w->z32, w->p32, w->q32, w->w32, w->d32, w->invdiag32, w->invmult, w->sc};
  for (void* b : bufs) fe_dfree(b, st);
  cudaFreeHost(w->hsc);
  if (w->st) cudaStreamDestroy(w->st);
  delete w;
}

fe_status fe_launch_invmult(const fe_mesh* m, float* out, cudaStream_t st) {
  k_invmult<<<grid_for(m->ncells * 32), 256, 0, st>>>(out, m->ncells, m->n, m->d.mx, m->d.my,
                                                      m->d.mz, fe_dir_mask(m), m->nbr_lo,
                                                      m->nbr_hi);
  return fe_cuda_check(cudaGetLastError(), "invmult launch");
}

static fe_status alloc_work(const fe_mesh* m, CgWork* w) {
  const long long n = m->ncw;
  w->n = n;
  FE_CUDA(cudaStreamCreateWithFlags(&w->st, cudaStreamNonBlocking), "cg stream");
  double** d[] = {&w->x, &w->r, &w->z, &w->p, &w->q, &w->w, &w->bs, &w->invdiag64};
  for (double** v : d) FE_TRY(fe_dalloc((void**)v, n * sizeof(double), w->st, "cg vector"));
  FE_TRY(fe_dalloc((void**)&w->invdiag32, n * sizeof(float), w->st, "cg vector"));
  FE_TRY(fe_dalloc((void**)&w->invmult, n * sizeof(float), w->st, "cg vector"));
  FE_TRY(fe_dalloc((void**)&w->partials,
                   ((size_t)RED_BLOCKS * RED_SLOTS + m->ncells / 2 + 1) * sizeof(double), w->st,
                   "cg partials"));
  FE_TRY(fe_dalloc((void**)&w->count, sizeof(unsigned), w->st, "cg counter"));
  FE_CUDA(cudaMemsetAsync(w->count, 0, sizeof(unsigned), w->st), "cg counter");
  FE_TRY(fe_dalloc((void**)&w->sc, 2 * sizeof(CgScal), w->st, "cg scalars"));
  FE_CUDA(cudaMallocHost(&w->hsc, 2 * sizeof(CgScal)), "cudaMallocHost cg scalars");
  return fe_launch_invmult(m, w->invmult, w->st);
}

// the mesh keeps a workspace only once it is whole: after a failed allocation the next solve starts anew
fe_status fe_cg_get_work(const fe_mesh* cm, bool mixed, CgWork** out) {
  fe_mesh* m = const_cast<fe_mesh*>(cm);
  CgWork* w = static_cast<CgWork*>(m->cg_work);
  if (!w) {
    w = new (std::nothrow) CgWork();
    if (!w) {
      fe_set_error("fe_cg_solve: host allocation failed");
      return FE_ERR_OOM;
    }
    const fe_status s = alloc_work(m, w);
    if (s != FE_OK) {
      free_work(w, w->st);
      return s;
    }
    m->cg_work = w;
    m->cg_free = [](void* p, cudaStream_t st) { free_work(static_cast<CgWork*>(p), st); };
  }
  if (mixed) {
    float** f[] = {&w->r32, &w->z32, &w->p32, &w->q32, &w->w32, &w->d32};
    for (float** v : f)
      if (!*v) FE_TRY(fe_dalloc((void**)v, w->n * sizeof(float), w->st, "cg fp32 vector"));
  }
  *out = w;
  return FE_OK;
}

fe_status fe_cg_ensure_diag(const fe_mesh* m, CgWork* w, int op) {
  if (w->diag_op == op) return FE_OK;
  // w->q as scratch for the assembled diagonal
  FE_TRY(fe_launch_diag(m, op, w->q, w->st));
  k_invdiag<<<grid_for(w->n), 256, 0, w->st>>>(w->q, w->invmult, w->invdiag64, w->invdiag32, w->n);
  FE_CUDA(cudaGetLastError(), "invdiag launch");
  w->diag_op = op;
  return FE_OK;
}

namespace {

// the operator of the FP32 inner solve: FP32, or 16-bit operands with FP32 accumulation
fe_status launch_inner_apply(const ApplyLaunch& L, const CgWork* w) {
  return w->inner_prec == FE_F32 ? fe_launch_apply_f32(L) : fe_launch_apply_lowp(L, w->inner_prec);
}

// Whether S r is gathered inside the preconditioner kernel instead of summed by three passes first:
// on small vectors the passes are three launches of little work, on larger ones their whole-sector
// traffic is cheaper than the gather's.  Gathered against passes, per iteration: FP32 Q5 12^3 (0.4
// million entries) 47 against 53 us, Q3 24^3 (0.9) 51 against 54, Q3 32^3 (2.1) 74 against 72; FP64 Q5
// 12^3 58 against 63, Q1 40^3 (0.5) 73 against 64, Q3 24^3 92 against 79.
template <class S>
bool gather_dss(const fe_mesh* m, long long n, DssGrid* g) {
  return fe_dss_grid(m, g) && n <= (sizeof(S) == 4 ? 1ll << 20 : 400000ll);
}

// w = S wv, z = D^{-1} w, the pairings and the scalars of `fin` (k_precond)
template <class S>
fe_status launch_precond(const fe_mesh* m, CgWork* w, S* wv, S* r, const S* q, const S* invdiag, S* z,
                         CgScal* sc, int check_done, int redistribute, const FinBeta& fin) {
  DssGrid g;
  void (*kernel)(const S*, S*, const S*, const S*, const float*, S*, double*, unsigned*, CgScal*,
                 long long, int, int, const DssGrid, const FinBeta) = k_precond<S, 0>;
  if (gather_dss<S>(m, w->n, &g)) {
    switch (m->n) {
      case 2: kernel = k_precond<S, 2>; break;
      case 3: kernel = k_precond<S, 3>; break;
      case 4: kernel = k_precond<S, 4>; break;
      case 5: kernel = k_precond<S, 5>; break;
      case 6: kernel = k_precond<S, 6>; break;
      case 7: kernel = k_precond<S, 7>; break;
      case 8: kernel = k_precond<S, 8>; break;
    }
  } else {
    FE_TRY(fe_launch_dss(m, sizeof(S) == 8 ? FE_F64 : FE_F32, wv, w->st));
  }
  kernel<<<red_grid(w->n), RED_THREADS, 0, w->st>>>(wv, r, q, invdiag, w->invmult, z, w->partials,
                                                    w->count, sc, w->n, check_done, redistribute, g,
                                                    fin);
  return fe_cuda_check(cudaGetLastError(), "preconditioner launch");
}

// whether the operator takes its neighbours of the iteration into its kernel
template <class S>
bool fuses(const fe_mesh* m, const CgWork* w) {
  return sizeof(S) == 8 ? fe_apply_fuses_cg(m, FE_F64)
                        : w->inner_prec == FE_F32 && fe_apply_fuses_cg(m, FE_F32);
}

// one PCG iteration on vectors of type S, solution of type U, scalars sc
template <class S, class U>
fe_status enqueue_iteration(const fe_mesh* m, CgWork* w, int op, bool flexible, U* u, S* r, S* z,
                            S* p, S* q, S* wv, const S* invdiag, CgScal* sc, double* hist) {
  const long long n = w->n;
  ApplyLaunch L{m, op, p, q, w->st, &sc->done};
  // FP32 iterations redistribute: r = (S r)/mult is formed by the preconditioner
  const int redistribute = sizeof(S) == 4 ? 1 : 0;
  const unsigned grid = red_grid(n);
  const CgApply cg{z, sc, w->partials + (size_t)RED_BLOCKS * RED_SLOTS, w->count, hist, 0};
  const bool fused = fuses<S>(m, w);
  if (fused)
    L.cg = &cg;
  else
    k_update_p<S><<<grid, RED_THREADS, 0, w->st>>>(p, z, sc, n);
  if (sizeof(S) == 8)
    FE_TRY(fe_launch_apply_f64dw(L));
  else
    FE_TRY(launch_inner_apply(L, w));
  if (!fused)
    k_qp<S><<<grid, RED_THREADS, 0, w->st>>>(q, p, w->partials, w->count, sc, n, hist);
  k_update_ur<S, U><<<grid, RED_THREADS, 0, w->st>>>(u, r, wv, p, q, sc, n, !redistribute);
  FE_CUDA(cudaGetLastError(), "cg iteration launch");
  return launch_precond<S>(m, w, wv, r, flexible ? q : nullptr, invdiag, z, sc, 1, redistribute,
                           {-1.0, FIN_ITER, flexible ? 1 : 0, hist});
}

// iterations per graph: between the graphs of a run the GPU waits for the launch
constexpr int GRAPH_ITERS = 4;

// the iteration graph; its stopping tolerance is read from sc->rtol at every replay
template <class S, class U>
fe_status build_graph(const fe_mesh* m, CgWork* w, int op, bool flexible, U* u, S* r, S* z, S* p,
                      S* q, S* wv, const S* invdiag, CgScal* sc, double* hist,
                      cudaGraphExec_t* exec) {
  cudaGraph_t g = nullptr;
  {  // per-kernel attributes are set outside the capture: by one apply first, the fused one's without a launch
    ApplyLaunch L{m, op, p, q, w->st, &sc->done};
    const CgApply cg{z, sc, nullptr, nullptr, nullptr, 1};
    if (fuses<S>(m, w)) L.cg = &cg;
    FE_TRY(sizeof(S) == 8 ? fe_launch_apply_f64dw(L) : launch_inner_apply(L, w));
  }
  FE_CUDA(cudaStreamBeginCapture(w->st, cudaStreamCaptureModeThreadLocal), "begin capture");
  fe_status s = FE_OK;
  for (int k = 0; k < GRAPH_ITERS && s == FE_OK; ++k)
    s = enqueue_iteration<S, U>(m, w, op, flexible, u, r, z, p, q, wv, invdiag, sc, hist);
  cudaError_t e = cudaStreamEndCapture(w->st, &g);
  if (s != FE_OK) {
    if (g) cudaGraphDestroy(g);
    return s;
  }
  FE_CUDA(e, "end capture");
  e = cudaGraphInstantiate(exec, g, 0);
  cudaGraphDestroy(g);
  return fe_cuda_check(e, "graph instantiate");
}

// run graph replays until the flag is set; returns the host copy of the scalars
fe_status run_until_done(CgWork* w, cudaGraphExec_t exec, int slot, CgScal* out) {
  const int batch = 8;  // iterations between two looks at the flag
  for (;;) {
    for (int b = 0; b < batch; b += GRAPH_ITERS) FE_CUDA(cudaGraphLaunch(exec, w->st), "graph launch");
    FE_CUDA(cudaMemcpyAsync(&w->hsc[slot], &w->sc[slot], sizeof(CgScal), cudaMemcpyDeviceToHost,
                            w->st),
            "scalar readback");
    FE_CUDA(cudaStreamSynchronize(w->st), "cg synchronize");
    if (w->hsc[slot].done) break;
  }
  *out = w->hsc[slot];
  return FE_OK;
}

// fresh scalars of a run; rtol is the stopping tolerance the replayed iteration graphs read
fe_status set_scal(CgWork* w, int slot, int maxit, int stall_limit, double rtol) {
  CgScal s;
  std::memset(&s, 0, sizeof(s));
  s.maxit = maxit;
  s.stall_limit = stall_limit;
  s.rtol = rtol;
  w->hsc[slot] = s;
  return fe_cuda_check(
      cudaMemcpyAsync(&w->sc[slot], &w->hsc[slot], sizeof(CgScal), cudaMemcpyHostToDevice, w->st),
      "scalar upload");
}

fe_status read_scal(CgWork* w, int slot, CgScal* out) {
  FE_CUDA(cudaMemcpyAsync(&w->hsc[slot], &w->sc[slot], sizeof(CgScal), cudaMemcpyDeviceToHost, w->st),
          "scalar readback");
  FE_CUDA(cudaStreamSynchronize(w->st), "cg synchronize");
  *out = w->hsc[slot];
  return FE_OK;
}

// ||G^T v||^2 / bnorm into slot's scalars: w = S v (v null: v is in w already), precond kernel without z
template <class S>
fe_status residual_norm(const fe_mesh* m, CgWork* w, const S* v, S* wv, CgScal* sc, int mode) {
  if (v)
    FE_CUDA(cudaMemcpyAsync(wv, v, w->n * sizeof(S), cudaMemcpyDeviceToDevice, w->st), "cg copy");
  FE_TRY(fe_launch_dss(m, sizeof(S) == 8 ? FE_F64 : FE_F32, wv, w->st));
  k_precond<S, 0><<<red_grid(w->n), RED_THREADS, 0, w->st>>>(
      wv, nullptr, nullptr, nullptr, w->invmult, nullptr, w->partials, w->count, sc, w->n, 0, 0,
      DssGrid(), {0.0, mode, 0, nullptr});
  return fe_cuda_check(cudaGetLastError(), "residual norm launch");
}

// initial preconditioned residual: w = S r, z = D^{-1} w, <r,z>, relres; p = z (and beta = 0, so the
// first iteration's z + beta p is z)
template <class S>
fe_status init_direction(const fe_mesh* m, CgWork* w, S* r, S* z, S* p, S* wv, const S* invdiag,
                         CgScal* sc, double rtol) {
  FE_CUDA(cudaMemcpyAsync(wv, r, w->n * sizeof(S), cudaMemcpyDeviceToDevice, w->st), "cg copy");
  FE_TRY(launch_precond<S>(m, w, wv, r, nullptr, invdiag, z, sc, 0, sizeof(S) == 4 ? 1 : 0,
                           {rtol, FIN_INIT_R, 0, nullptr}));
  FE_CUDA(cudaMemcpyAsync(p, z, w->n * sizeof(S), cudaMemcpyDeviceToDevice, w->st), "cg copy");
  return fe_cuda_check(cudaGetLastError(), "init launch");
}

// start of an FP32 run (k_start_run); first: the direction is z, else z + keep <r,z> p
fe_status launch_start_run(CgWork* w, double s, bool first, double keep) {
  k_start_run<<<red_grid(w->n), RED_THREADS, 0, w->st>>>(
      w->w, w->invmult, w->invdiag32, s, w->r32, w->z32, w->d32, first ? w->p32 : nullptr, w->partials,
      w->count, &w->sc[1], w->n, {-1.0, FIN_START, 0, nullptr, first ? 0.0 : keep});
  return fe_cuda_check(cudaGetLastError(), "run start launch");
}

// Inner FP32 PCG on A d = s S(r)/mult with s = 1/||G^T r|| (w must hold S r in FP64, rnorm2
// its squared norm).  Returns the inner iteration count in *iters and the scale s.
fe_status inner_solve(const fe_mesh* m, CgWork* w, int op, int flex, double rnorm2, double irtol,
                      int maxit, int* iters, double* s_out) {
  const double s = 1.0 / sqrt(rnorm2);
  FE_TRY(set_scal(w, 1, maxit, 20, irtol));
  FE_TRY(launch_start_run(w, s, true, 0.0));
  CgScal h;
  if (!w->g32[flex])
    FE_TRY((build_graph<float, float>(m, w, op, flex, w->d32, w->r32, w->z32, w->p32, w->q32, w->w32,
                                      w->invdiag32, &w->sc[1], nullptr, &w->g32[flex])));
  FE_TRY(run_until_done(w, w->g32[flex], 1, &h));
  *iters = h.iter;
  *s_out = s;
  if (h.status == FE_ERR_BREAKDOWN && h.iter == 0) {
    fe_set_error("fe_cg_solve: inner breakdown");
    return FE_ERR_BREAKDOWN;
  }
  return FE_OK;
}

// FP64 flexible CG whose preconditioner is an FP32 PCG solve: z = P(r) = d / s.  P consumes r only
// through S r = G (G^T r) and returns a continuous vector, the consistency the Equivalence theorem
// asks of a (variable) preconditioner; FCG (Notay) absorbs the variation between applications.
fe_status solve_fcg_outer(const fe_mesh* m, CgWork* w, int op, const double* b, double bnorm2,
                          const fe_cg_opts* opts, fe_cg_result* res, fe_status* status) {
  const long long n = w->n;
  const double irtol = opts->inner_rtol > 0.0 ? opts->inner_rtol : 1e-2;
  CgScal h;
  int total = 0, outer = 0, its = 0;
  double s = 1.0;
  // r = b - A x ; ||G^T r||
  {
    ApplyLaunch L{m, op, w->x, w->q, w->st, nullptr};
    FE_TRY(fe_launch_apply_f64dw(L));
  }
  k_residual<<<grid_for(n), 256, 0, w->st>>>(b, w->q, w->r, n);
  FE_TRY(residual_norm<double>(m, w, w->r, w->w, &w->sc[0], FIN_NORM));
  FE_TRY(read_scal(w, 0, &h));
  res->rel_res = sqrt(h.rnorm2 / bnorm2);
  if (res->rel_res <= opts->rtol) {
    *status = FE_OK;
    return FE_OK;
  }
  // z = P(r), p = z, rz = <r, z>
  FE_TRY(inner_solve(m, w, op, 0, h.rnorm2, irtol, opts->maxit, &its, &s));
  total += its;
  k_from_inner<<<grid_for(n), 256, 0, w->st>>>(w->z, w->d32, 1.0 / s, n);
  k_zpairs<<<RED_BLOCKS, RED_THREADS, 0, w->st>>>(w->r, nullptr, w->z, w->partials, n);
  k_fin_fcg<<<1, RED_THREADS, 0, w->st>>>(w->partials, &w->sc[0], 1);
  FE_CUDA(cudaMemcpyAsync(w->p, w->z, n * sizeof(double), cudaMemcpyDeviceToDevice, w->st), "copy");
  *status = FE_ERR_NOT_CONVERGED;
  while (total < opts->maxit) {
    ApplyLaunch L{m, op, w->p, w->q, w->st, nullptr};
    FE_TRY(fe_launch_apply_f64dw(L));
    k_qp<double><<<red_grid(n), RED_THREADS, 0, w->st>>>(w->q, w->p, w->partials, w->count,
                                                         &w->sc[0], n, nullptr);
    k_update_ur<double, double><<<RED_BLOCKS, RED_THREADS, 0, w->st>>>(
        w->x, w->r, w->w, w->p, w->q, &w->sc[0], n, 1);
    FE_TRY(residual_norm<double>(m, w, w->r, w->w, &w->sc[0], FIN_NORM));
    FE_TRY(read_scal(w, 0, &h));
    ++outer;
    res->rel_res = h.relres;
    if (h.done) {  // breakdown flagged by fin_alpha
      *status = (fe_status)h.status;
      break;
    }
    if (!std::isfinite(h.relres)) {
      *status = FE_ERR_BREAKDOWN;
      break;
    }
    if (h.relres <= opts->rtol) {
      *status = FE_OK;
      break;
    }
    FE_TRY(inner_solve(m, w, op, 0, h.rnorm2, irtol, opts->maxit - total, &its, &s));
    total += its;
    k_from_inner<<<grid_for(n), 256, 0, w->st>>>(w->z, w->d32, 1.0 / s, n);
    k_zpairs<<<RED_BLOCKS, RED_THREADS, 0, w->st>>>(w->r, w->q, w->z, w->partials, n);
    k_fin_fcg<<<1, RED_THREADS, 0, w->st>>>(w->partials, &w->sc[0], 0);
    k_update_p<double><<<RED_BLOCKS, RED_THREADS, 0, w->st>>>(w->p, w->z, &w->sc[0], n);
    FE_CUDA(cudaGetLastError(), "fcg launch");
  }
  res->iters = total;
  res->outer_iters = outer;
  return FE_OK;
}

// FP32 PCG with FP64 reliable updates (residual replacement; Sleijpen & van der Vorst 1996, the
// mixed-precision form of Clark et al. 2010): the iteration runs on FP32 vectors and the FP32
// operator; whenever its recursive residual has dropped by the factor delta since the last
// replacement, the correction accumulated in FP32 is added to the FP64 solution, the true residual
// b - A x is formed with the FP64 operator and replaces the recursive one (assembled in FP64 and
// split evenly over the copies of each node, scaled to unit norm), and the search direction is
// kept: p = P r' + beta p with beta = <r', P r'> / <r_{k-1}, z_{k-1}>.  Keeping p keeps the
// Krylov space, so the iteration count stays near that of FP64 PCG, while every step but the few
// replacements runs in FP32.  The FP64 residual of the final iterate decides convergence.
fe_status solve_reliable(const fe_mesh* m, CgWork* w, int op, const double* b, double bnorm2,
                         const fe_cg_opts* opts, fe_cg_result* res, fe_status* status) {
  const long long n = w->n;
  const double delta = opts->inner_rtol > 0.0 ? opts->inner_rtol : 0.1;
  int total = 0, outer = 0;
  double s_old = 0.0, rz_old = 0.0;  // scale and <r, z> (scaled units) when the FP32 run stopped
  bool have_p = false;
  CgScal h;
  for (;;) {
    // true FP64 residual of the current iterate; w = S r for the inner right-hand side
    ApplyLaunch L{m, op, w->x, w->q, w->st, nullptr};
    FE_TRY(fe_launch_apply_f64dw(L));
    k_residual<<<grid_for(n), 256, 0, w->st>>>(b, w->q, w->w, n);
    FE_TRY(residual_norm<double>(m, w, nullptr, w->w, &w->sc[0], FIN_NORM));
    FE_TRY(read_scal(w, 0, &h));
    const double rel = sqrt(h.rnorm2 / bnorm2);
    res->rel_res = rel;
    if (rel <= opts->rtol) {
      *status = FE_OK;
      break;
    }
    if (!std::isfinite(rel)) {
      *status = FE_ERR_BREAKDOWN;
      break;
    }
    if (total >= opts->maxit) {
      *status = FE_ERR_NOT_CONVERGED;
      break;
    }
    // run the FP32 iteration down to delta, or to just below the outer target
    const double irtol = std::max(delta, 0.5 * opts->rtol / rel);
    FE_TRY(set_scal(w, 1, opts->maxit - total, 0, irtol));
    // p := z + beta p in the new scale (p and rz_old were in units of s_old):
    // beta = <r', z'> / (rz_old (s / s_old)^2), times s / s_old for p
    const double s = 1.0 / sqrt(h.rnorm2);
    FE_TRY(launch_start_run(w, s, !have_p, have_p ? s_old / (rz_old * s) : 0.0));
    if (!w->g32[0])
      FE_TRY((build_graph<float, float>(m, w, op, false, w->d32, w->r32, w->z32, w->p32, w->q32, w->w32,
                                        w->invdiag32, &w->sc[1], nullptr, &w->g32[0])));
    FE_TRY(run_until_done(w, w->g32[0], 1, &h));
    if (h.status == FE_ERR_BREAKDOWN) {
      *status = FE_ERR_BREAKDOWN;
      break;
    }
    total += h.iter;
    ++outer;
    s_old = s;
    rz_old = h.rz;  // <r_{k-1}, z_{k-1}>: the run stopped before its last beta
    have_p = h.iter > 0 || have_p;
    if (h.iter == 0 && !have_p) {  // converged in FP32 before any step: nothing to add
      *status = FE_ERR_NOT_CONVERGED;
      break;
    }
    k_correct<<<grid_for(n), 256, 0, w->st>>>(w->x, w->d32, 1.0 / s, n);
    FE_CUDA(cudaGetLastError(), "correction launch");
  }
  res->iters = total;
  res->outer_iters = outer;
  return FE_OK;
}

}  // namespace

fe_status fe_launch_absmax(const double* v, long long n, unsigned long long* out, cudaStream_t st) {
  FE_CUDA(cudaMemsetAsync(out, 0, sizeof(*out), st), "absmax");
  k_absmax_bits<<<grid_for(n), 256, 0, st>>>(v, n, out);
  return fe_cuda_check(cudaGetLastError(), "absmax launch");
}

bool fe_scale_of_max(double mx, double* s) {
  if (!std::isfinite(mx)) return false;
  *s = mx > 0.0 ? std::ldexp(1.0, -std::ilogb(mx)) : 1.0;
  return true;
}

fe_status fe_cg_rhs_scale(CgWork* w, const double* b, long long n, double* s) {
  unsigned long long* d = reinterpret_cast<unsigned long long*>(w->partials);
  FE_TRY(fe_launch_absmax(b, n, d, w->st));
  unsigned long long bits = 0;
  FE_CUDA(cudaMemcpyAsync(&bits, d, sizeof(bits), cudaMemcpyDeviceToHost, w->st), "rhs scale");
  FE_CUDA(cudaStreamSynchronize(w->st), "rhs scale");
  double mx;
  std::memcpy(&mx, &bits, sizeof(mx));
  if (!fe_scale_of_max(mx, s)) {
    fe_set_error("cg: the right-hand side holds a non-finite value");
    return FE_ERR_INVALID;
  }
  return FE_OK;
}

fe_status fe_cg_scale(const double* src, double* dst, double s, long long n, cudaStream_t st) {
  k_scale_vec<<<grid_for(n), 256, 0, st>>>(src, dst, s, n);
  return fe_cuda_check(cudaGetLastError(), "cg scale launch");
}

extern "C" fe_status fe_cg_solve(const fe_mesh* m, const double* b, double* x,
                                 const fe_cg_opts* opts, fe_cg_result* res, void* stream) {
  if (!m || !b || !x || !opts || !res) {
    fe_set_error("fe_cg_solve: null argument");
    return FE_ERR_INVALID;
  }
  if (!fe_aligned(b) || !fe_aligned(x)) {
    fe_set_error("fe_cg_solve: vectors must be 16-byte aligned");
    return FE_ERR_INVALID;
  }
  const bool lowp = opts->mixed == FE_BF16_F32ACC || opts->mixed == FE_F16_F32ACC;
  if (opts->maxit < 1 || !(opts->rtol >= 0.0) ||
      (opts->mixed != 0 && opts->mixed != FE_F32 && !lowp)) {
    fe_set_error("fe_cg_solve: invalid options (maxit %d, rtol %g, mixed %d)", opts->maxit,
                 opts->rtol, opts->mixed);
    return FE_ERR_INVALID;
  }
  if (m->packed || m->mzg > 0) {
    fe_set_error("fe_cg_solve: FE_LAYOUT_CELLS meshes only (slabs: fe_slab_cg_solve)");
    return FE_ERR_INVALID;
  }
  if (lowp && m->d.geom_mode != FE_GEOM_STORED) {
    fe_set_error("fe_cg_solve: a 16-bit inner operator needs FE_GEOM_STORED geometry");
    return FE_ERR_INVALID;
  }
  std::memset(res, 0, sizeof(*res));
  FeDeviceGuard device_guard;
  FE_CUDA(device_guard.set(m->d.device), "cudaSetDevice");
  const bool mixed = opts->mixed != 0;
  const int op = FE_LAPLACE;
  CgWork* w = nullptr;
  FE_TRY(fe_cg_get_work(m, mixed, &w));
  FE_CUDA(cudaStreamSynchronize((cudaStream_t)stream), "cg: caller stream");
  FE_TRY(fe_ensure_geometry(m, FE_F64, false));
  if (mixed) {
    FE_TRY(fe_ensure_geometry(m, FE_F32, false));
    if (lowp) FE_TRY(fe_ensure_geometry(m, opts->mixed, false));
    w->inner_prec = opts->mixed;
    if (w->g32_prec != w->inner_prec) {  // the inner graphs bake the operator in
      for (int f = 0; f < 2; ++f)
        if (w->g32[f]) {
          cudaGraphExecDestroy(w->g32[f]);
          w->g32[f] = nullptr;
        }
      w->g32_prec = w->inner_prec;
    }
  }
  FE_TRY(fe_cg_ensure_diag(m, w, op));
  const long long n = w->n;
  const int flex = opts->flexible ? 1 : 0;
  if (opts->history && (!w->hist || w->hist_cap < opts->maxit)) {
    fe_dfree(w->hist, w->st);
    w->hist = nullptr;
    FE_TRY(fe_dalloc((void**)&w->hist, 3 * (size_t)opts->maxit * sizeof(double), w->st, "history"));
    w->hist_cap = opts->maxit;
    for (int f = 0; f < 2; ++f)
      if (w->g64[f]) {
        cudaGraphExecDestroy(w->g64[f]);
        w->g64[f] = nullptr;
      }
  }
  double* hist = opts->history ? w->hist : nullptr;
  if (w->g64_hist != hist) {  // graphs bake the history pointer in
    for (int f = 0; f < 2; ++f)
      if (w->g64[f]) {
        cudaGraphExecDestroy(w->g64[f]);
        w->g64[f] = nullptr;
      }
    w->g64_hist = hist;
  }

  // the system scaled by an exact power of two (fe_cg_rhs_scale): b := sb b, u := sb x, ||G^T b||
  double sb = 1.0;
  FE_TRY(fe_cg_rhs_scale(w, b, n, &sb));
  FE_TRY(fe_cg_scale(b, w->bs, sb, n, w->st));
  FE_TRY(fe_cg_scale(x, w->x, sb, n, w->st));
  b = w->bs;
  FE_TRY(set_scal(w, 0, opts->maxit, 0, opts->rtol));
  FE_TRY(residual_norm<double>(m, w, b, w->w, &w->sc[0], FIN_INIT_B));
  CgScal h;
  FE_TRY(read_scal(w, 0, &h));
  const double bnorm2 = h.bnorm2;
  if (!(bnorm2 > 0.0)) {  // zero right-hand side: the solution is zero
    FE_CUDA(cudaMemsetAsync(x, 0, n * sizeof(double), w->st), "cg zero");
    FE_CUDA(cudaStreamSynchronize(w->st), "cg synchronize");
    res->iters = 0;
    res->outer_iters = 0;
    res->rel_res = 0.0;
    res->status = FE_OK;
    return FE_OK;
  }
  fe_status status = FE_OK;

  if (!mixed) {
    // r = b - A u, z = P r, p = z
    ApplyLaunch L{m, op, w->x, w->q, w->st, nullptr};
    FE_TRY(fe_launch_apply_f64dw(L));
    k_residual<<<grid_for(n), 256, 0, w->st>>>(b, w->q, w->r, n);
    FE_TRY(init_direction<double>(m, w, w->r, w->z, w->p, w->w, w->invdiag64, &w->sc[0], opts->rtol));
    FE_TRY(read_scal(w, 0, &h));
    if (!h.done) {
      if (!w->g64[flex])
        FE_TRY((build_graph<double, double>(m, w, op, flex, w->x, w->r, w->z, w->p, w->q,
                                            w->w, w->invdiag64, &w->sc[0], hist, &w->g64[flex])));
      FE_TRY(run_until_done(w, w->g64[flex], 0, &h));
    }
    res->iters = h.iter;
    res->outer_iters = 1;
    res->rel_res = h.relres;
    status = (fe_status)h.status;
    if (hist && h.iter > 0)
      FE_CUDA(cudaMemcpy(opts->history, hist, 3 * (size_t)h.iter * sizeof(double),
                         cudaMemcpyDeviceToHost),
              "history readback");
  } else if (flex || lowp) {
    // 16-bit inner operators are too coarse to keep a direction across reliable updates (Q3 64^3
    // to 1e-10: bf16 diverged, fp16 needed 3658 iterations at inner_rtol 0.3 against 1013 for
    // FP32), so they precondition FCG
    FE_TRY(solve_fcg_outer(m, w, op, b, bnorm2, opts, res, &status));
  } else {
    FE_TRY(solve_reliable(m, w, op, b, bnorm2, opts, res, &status));
  }
  FE_TRY(fe_cg_scale(w->x, x, 1.0 / sb, n, w->st));  // 1/sb: a power of two, exact
  FE_CUDA(cudaStreamSynchronize(w->st), "cg synchronize");
  res->status = status;
  if (status == FE_ERR_NOT_CONVERGED) fe_set_error("fe_cg_solve: not converged");
  if (status == FE_ERR_BREAKDOWN) fe_set_error("fe_cg_solve: breakdown");
  return status;
}
