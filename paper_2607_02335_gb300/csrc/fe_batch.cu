// fe_batch.cu -- many independent solves advanced together (batched CG, and the engine of the
// request server).
//
// Each problem keeps its own mesh, geometry and cell-wise state; the engine advances all active
// problems in lockstep.  Every CG iteration applies the operators of all problems in ONE
// persistent launch over a work list of (problem, cell-tile) items with a per-item degree switch
// into the degree-templated cell kernel; the vector kernels run over lists of (problem, chunk)
// items, and per-problem scalars are reduced one CTA per problem over that problem's chunk
// partials in a fixed order.  A problem's arithmetic therefore never depends on which other
// problems share the launch: its result is bitwise the same alone and in a mix.
//
// Precisions: FP64 Jacobi-PCG (double-word apply), or the mixed scheme of fe_cg_solve with
// mixed = FE_F32: FP32 Jacobi-PCG with FP64 reliable updates (every run of FP32 iterations ends
// with the FP32 correction added to the FP64 solution, the true residual b - A x formed in FP64
// and put in place of the recursive one, and the search direction kept).  The phases (FP64
// replacement, FP32 iterations) are global: a problem whose FP32 run ends early waits for the
// others, which changes nothing in its own sequence of operations.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "fe_apply_launch.cuh"
#include "fe_batch.h"
#include "fe_vec.cuh"

namespace {

constexpr int BT = 256;            // threads of every batched CTA
constexpr long long CHUNK = 4096;  // elements per vector work item (small batches still fill the GPU)

// ---- 1D tables of every degree, in constant memory -------------------------------------------
template <class V>
struct AllTabs {
  Tab1D<2, V> t2;
  Tab1D<3, V> t3;
  Tab1D<4, V> t4;
  Tab1D<5, V> t5;
  Tab1D<6, V> t6;
  Tab1D<7, V> t7;
  Tab1D<8, V> t8;
};
__constant__ AllTabs<dw2> c_tabs_dw;
__constant__ AllTabs<float> c_tabs_f32;

template <int N, class V>
__device__ __forceinline__ const Tab1D<N, V>& tab_of();
#define FE_TAB_OF(NN)                                                            \
  template <>                                                                    \
  __device__ __forceinline__ const Tab1D<NN, dw2>& tab_of<NN, dw2>() {             \
    return c_tabs_dw.t##NN;                                                      \
  }                                                                              \
  template <>                                                                    \
  __device__ __forceinline__ const Tab1D<NN, float>& tab_of<NN, float>() {       \
    return c_tabs_f32.t##NN;                                                     \
  }
FE_TAB_OF(2)
FE_TAB_OF(3)
FE_TAB_OF(4)
FE_TAB_OF(5)
FE_TAB_OF(6)
FE_TAB_OF(7)
FE_TAB_OF(8)
#undef FE_TAB_OF

std::mutex g_tab_mu;
bool g_tab_ready[64] = {};

fe_status ensure_tables(int dev) {
  std::lock_guard<std::mutex> lock(g_tab_mu);
  if (dev < 0 || dev >= 64) return FE_ERR_INVALID;
  if (g_tab_ready[dev]) return FE_OK;
  AllTabs<dw2> tdw;
  AllTabs<float> t32;
  HostTab h[8];
  for (int p = 1; p <= 7; ++p) fe_host_tables(p, &h[p]);
  tdw.t2 = make_tab<2, dw2>(h[1]);
  tdw.t3 = make_tab<3, dw2>(h[2]);
  tdw.t4 = make_tab<4, dw2>(h[3]);
  tdw.t5 = make_tab<5, dw2>(h[4]);
  tdw.t6 = make_tab<6, dw2>(h[5]);
  tdw.t7 = make_tab<7, dw2>(h[6]);
  tdw.t8 = make_tab<8, dw2>(h[7]);
  t32.t2 = make_tab<2, float>(h[1]);
  t32.t3 = make_tab<3, float>(h[2]);
  t32.t4 = make_tab<4, float>(h[3]);
  t32.t5 = make_tab<5, float>(h[4]);
  t32.t6 = make_tab<6, float>(h[5]);
  t32.t7 = make_tab<7, float>(h[6]);
  t32.t8 = make_tab<8, float>(h[7]);
  FE_CUDA(cudaMemcpyToSymbol(c_tabs_dw, &tdw, sizeof(tdw)), "batch tables");
  FE_CUDA(cudaMemcpyToSymbol(c_tabs_f32, &t32, sizeof(t32)), "batch tables");
  g_tab_ready[dev] = true;
  return FE_OK;
}

// ---- work items ------------------------------------------------------------------------------
struct Tile {
  int prob;
  int pad;
  long long cell0;
};
struct Chunk {
  int prob;
  int pad;
  long long lo, hi;
};
struct DssRow {  // one row of interfaces of one problem (see kb_dss)
  int prob, row;
};

// ---- persistent apply ------------------------------------------------------------------------
template <int N, class V>
__device__ __forceinline__ void apply_item(const BProb& P, int prec, int src, long long cell0,
                                           unsigned char* sm) {
  CellArgs<N, V> a;
  if (prec == FE_F64) {
    a.x = reinterpret_cast<const typename NT<V>::SV*>(src ? P.x64 : P.p64);
    a.y = reinterpret_cast<typename NT<V>::SV*>(P.q64);
    a.geo = reinterpret_cast<const typename NT<V>::GV*>(P.geodw);
  } else {
    a.x = reinterpret_cast<const typename NT<V>::SV*>(P.p32);
    a.y = reinterpret_cast<typename NT<V>::SV*>(P.q32);
    a.geo = reinterpret_cast<const typename NT<V>::GV*>(P.geo32);
  }
  a.ncells = P.ncells;
  a.cell_base = 0;
  a.geo_cell0 = 0;
  a.mx = P.mx;
  a.my = P.my;
  a.mz = P.mz;
  a.dirichlet = P.dirichlet;
  for (int c = 0; c < 4; ++c) {
    if constexpr (std::is_same<V, dw2>::value) {
      const dw v = dw_from_double(P.aff[c]);
      a.aff[c] = {f2_pack(v.h, v.h), f2_pack(v.l, v.l)};
    } else
      a.aff[c] = (V)P.aff[c];
  }
  if constexpr (std::is_same<V, dw2>::value) {
    if (P.affine)
      apply_pairs<N, FE_LAPLACE, GEOM_AFFINE_K, MODE_CELLS>(a, tab_of<N, V>(), cell0, sm);
    else
      apply_pairs<N, FE_LAPLACE, GEOM_STORED_K, MODE_CELLS>(a, tab_of<N, V>(), cell0, sm);
  } else {
    if (P.affine)
      apply_cells<N, V, FE_LAPLACE, GEOM_AFFINE_K>(a, tab_of<N, V>(), cell0, sm);
    else
      apply_cells<N, V, FE_LAPLACE, GEOM_STORED_K>(a, tab_of<N, V>(), cell0, sm);
  }
}

// register budget of the persistent apply (FP64: that of the one-layer pair kernel)
template <int N, class V>
__host__ __device__ constexpr int batch_minb() {
  return std::is_same<V, dw2>::value ? pair_minb<N, FE_LAPLACE, MODE_CELLS>() : 1;
}

// persistent apply over the tiles [lo, hi) of one degree (tiles are grouped by degree), each kernel
// compiled for its own degree: registers and shared memory of that degree, not of the largest.
// The next work item is claimed before the current tile's apply (its atomic round trip overlaps
// the apply) and published through a double-buffered shared slot.
template <int N, class V>
__global__ void __launch_bounds__(Shape<N, V>::THREADS, (batch_minb<N, V>()))
    kb_apply_n(const BProb* __restrict__ probs, const Tile* __restrict__ tiles, long long lo,
               long long hi, int slot, int prec, int src, unsigned long long* counter) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ long long item[2];  // written one tile ahead by thread 0
  if (threadIdx.x == 0) item[0] = lo + (long long)atomicAdd(counter, 1ULL);
  __syncthreads();
  int buf = 0;
  long long it = item[0];
  while (it < hi) {  // uniform: every thread reads the same item
    unsigned long long nxt = 0;
    if (threadIdx.x == 0) nxt = atomicAdd(counter, 1ULL);  // consumed after this tile
    const Tile T = tiles[it];
    const BProb& P = probs[T.prob];
    if (!*(volatile const int*)&P.sc[slot].done)  // uniform over the CTA
      apply_item<N, V>(P, prec, src, T.cell0, sm);
    if (threadIdx.x == 0) item[buf ^ 1] = lo + (long long)nxt;
    __syncthreads();  // the shared-memory tile is free and the next item visible
    buf ^= 1;
    it = item[buf];
  }
}

// ---- vector kernels over chunks ----------------------------------------------------------------
template <class S>
__device__ __forceinline__ S* vec(const BProb& P, int which);
// which: 0 x/d, 1 r, 2 z, 3 p, 4 q, 5 w
template <>
__device__ __forceinline__ double* vec<double>(const BProb& P, int which) {
  switch (which) {
    case 0: return P.x64;
    case 1: return P.r64;
    case 2: return P.z64;
    case 3: return P.p64;
    case 4: return P.q64;
    case 5: return P.w64;
    default: return const_cast<double*>(P.b64);
  }
}
template <>
__device__ __forceinline__ float* vec<float>(const BProb& P, int which) {
  switch (which) {
    case 0: return P.d32;
    case 1: return P.r32;
    case 2: return P.z32;
    case 3: return P.p32;
    case 4: return P.q32;
    default: return P.w32;
  }
}

// 16-byte pieces of a chunk.  A thread issues the loads of all its pieces (of every vector of the
// kernel) before the first store or sum: one memory round trip per chunk in FP32, two in FP64, where
// single elements four at a time took four (16-problem FP32 batch: <q,p> 10 us, the u/r update 13, the
// preconditioner 13, the p update 8 per launch).
template <class S, int UN = 4>
struct Vec {
  static constexpr int W = 16 / sizeof(S), U = UN;
  S v[U][W];
  __device__ __forceinline__ void load(int u, const S* p) {
    using T = typename std::conditional<sizeof(S) == 8, double2, float4>::type;
    *reinterpret_cast<T*>(v[u]) = *reinterpret_cast<const T*>(p);
  }
  __device__ __forceinline__ void store(int u, S* p) const {
    using T = typename std::conditional<sizeof(S) == 8, double2, float4>::type;
    *reinterpret_cast<T*>(p) = *reinterpret_cast<const T*>(v[u]);
  }
};
// the float companion (1/mult) of a Vec<S>'s pieces
template <class S>
__device__ __forceinline__ void load_mult(float (&o)[Vec<S>::W], const float* p) {
  if constexpr (sizeof(S) == 4)
    *reinterpret_cast<float4*>(o) = *reinterpret_cast<const float4*>(p);
  else
    *reinterpret_cast<float2*>(o) = *reinterpret_cast<const float2*>(p);
}
// pieces(v0) for every group of U pieces of the chunk [lo, hi) (piece v starts at element lo + v W), then
// single(e) for the elements after the last whole piece
template <class V, class F, class G>
__device__ __forceinline__ void over_chunk(long long lo, long long hi, F pieces, G single) {
  constexpr int W = V::W, U = V::U;
  const int n = (int)(hi - lo), nv = n / W;
  for (int v0 = threadIdx.x; v0 < nv; v0 += U * BT) pieces(v0, nv);
  const int t = nv * W + threadIdx.x;
  if (t < n) single(lo + t);
}

// ---- per-problem scalars, finished by the CTA that writes the last of the problem's partials ----------
template <int NS>
__device__ __forceinline__ void sum_chunks(const BProb& P, const double* partials, double (&v)[NS],
                                           double* sh) {
#pragma unroll
  for (int s = 0; s < NS; ++s) v[s] = 0.0;
  for (int c = P.chunk0 + threadIdx.x; c < P.chunk1; c += BT)
#pragma unroll
    for (int s = 0; s < NS; ++s) v[s] += __ldcg(partials + (size_t)c * 4 + s);
  block_sums_f64<NS>(v, sh);
}

__device__ __forceinline__ void batch_fin_alpha(const BProb& P, int slot, const double* partials,
                                                double* sh) {
  CgScal* sc = &P.sc[slot];
  double qp[1];
  sum_chunks<1>(P, partials, qp, sh);
  if (threadIdx.x != 0) return;
  sc->qp = qp[0];
  if (!(qp[0] > 0.0) || !isfinite(qp[0]) || !isfinite(sc->rz)) {
    sc->status = FE_ERR_BREAKDOWN;
    sc->done = 1;
  } else {
    sc->alpha = sc->rz / qp[0];
  }
}

// mode: FIN_INIT_B, FIN_INIT_R, FIN_ITER, FIN_NORM, FIN_OUTER (fe_cgcore.h); tolerances and the
// FCG switch are per problem (slot 0: the outer or FP64 solve, slot 1: the inner FP32 solve).  The
// divisions and the square root, long on the FP64 pipe, in two warps.
__device__ __forceinline__ void batch_fin_beta(const BProb& P, int slot, int mode,
                                               const double* partials, double* sh) {
  CgScal* sc = &P.sc[slot];
  const int flexible = slot == 0 ? P.flexible : 0;
  const double rtol = slot == 0 ? P.rtol : sc->rtol;
  double v[3] = {0.0, 0.0, 0.0};
  if (mode == FIN_ITER && flexible) {
    sum_chunks<3>(P, partials, v, sh);
  } else {
    double t[2];  // slot 1 is stale, and not used, in the modes without <r,z>
    sum_chunks<2>(P, partials, t, sh);
    v[0] = t[0], v[1] = t[1];
  }
  if (threadIdx.x == 0) sh[0] = v[0];
  __syncthreads();
  if (threadIdx.x == 32 && mode != FIN_INIT_B) sh[1] = fin_rel(sc, sh[0], mode);
  const double beta = threadIdx.x == 0 && mode == FIN_ITER ? fin_new_beta(sc, v[1], v[2], flexible) : 0.0;
  __syncthreads();
  if (threadIdx.x == 0) fin_scalars(sc, v[0], v[1], sh[1], beta, rtol, mode);
  __syncthreads();  // sh is used again by the CTA's next chunk
}

// called by every thread once the chunk's partials are written (by thread 0); true in the CTA whose
// chunk is the last of its problem's.  A problem's chunks all arrive or, when it is done, none.
__device__ __forceinline__ bool last_chunk(const BProb& P, unsigned* arrive) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(arrive, 1u) == (unsigned)(P.chunk1 - P.chunk0 - 1);
    if (last) *arrive = 0u;
  }
  __syncthreads();
  const bool mine = last != 0;
  __syncthreads();
  if (mine) __threadfence();
  return mine;
}

// <q, p> and alpha of every problem (partials[chunk*4 + 0])
template <class S>
__global__ void __launch_bounds__(BT)
    kb_qp(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks, int slot,
          double* partials, unsigned* arrive) {
  using V = Vec<S>;
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[slot].done) continue;
    const S* q = vec<S>(P, 4);
    const S* p = vec<S>(P, 3);
    Acc<S> acc;
    over_chunk<V>(
        C.lo, C.hi,
        [&](int v0, int nv) {
          V qv, pv;
#pragma unroll
          for (int u = 0; u < V::U; ++u) {
            const int v = v0 + u * BT;
            if (v < nv) qv.load(u, q + C.lo + v * V::W), pv.load(u, p + C.lo + v * V::W);
          }
#pragma unroll
          for (int u = 0; u < V::U; ++u)
            if (v0 + u * BT < nv)
#pragma unroll
              for (int w = 0; w < V::W; ++w) acc.add_prod(qv.v[u][w], pv.v[u][w]);
        },
        [&](long long e) { acc.add_prod(q[e], p[e]); });
    double v[1] = {acc.value()};
    block_sums_f64<1>(v, sh);
    if (threadIdx.x == 0) partials[(size_t)c * 4 + 0] = v[0];
    if (arrive && last_chunk(P, arrive + C.prob)) batch_fin_alpha(P, slot, partials, sh);
  }
}

// u += alpha p ; r -= alpha q ; w = r.  keep_r = 0 leaves r unwritten: with redistribution the
// preconditioner overwrites r with (S r)/mult before anything reads it.
template <class S>
__global__ void __launch_bounds__(BT)
    kb_update_ur(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks,
                 int slot, int keep_r) {
  using V = Vec<S, sizeof(S) == 4 ? 4 : 2>;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[slot].done) continue;
    const S a = (S)P.sc[slot].alpha;
    S* u = vec<S>(P, 0);
    S* r = vec<S>(P, 1);
    const S* p = vec<S>(P, 3);
    const S* q = vec<S>(P, 4);
    S* w = vec<S>(P, 5);
    auto fma_ = [](S x, S y, S z) {
      if constexpr (sizeof(S) == 4)
        return fmaf(x, y, z);
      else
        return fma(x, y, z);
    };
    over_chunk<V>(
        C.lo, C.hi,
        [&](int v0, int nv) {
          V uv, pv, qv, rv;
#pragma unroll
          for (int k = 0; k < V::U; ++k) {
            const int v = v0 + k * BT;
            const long long e = C.lo + (long long)v * V::W;
            if (v < nv) uv.load(k, u + e), pv.load(k, p + e), qv.load(k, q + e), rv.load(k, r + e);
          }
#pragma unroll
          for (int k = 0; k < V::U; ++k) {
            const int v = v0 + k * BT;
            if (v >= nv) continue;
            const long long e = C.lo + (long long)v * V::W;
#pragma unroll
            for (int t = 0; t < V::W; ++t) {
              uv.v[k][t] = fma_(a, pv.v[k][t], uv.v[k][t]);
              rv.v[k][t] = fma_(-a, qv.v[k][t], rv.v[k][t]);
            }
            uv.store(k, u + e);
            if (keep_r) rv.store(k, r + e);
            rv.store(k, w + e);
          }
        },
        [&](long long e) {
          u[e] = fma_(a, p[e], u[e]);
          const S re = fma_(-a, q[e], r[e]);
          if (keep_r) r[e] = re;
          w[e] = re;
        });
  }
}

// structured DSS pass of one axis over rows of interfaces of every problem, DSS_TEAM threads per row
// (one warp per row left a row of 12 cells six round trips long: 12 us a pass in the 16-problem batch):
// x-pass row (cz, cy) with items (interface, face node), y-pass row (cz, interface) and z-pass row
// (interface, cy) with items (cx, face node); node counts are compile-time, so the index
// arithmetic inside a row is multiplications and shifts.  Pairs of one pass are disjoint.
constexpr int DSS_TEAM = 128;
template <class S, int N>
__device__ __forceinline__ void dss_row(S* __restrict__ v, int axis, int row, int mx, int my,
                                        int lane) {
  constexpr int P = N - 1, N2 = N * N, N3 = N2 * N;
  long long first, rstep;  // left cell of the row's first item; right cell - left cell
  int items, locL0, locR0, sa, sb;
  if (axis == 0) {
    first = (long long)row * mx;
    items = (mx - 1) * N2;
    rstep = 1;
    locL0 = P, locR0 = 0, sa = N, sb = N2;
  } else if (axis == 1) {
    const int cz = row / (my - 1), u = row - cz * (my - 1);
    first = ((long long)cz * my + u) * mx;
    items = mx * N2;
    rstep = mx;
    locL0 = P * N, locR0 = 0, sa = 1, sb = N2;
  } else {
    const int u = row / my, cy = row - u * my;
    first = ((long long)u * my + cy) * mx;
    items = mx * N2;
    rstep = (long long)mx * my;
    locL0 = P * N2, locR0 = 0, sa = 1, sb = N;
  }
  S* const left = v + first * N3 + locL0;
  S* const right = v + (first + rstep) * N3 + locR0;
  // DU pairs' loads in flight before their stores (pairs of a pass are disjoint)
  constexpr int DU = 4;
  for (int it = lane; it < items; it += DU * DSS_TEAM) {
    int off[DU];
    S l[DU], r[DU];
#pragma unroll
    for (int k = 0; k < DU; ++k) {
      const int t = min(it + k * DSS_TEAM, items - 1);  // past the end: read again, not stored
      const int g = t / N2, f = t - g * N2, fb = f / N, fa = f - fb * N;
      off[k] = g * N3 + fa * sa + fb * sb;
      l[k] = left[off[k]];
      r[k] = right[off[k]];
    }
#pragma unroll
    for (int k = 0; k < DU; ++k)
      if (it + k * DSS_TEAM < items) {
        const S sum = l[k] + r[k];
        left[off[k]] = sum;
        right[off[k]] = sum;
      }
  }
}

template <class S>
__global__ void __launch_bounds__(BT)
    kb_dss(const BProb* __restrict__ probs, const DssRow* __restrict__ rows, int nrows, int slot,
           int axis) {
  constexpr int TEAMS = BT / DSS_TEAM;
  const int lane = threadIdx.x % DSS_TEAM;
  for (int w = blockIdx.x * TEAMS + threadIdx.x / DSS_TEAM; w < nrows; w += gridDim.x * TEAMS) {
    const DssRow R = rows[w];
    const BProb& P = probs[R.prob];
    if (*(volatile const int*)&P.sc[slot].done) continue;  // uniform over the team
    S* v = vec<S>(P, 5);
    switch (P.n) {
      case 2: dss_row<S, 2>(v, axis, R.row, P.mx, P.my, lane); break;
      case 3: dss_row<S, 3>(v, axis, R.row, P.mx, P.my, lane); break;
      case 4: dss_row<S, 4>(v, axis, R.row, P.mx, P.my, lane); break;
      case 5: dss_row<S, 5>(v, axis, R.row, P.mx, P.my, lane); break;
      case 6: dss_row<S, 6>(v, axis, R.row, P.mx, P.my, lane); break;
      case 7: dss_row<S, 7>(v, axis, R.row, P.mx, P.my, lane); break;
      case 8: dss_row<S, 8>(v, axis, R.row, P.mx, P.my, lane); break;
    }
  }
}

// z = w * invdiag (pmode & 1), r = w * invmult (pmode & 2, redistribute); partials slot 0 sum
// w^2/mult, slot 1 <r,z>, slot 2 <q,z> (pmode & 4); then the problem's scalars (batch_fin_beta, mode)
template <class S>
__global__ void __launch_bounds__(BT)
    kb_precond(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks,
               int slot, int pmode, int mode, double* partials, unsigned* arrive) {
  // one 16-byte group per vector in flight: two need 80 registers, and a third of the warps goes (64
  // problems of 4^3 to 32^3: 3.62 s against 3.47; 32 of up to 20^3, FP64: 0.670 against 0.653)
  using V = Vec<S, 1>;
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[slot].done) continue;
    const S* w = vec<S>(P, 5);
    S* r = vec<S>(P, 1);
    S* z = vec<S>(P, 2);
    const S* q = vec<S>(P, 4);
    const S* idg = (sizeof(S) == 8) ? (const S*)P.invdiag64 : (const S*)P.invdiag32;
    const float* im = P.invmult;
    const bool dir = pmode & 1, redist = pmode & 2, flex = pmode & 4;
    DwSum a0, a1, a2;
    auto body = [&](S we, float ime, S dg, S& re, S qe) -> S {  // returns z, updates r
      const dw w2 = prod_dw(we, we);
      a0.add({w2.h * ime, w2.l * ime});
      if (!dir) return S(0);
      const S ze = we * dg;
      if (redist) re = we * (S)ime;
      a1.add(prod_dw(re, ze));
      if (flex) a2.add(prod_dw(qe, ze));
      return ze;
    };
    over_chunk<V>(
        C.lo, C.hi,
        [&](int v0, int nv) {
          V wv, dv, rv, qv;
          float mv[V::U][V::W];
#pragma unroll
          for (int k = 0; k < V::U; ++k) {
            const int v = v0 + k * BT;
            const long long e = C.lo + (long long)v * V::W;
            if (v >= nv) continue;
            wv.load(k, w + e);
            load_mult<S>(mv[k], im + e);
            if (dir) dv.load(k, idg + e);
            if (dir && !redist) rv.load(k, r + e);
            if (dir && flex) qv.load(k, q + e);
          }
#pragma unroll
          for (int k = 0; k < V::U; ++k) {
            const int v = v0 + k * BT;
            const long long e = C.lo + (long long)v * V::W;
            if (v >= nv) continue;
#pragma unroll
            for (int t = 0; t < V::W; ++t)
              wv.v[k][t] = body(wv.v[k][t], mv[k][t], dv.v[k][t], rv.v[k][t], qv.v[k][t]);
            if (dir) wv.store(k, z + e);
            if (dir && redist) rv.store(k, r + e);
          }
        },
        [&](long long e) {
          S re = dir && !redist ? r[e] : S(0);
          const S ze = body(w[e], im[e], dir ? idg[e] : S(0), re, dir && flex ? q[e] : S(0));
          if (dir) z[e] = ze;
          if (dir && redist) r[e] = re;
        });
    // slots 1 and 2 only where they are formed
    if (flex) {
      double v[3] = {a0.value(), a1.value(), a2.value()};
      block_sums_f64<3>(v, sh);
      if (threadIdx.x == 0)
        for (int k = 0; k < 3; ++k) partials[(size_t)c * 4 + k] = v[k];
    } else {
      double v[2] = {a0.value(), a1.value()};
      block_sums_f64<2>(v, sh);
      if (threadIdx.x == 0)
        for (int k = 0; k < (dir ? 2 : 1); ++k) partials[(size_t)c * 4 + k] = v[k];
    }
    if (arrive && last_chunk(P, arrive + C.prob)) batch_fin_beta(P, slot, mode, partials, sh);
  }
}

// p = z + beta p
template <class S>
__global__ void __launch_bounds__(BT)
    kb_update_p(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks,
                int slot) {
  using V = Vec<S>;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[slot].done) continue;
    const S b = (S)P.sc[slot].beta;
    S* p = vec<S>(P, 3);
    const S* z = vec<S>(P, 2);
    over_chunk<V>(
        C.lo, C.hi,
        [&](int v0, int nv) {
          V zv, pv;
#pragma unroll
          for (int k = 0; k < V::U; ++k) {
            const int v = v0 + k * BT;
            const long long e = C.lo + (long long)v * V::W;
            if (v < nv) zv.load(k, z + e), pv.load(k, p + e);
          }
#pragma unroll
          for (int k = 0; k < V::U; ++k) {
            const int v = v0 + k * BT;
            if (v >= nv) continue;
#pragma unroll
            for (int t = 0; t < V::W; ++t) pv.v[k][t] = zv.v[k][t] + b * pv.v[k][t];
            pv.store(k, p + C.lo + (long long)v * V::W);
          }
        },
        [&](long long e) { p[e] = z[e] + b * p[e]; });
  }
}

// dst = src (which -> which)
template <class S>
__global__ void __launch_bounds__(BT)
    kb_copy(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks, int slot,
            int dst, int src) {
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[slot].done) continue;
    S* d = vec<S>(P, dst);
    const S* s = vec<S>(P, src);
    for (long long e = C.lo + threadIdx.x; e < C.hi; e += BT) d[e] = s[e];
  }
}

// a value formed by one thread for its CTA (divisions and square roots in every thread would queue on the
// FP64 pipe: 35 us for the run start of a 16-problem batch)
template <class F>
__device__ __forceinline__ double by_one_thread(double* sh, F f) {
  __syncthreads();  // the previous chunk's value has been read
  if (threadIdx.x == 0) *sh = f();
  __syncthreads();
  return *sh;
}

// start of an FP32 run (k_start_run of fe_cg.cu): w64 holds S r64, s = 1/sqrt(rnorm2); r32 = s w / mult,
// z32 = D^{-1} (s w), d32 = 0, and the run's initial scalars (FIN_START)
__global__ void __launch_bounds__(BT)
    kb_start_run(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks,
                 double* partials, unsigned* arrive) {
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  __shared__ double scale;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[0].done) continue;
    const double s = by_one_thread(&scale, [&] { return 1.0 / sqrt(P.sc[0].rnorm2); });
    DwSum a0;
    Acc<float> a1;
    for (long long e = C.lo + threadIdx.x; e < C.hi; e += RED_U * BT) {
      double wv[RED_U];
      float im[RED_U], dg[RED_U];
#pragma unroll
      for (int u = 0; u < RED_U; ++u) {
        const long long f = e + u * BT;
        if (f < C.hi) wv[u] = P.w64[f], im[u] = P.invmult[f], dg[u] = P.invdiag32[f];
      }
#pragma unroll
      for (int u = 0; u < RED_U; ++u) {
        const long long f = e + u * BT;
        if (f >= C.hi) continue;
        const float we = (float)(s * wv[u]), ze = we * dg[u], re = we * im[u];
        P.r32[f] = re;
        P.z32[f] = ze;
        P.d32[f] = 0.0f;
        const dw w2 = prod_dw(we, we);
        a0.add({w2.h * im[u], w2.l * im[u]});
        a1.add_prod(re, ze);
      }
    }
    double v[2] = {a0.value(), a1.value()};
    block_sums_f64<2>(v, sh);
    if (threadIdx.x == 0)
      for (int k = 0; k < 2; ++k) partials[(size_t)c * 4 + k] = v[k];
    if (arrive && last_chunk(P, arrive + C.prob)) batch_fin_beta(P, 1, FIN_START, partials, sh);
  }
}

// reliable update: x64 += d32 / s (s = 1/||G^T r|| of the run's residual)
__global__ void __launch_bounds__(BT)
    kb_correct(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks) {
  __shared__ double scale;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[0].done) continue;
    const double inv_s = by_one_thread(&scale, [&] { return sqrt(P.sc[0].rnorm2); });
    for (long long e = C.lo + threadIdx.x; e < C.hi; e += RED_U * BT) {
      double xv[RED_U];
      float dv[RED_U];
#pragma unroll
      for (int u = 0; u < RED_U; ++u)
        if (e + u * BT < C.hi) xv[u] = P.x64[e + u * BT], dv[u] = P.d32[e + u * BT];
#pragma unroll
      for (int u = 0; u < RED_U; ++u)
        if (e + u * BT < C.hi) P.x64[e + u * BT] = xv[u] + inv_s * (double)dv[u];
    }
  }
}

// search direction at the start of an FP32 run: z for a problem's first run (sc[0].pad), else the
// previous run's direction kept across the reliable update, p = z + beta p in the new scale with
// beta = <r',z'> / <r_{k-1},z_{k-1}> (saved by kb_save_run in sc[0].rz_new, the scale in sc[0].qz)
__global__ void __launch_bounds__(BT)
    kb_keep_direction(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks) {
  __shared__ double scale;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[0].done) continue;
    const bool first = P.sc[0].pad != 0;  // the buffer's old contents are not read
    const float cf = (float)by_one_thread(&scale, [&] {
      if (first) return 0.0;
      const double ratio = (1.0 / sqrt(P.sc[0].rnorm2)) / P.sc[0].qz;
      return P.sc[1].rz / (P.sc[0].rz_new * ratio);
    });
    for (long long e = C.lo + threadIdx.x; e < C.hi; e += RED_U * BT) {
      float zv[RED_U], pv[RED_U];
#pragma unroll
      for (int u = 0; u < RED_U; ++u)
        if (e + u * BT < C.hi) zv[u] = P.z32[e + u * BT], pv[u] = first ? 0.0f : P.p32[e + u * BT];
#pragma unroll
      for (int u = 0; u < RED_U; ++u)
        if (e + u * BT < C.hi) P.p32[e + u * BT] = fmaf(cf, pv[u], zv[u]);
    }
  }
}

// ---- per-problem kernels -----------------------------------------------------------------------
// the scalars of large batches, and FIN_OUTER from the partials of a preceding FIN_NORM: one CTA per
// problem
__global__ void __launch_bounds__(BT)
    kb_fin_alpha(const BProb* __restrict__ probs, int slot, const double* __restrict__ partials) {
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  const BProb& P = probs[blockIdx.x];
  if (*(volatile const int*)&P.sc[slot].done) return;
  batch_fin_alpha(P, slot, partials, sh);
}
__global__ void __launch_bounds__(BT)
    kb_fin_beta(const BProb* __restrict__ probs, int slot, int mode,
                const double* __restrict__ partials) {
  __shared__ double sh[SUM_MAX * SUM_THREADS];
  const BProb& P = probs[blockIdx.x];
  if (*(volatile const int*)&P.sc[slot].done) return;
  batch_fin_beta(P, slot, mode, partials, sh);
}

// reset the inner scalars for a new inner solve (done mirrors the outer state)
__global__ void kb_reset_inner(BProb* __restrict__ probs, int nprob) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nprob) return;
  const int maxit = probs[i].maxit;
  CgScal* o = &probs[i].sc[0];
  CgScal* in = &probs[i].sc[1];
  const int spent = in->stall_total;  // inner iterations so far
  if (!o->done && spent >= maxit) {
    o->status = FE_ERR_NOT_CONVERGED;
    o->done = 1;
  }
  CgScal s;
  memset(&s, 0, sizeof(s));
  s.maxit = maxit - spent > 0 ? maxit - spent : 1;
  s.stall_total = spent;
  s.done = o->done;
  // run the FP32 iterations down to delta, or to just below the outer target
  s.rtol = fmax(probs[i].irtol, 0.5 * probs[i].rtol / o->relres);
  *in = s;
}

// end of a run: keep <r_{k-1}, z_{k-1}> (the run stopped before its last beta) and the scale
__global__ void kb_save_run(BProb* __restrict__ probs, int nprob) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nprob) return;
  CgScal* o = &probs[i].sc[0];
  if (o->done) return;
  o->rz_new = probs[i].sc[1].rz;
  o->qz = 1.0 / sqrt(o->rnorm2);
  o->pad = 0;
}

// accumulate the finished inner iteration count
__global__ void kb_count_inner(BProb* __restrict__ probs, int nprob) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nprob) return;
  CgScal* in = &probs[i].sc[1];
  if (!probs[i].sc[0].done) in->stall_total += in->iter;
}

// r = b - q, also into w (whose sums over the interfaces follow)
__global__ void __launch_bounds__(BT)
    kb_residual(const BProb* __restrict__ probs, const Chunk* __restrict__ chunks, int nchunks) {
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const Chunk C = chunks[c];
    const BProb& P = probs[C.prob];
    if (*(volatile const int*)&P.sc[0].done) continue;
    for (long long e = C.lo + threadIdx.x; e < C.hi; e += RED_U * BT) {
      double bv[RED_U], qv[RED_U];
#pragma unroll
      for (int u = 0; u < RED_U; ++u)
        if (e + u * BT < C.hi) bv[u] = P.b64[e + u * BT], qv[u] = P.q64[e + u * BT];
#pragma unroll
      for (int u = 0; u < RED_U; ++u)
        if (e + u * BT < C.hi) P.r64[e + u * BT] = P.w64[e + u * BT] = bv[u] - qv[u];
    }
  }
}

// fresh scalars for a solve
__global__ void kb_init_scal(BProb* __restrict__ probs, int nprob) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nprob) return;
  const int maxit = probs[i].maxit;
  CgScal s;
  memset(&s, 0, sizeof(s));
  s.maxit = maxit;
  probs[i].sc[1] = s;
  s.pad = 1;  // first outer direction still to come
  probs[i].sc[0] = s;
}

// contiguous copy of every problem's two scalar records, for one readback
__global__ void kb_gather_sc(const BProb* __restrict__ probs, int nprob, CgScal* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nprob) return;
  out[2 * i] = probs[i].sc[0];
  out[2 * i + 1] = probs[i].sc[1];
}

unsigned grid_chunks(int n) { return (unsigned)std::max(1, std::min(n, 152 * 8)); }

}  // namespace

// ---------------------------------------------------------------------------------------------
// host engine
// ---------------------------------------------------------------------------------------------
fe_status fe_batch_build(FeBatch* B) {
  const int np = (int)B->hp.size();
  std::vector<Tile> tiles_n[2][FE_MAXN + 1];  // [FP64, FP32]
  std::vector<Chunk> vch;
  std::vector<DssRow> dch[3];
  for (int i = 0; i < np; ++i) {
    BProb& P = B->hp[i];
    const int n = P.n;
    int cpb[2] = {0, 0};  // cells per tile
    auto shape = [&](auto N) {
      cpb[0] = Shape<decltype(N)::value, dw2>::CELLS;
      cpb[1] = Shape<decltype(N)::value, float>::CELLS;
    };
    switch (n) {
      case 2: shape(std::integral_constant<int, 2>()); break;
      case 3: shape(std::integral_constant<int, 3>()); break;
      case 4: shape(std::integral_constant<int, 4>()); break;
      case 5: shape(std::integral_constant<int, 5>()); break;
      case 6: shape(std::integral_constant<int, 6>()); break;
      case 7: shape(std::integral_constant<int, 7>()); break;
      case 8: shape(std::integral_constant<int, 8>()); break;
    }
    if (!B->active[i]) {
      P.chunk0 = P.chunk1 = (int)vch.size();
      continue;
    }
    for (int f = 0; f < 2; ++f)
      for (long long c = 0; c < P.ncells; c += cpb[f]) tiles_n[f][n].push_back({i, 0, c});
    P.chunk0 = (int)vch.size();
    for (long long e = 0; e < P.ncw; e += CHUNK) vch.push_back({i, 0, e, std::min(P.ncw, e + CHUNK)});
    P.chunk1 = (int)vch.size();
    // rows of interfaces per axis: x (cz, cy) if mx > 1; y (cz, interface); z (interface, cy)
    const int rows[3] = {P.mx > 1 ? P.my * P.mz : 0, P.mz * (P.my - 1), (P.mz - 1) * P.my};
    for (int a = 0; a < 3; ++a)
      for (int r = 0; r < rows[a]; ++r) dch[a].push_back({i, r});
  }
  // tiles grouped by degree: one persistent apply launch per degree present
  std::vector<Tile> tiles;
  for (int f = 0; f < 2; ++f)
    for (int nn = 0; nn <= FE_MAXN; ++nn) {
      B->tile_lo[f][nn] = (long long)tiles.size();
      tiles.insert(tiles.end(), tiles_n[f][nn].begin(), tiles_n[f][nn].end());
      B->tile_hi[f][nn] = (long long)tiles.size();
    }
  B->ntiles = (long long)tiles.size();
  B->nvch = (int)vch.size();
  for (int a = 0; a < 3; ++a) B->ndch[a] = (int)dch[a].size();
  auto up = [&](void** dst, size_t* cap, const void* src, size_t bytes) -> fe_status {
    if (bytes > *cap) {
      fe_dfree(*dst, B->st);
      *dst = nullptr;
      const size_t nb = std::max<size_t>(bytes + bytes / 2, 256);
      FE_TRY(fe_dalloc(dst, nb, B->st, "batch work list"));
      *cap = nb;
    }
    if (bytes) FE_CUDA(cudaMemcpyAsync(*dst, src, bytes, cudaMemcpyHostToDevice, B->st), "batch upload");
    return FE_OK;
  };
  FE_TRY(up(&B->d_tiles, &B->cap_tiles, tiles.data(), tiles.size() * sizeof(Tile)));
  FE_TRY(up(&B->d_vch, &B->cap_vch, vch.data(), vch.size() * sizeof(Chunk)));
  for (int a = 0; a < 3; ++a)
    FE_TRY(up(&B->d_dch[a], &B->cap_dch[a], dch[a].data(), dch[a].size() * sizeof(DssRow)));
  FE_TRY(up((void**)&B->d_probs, &B->cap_probs, B->hp.data(), np * sizeof(BProb)));
  const size_t pbytes = std::max<size_t>(1, vch.size()) * 4 * sizeof(double);
  if (pbytes > B->cap_partials) {
    fe_dfree(B->d_partials, B->st);
    B->d_partials = nullptr;
    FE_TRY(fe_dalloc((void**)&B->d_partials, pbytes + pbytes / 2, B->st, "batch partials"));
    B->cap_partials = pbytes + pbytes / 2;
  }
  if (B->cap_arrive < (size_t)np) {
    fe_dfree(B->d_arrive, B->st);
    B->d_arrive = nullptr;
    FE_TRY(fe_dalloc((void**)&B->d_arrive, 2 * (size_t)np * sizeof(unsigned), B->st, "batch arrivals"));
    B->cap_arrive = 2 * (size_t)np;
    FE_CUDA(cudaMemsetAsync(B->d_arrive, 0, B->cap_arrive * sizeof(unsigned), B->st), "batch arrivals");
  }
  if (!B->d_counter)
    FE_TRY(fe_dalloc((void**)&B->d_counter, 64 * sizeof(unsigned long long), B->st, "counter"));
  FE_TRY(up((void**)&B->d_sc, &B->cap_sc, nullptr, 0));
  if (B->cap_sc < 2 * np * sizeof(CgScal)) {
    fe_dfree(B->d_sc, B->st);
    B->d_sc = nullptr;
    B->cap_sc = 2 * (size_t)np * sizeof(CgScal) + 64 * sizeof(CgScal);
    FE_TRY(fe_dalloc((void**)&B->d_sc, B->cap_sc, B->st, "batch scalar gather"));
  }
  return FE_OK;
}

template <int N, class V>
static fe_status launch_apply_degree(FeBatch* B, int slot, int src, cudaStream_t st) {
  constexpr int f = std::is_same<V, dw2>::value ? 0 : 1;
  const long long lo = B->tile_lo[f][N], hi = B->tile_hi[f][N];
  if (hi <= lo) return FE_OK;
  using Sh = Shape<N, V>;
  const size_t smem = Sh::smem(FE_LAPLACE);
  static int per_sm_dev[64] = {};  // resident CTAs per SM, per device (attribute set once)
  int dev = 0;
  FE_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
  int per_sm = (dev >= 0 && dev < 64) ? per_sm_dev[dev] : 0;
  if (per_sm == 0) {
    FE_CUDA(cudaFuncSetAttribute(kb_apply_n<N, V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem),
            "batch apply attribute");
    FE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kb_apply_n<N, V>, Sh::THREADS, smem),
            "occupancy");
    per_sm = std::max(1, per_sm);
    if (dev >= 0 && dev < 64) per_sm_dev[dev] = per_sm;
  }
  const long long grid = std::min<long long>(hi - lo, 152LL * per_sm);
  kb_apply_n<N, V><<<(unsigned)grid, Sh::THREADS, smem, st>>>(
      B->d_probs, (const Tile*)B->d_tiles, lo, hi, slot, f == 0 ? FE_F64 : FE_F32,
      src, B->d_counter + N);
  return fe_cuda_check(cudaGetLastError(), "batch apply launch");
}

template <class V>
static fe_status launch_apply_degree(FeBatch* B, int n, int slot, int src, cudaStream_t st) {
  switch (n) {
    case 2: return launch_apply_degree<2, V>(B, slot, src, st);
    case 3: return launch_apply_degree<3, V>(B, slot, src, st);
    case 4: return launch_apply_degree<4, V>(B, slot, src, st);
    case 5: return launch_apply_degree<5, V>(B, slot, src, st);
    case 6: return launch_apply_degree<6, V>(B, slot, src, st);
    case 7: return launch_apply_degree<7, V>(B, slot, src, st);
    default: return launch_apply_degree<8, V>(B, slot, src, st);
  }
}

// The applies of the degrees present, side by side on forked streams: in a small batch each alone leaves
// most of the SMs idle (16 problems of degrees 2, 3, 5 and 7: 7, 7, 15 and 24 us one after the other).
template <class S>
static fe_status launch_apply_batched(FeBatch* B, int slot, int src = 0) {
  using V = typename std::conditional<sizeof(S) == 8, dw2, float>::type;
  constexpr int f = sizeof(S) == 8 ? 0 : 1;
  FE_CUDA(cudaMemsetAsync(B->d_counter, 0, (FE_MAXN + 1) * sizeof(unsigned long long), B->st),
          "counter reset");
  int deg[FE_MAXN], nd = 0;
  for (int n = FE_MAXN; n >= 2; --n)  // the largest degree on the batch's own stream
    if (B->tile_hi[f][n] > B->tile_lo[f][n]) deg[nd++] = n;
  const int forks = std::min(nd - 1, FeBatch::FORKS);
  if (forks > 0) {
    for (int k = 0; k <= forks; ++k) {
      if (k < forks && !B->fork_st[k])
        FE_CUDA(cudaStreamCreateWithFlags(&B->fork_st[k], cudaStreamNonBlocking), "batch fork");
      if (!B->fork_ev[k])
        FE_CUDA(cudaEventCreateWithFlags(&B->fork_ev[k], cudaEventDisableTiming), "batch fork");
    }
    FE_CUDA(cudaEventRecord(B->fork_ev[forks], B->st), "batch fork");
    for (int k = 0; k < forks; ++k)
      FE_CUDA(cudaStreamWaitEvent(B->fork_st[k], B->fork_ev[forks], 0), "batch fork");
  }
  fe_status status = FE_OK;
  for (int k = 0; k < nd && status == FE_OK; ++k)
    status = launch_apply_degree<V>(B, deg[k], slot, src,
                                    k == 0 ? B->st : B->fork_st[(k - 1) % FeBatch::FORKS]);
  // joined also after a failure: the batch's buffers are freed or rebuilt in the order of st
  for (int k = 0; k < forks; ++k) {
    cudaError_t e = cudaEventRecord(B->fork_ev[k], B->fork_st[k]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(B->st, B->fork_ev[k], 0);
    if (e == cudaSuccess) continue;
    cudaStreamSynchronize(B->fork_st[k]);
    const fe_status s = fe_cuda_check(e, "batch join");
    if (status == FE_OK) status = s;
  }
  return status;
}

template <class S>
static fe_status launch_dss_batched(FeBatch* B, int slot) {
  for (int axis = 2; axis >= 0; --axis)
    if (B->ndch[axis] > 0)
      kb_dss<S><<<grid_chunks((B->ndch[axis] * DSS_TEAM + BT - 1) / BT), BT, 0, B->st>>>(
          B->d_probs, (const DssRow*)B->d_dch[axis], B->ndch[axis], slot, axis);
  return fe_cuda_check(cudaGetLastError(), "batch dss launch");
}

// Arrival counters of the kernels that finish the scalars themselves: for batches whose chunks are all
// resident at once.  In larger ones a CTA waits at the end of each chunk for its arrival (about the
// time of the chunk's own traffic), and kernels of their own do it (64 problems of 135 million entries:
// 3865 ms with arrivals, 3731 without).
static unsigned* arrivals(const FeBatch* B) { return B->nvch <= 152 * 8 ? B->d_arrive : nullptr; }
template <class S>
static void launch_precond_batched(FeBatch* B, int slot, int pmode, int mode) {
  unsigned* arrive = arrivals(B);
  kb_precond<S><<<grid_chunks(B->nvch), BT, 0, B->st>>>(B->d_probs, (const Chunk*)B->d_vch, B->nvch, slot,
                                                        pmode, mode, B->d_partials, arrive);
  if (!arrive)
    kb_fin_beta<<<(unsigned)B->hp.size(), BT, 0, B->st>>>(B->d_probs, slot, mode, B->d_partials);
}

// one PCG iteration of every active problem on vectors of type S, scalars `slot`
template <class S>
fe_status fe_batch_iteration(FeBatch* B, int slot, int redistribute) {
  const int flexible = slot == 0 ? B->any_flexible : 0;
  const unsigned g = grid_chunks(B->nvch);
  const Chunk* ch = (const Chunk*)B->d_vch;
  FE_TRY(launch_apply_batched<S>(B, slot));
  unsigned* arrive = arrivals(B);
  kb_qp<S><<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch, slot, B->d_partials, arrive);
  if (!arrive)
    kb_fin_alpha<<<(unsigned)B->hp.size(), BT, 0, B->st>>>(B->d_probs, slot, B->d_partials);
  kb_update_ur<S><<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch, slot, !redistribute);
  FE_TRY(launch_dss_batched<S>(B, slot));
  launch_precond_batched<S>(B, slot, 1 | (redistribute ? 2 : 0) | (flexible ? 4 : 0), FIN_ITER);
  kb_update_p<S><<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch, slot);
  return fe_cuda_check(cudaGetLastError(), "batch iteration launch");
}
template fe_status fe_batch_iteration<double>(FeBatch*, int, int);
template fe_status fe_batch_iteration<float>(FeBatch*, int, int);

// w = S(src) (src < 0: of what w holds) and the norm (FIN_INIT_R: also z = D^{-1} w, p = z, <r,z>) of
// every active problem, in FP64
fe_status fe_batch_norm(FeBatch* B, int src, int mode) {
  const unsigned g = grid_chunks(B->nvch);
  const Chunk* ch = (const Chunk*)B->d_vch;
  if (src >= 0) kb_copy<double><<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch, 0, 5, src);
  FE_TRY(launch_dss_batched<double>(B, 0));
  launch_precond_batched<double>(B, 0, mode == FIN_INIT_R ? 1 : 0, mode);
  if (mode == FIN_INIT_R) kb_copy<double><<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch, 0, 3, 2);
  return fe_cuda_check(cudaGetLastError(), "batch norm launch");
}

fe_status fe_batch_read(FeBatch* B) {
  const int np = (int)B->hp.size();
  if (np == 0) return FE_OK;
  kb_gather_sc<<<(np + 127) / 128, 128, 0, B->st>>>(B->d_probs, np, B->d_sc);
  FE_CUDA(cudaMemcpyAsync(B->hsc, B->d_sc, 2 * np * sizeof(CgScal), cudaMemcpyDeviceToHost, B->st),
          "batch scalar readback");
  return fe_cuda_check(cudaStreamSynchronize(B->st), "batch synchronize");
}

// start of an FP32 run for every unconverged problem: r32 = s (S r)/mult, z32 = P r32, <r32, z32>,
// and the direction (first run: p = z; later: the previous direction kept, kb_keep_direction)
fe_status fe_batch_inner_start(FeBatch* B) {
  const int np = (int)B->hp.size();
  const unsigned g = grid_chunks(B->nvch);
  const Chunk* ch = (const Chunk*)B->d_vch;
  kb_reset_inner<<<(np + 127) / 128, 128, 0, B->st>>>(B->d_probs, np);
  unsigned* arrive = arrivals(B);
  kb_start_run<<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch, B->d_partials, arrive);
  if (!arrive) kb_fin_beta<<<np, BT, 0, B->st>>>(B->d_probs, 1, FIN_START, B->d_partials);
  kb_keep_direction<<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch);
  return fe_cuda_check(cudaGetLastError(), "batch run start");
}

// end of an FP32 run (the reliable update): x += d / s, r = b - A x in FP64, ||G^T r||, convergence
fe_status fe_batch_inner_finish(FeBatch* B) {
  const int np = (int)B->hp.size();
  const unsigned g = grid_chunks(B->nvch);
  const Chunk* ch = (const Chunk*)B->d_vch;
  kb_count_inner<<<(np + 127) / 128, 128, 0, B->st>>>(B->d_probs, np);
  kb_save_run<<<(np + 127) / 128, 128, 0, B->st>>>(B->d_probs, np);
  kb_correct<<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch);
  FE_TRY(launch_apply_batched<double>(B, 0, 1));  // q = A x
  kb_residual<<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch);
  FE_TRY(fe_batch_norm(B, -1, FIN_NORM));
  kb_fin_beta<<<np, BT, 0, B->st>>>(B->d_probs, 0, FIN_OUTER, B->d_partials);
  return fe_cuda_check(cudaGetLastError(), "batch reliable update");
}

fe_status fe_batch_prepare() {
  int dev = 0;
  FE_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
  return ensure_tables(dev);
}

FeBatch::~FeBatch() {
  if (st) cudaStreamSynchronize(st);
  fe_dfree(d_probs, st);
  fe_dfree(d_tiles, st);
  fe_dfree(d_vch, st);
  for (int a = 0; a < 3; ++a) fe_dfree(d_dch[a], st);
  fe_dfree(d_partials, st);
  fe_dfree(d_counter, st);
  fe_dfree(d_arrive, st);
  for (cudaEvent_t e : fork_ev)
    if (e) cudaEventDestroy(e);
  for (cudaStream_t f : fork_st)
    if (f) cudaStreamDestroy(f);
  fe_dfree(d_sc, st);
  if (st) cudaStreamSynchronize(st);
  cudaFreeHost(hsc);
  if (st && own_stream) cudaStreamDestroy(st);
}

fe_status fe_batch_fill(FeBatch* B, int i, const fe_mesh* m, CgWork* w, const double* b,
                        const fe_cg_opts* opts) {
  BProb& P = B->hp[i];
  std::memset(&P, 0, sizeof(P));
  P.rtol = opts->rtol;
  P.irtol = opts->inner_rtol > 0.0 ? opts->inner_rtol : 0.1;
  P.maxit = opts->maxit;
  P.flexible = (opts->mixed == 0 && opts->flexible) ? 1 : 0;
  P.n = m->n;
  P.affine = m->d.geom_mode == FE_GEOM_AFFINE;
  P.ncells = m->ncells;
  P.ncw = m->ncw;
  P.mx = m->d.mx;
  P.my = m->d.my;
  P.mz = m->d.mz;
  P.dirichlet = fe_dir_mask(m);
  const double hx = 1.0 / m->d.mx, hy = 1.0 / m->d.my, hz = 1.0 / m->d.mz, det = hx * hy * hz;
  P.aff[0] = det / (hx * hx);
  P.aff[1] = det / (hy * hy);
  P.aff[2] = det / (hz * hz);
  P.aff[3] = det;
  P.geodw = m->geodw;
  P.geo32 = m->geo32;
  P.x64 = w->x;
  P.r64 = w->r;
  P.z64 = w->z;
  P.p64 = w->p;
  P.q64 = w->q;
  P.w64 = w->w;
  P.b64 = b;
  P.d32 = w->d32;
  P.r32 = w->r32;
  P.z32 = w->z32;
  P.p32 = w->p32;
  P.q32 = w->q32;
  P.w32 = w->w32;
  P.invdiag64 = w->invdiag64;
  P.invdiag32 = w->invdiag32;
  P.invmult = w->invmult;
  P.sc = w->sc;
  return FE_OK;
}

fe_status fe_batch_setup(FeBatch* B) {
  const int np = (int)B->hp.size();
  const unsigned g = grid_chunks(B->nvch);
  const Chunk* ch = (const Chunk*)B->d_vch;
  kb_init_scal<<<(np + 127) / 128, 128, 0, B->st>>>(B->d_probs, np);
  FE_TRY(fe_batch_norm(B, 6, FIN_INIT_B));  // ||G^T b||
  FE_TRY(launch_apply_batched<double>(B, 0, 1));               // q = A x
  kb_residual<<<g, BT, 0, B->st>>>(B->d_probs, ch, B->nvch);
  return fe_cuda_check(cudaGetLastError(), "batch setup");
}

bool fe_batch_all_done(FeBatch* B, int slot) {
  for (size_t i = 0; i < B->hp.size(); ++i)
    if (B->active[i] && !B->hsc[2 * i + slot].done) return false;
  return true;
}

fe_status fe_batch_start(FeBatch* B, bool mixed) {
  FE_TRY(fe_batch_setup(B));
  if (!mixed) return fe_batch_norm(B, -1, FIN_INIT_R);
  FE_TRY(fe_batch_norm(B, -1, FIN_NORM));
  const int np = (int)B->hp.size();
  kb_fin_beta<<<np, BT, 0, B->st>>>(B->d_probs, 0, FIN_OUTER, B->d_partials);  // converged at x0?
  return fe_cuda_check(cudaGetLastError(), "batch start");
}

// after a read-back: converged problems leave the work lists, so the launches of the following
// iterations walk the unconverged problems' tiles and chunks only
static fe_status drop_converged(FeBatch* B) {
  bool changed = false;
  for (size_t i = 0; i < B->hp.size(); ++i)
    if (B->active[i] && B->hsc[2 * i].done) {
      B->active[i] = 0;
      changed = true;
    }
  return changed ? fe_batch_build(B) : FE_OK;
}

fe_status fe_batch_solve(FeBatch* B, const fe_cg_opts* opts) {
  const int batch = 8;
  const bool mixed = opts->mixed == FE_F32;
  FE_TRY(fe_batch_start(B, mixed));
  if (!mixed) {
    FE_TRY(fe_batch_read(B));
    while (!fe_batch_all_done(B, 0)) {
      FE_TRY(drop_converged(B));
      for (int k = 0; k < batch; ++k) FE_TRY(fe_batch_iteration<double>(B, 0, 0));
      FE_TRY(fe_batch_read(B));
    }
    return FE_OK;
  }
  // mixed: FP32 PCG runs between FP64 reliable updates, each problem on its own: after every
  // round of iterations the problems whose run has ended take their reliable update in a batch of
  // their own and leave converged or start their next run (the running batch's kernels skip a
  // problem whose run has ended), so a round costs the iterations it runs, not the longest run
  FE_TRY(fe_batch_read(B));
  FE_TRY(drop_converged(B));
  if (fe_batch_all_done(B, 0)) return FE_OK;
  FE_TRY(fe_batch_inner_start(B));
  auto subset = [&](const std::vector<int>& idx, FeBatch& J) -> fe_status {
    J.st = B->st;
    J.own_stream = false;
    J.hp.resize(idx.size());
    for (size_t k = 0; k < idx.size(); ++k) J.hp[k] = B->hp[idx[k]];
    J.active.assign(idx.size(), 1);
    FE_CUDA(cudaMallocHost(&J.hsc, 2 * idx.size() * sizeof(CgScal)), "batch scalars");
    J.cap_hsc = 2 * idx.size();
    return fe_batch_build(&J);
  };
  for (;;) {
    for (int k = 0; k < batch; ++k) FE_TRY(fe_batch_iteration<float>(B, 1, 1));
    FE_TRY(fe_batch_read(B));
    std::vector<int> ended;
    for (size_t i = 0; i < B->hp.size(); ++i)
      if (B->active[i] && B->hsc[2 * i + 1].done) ended.push_back((int)i);
    if (ended.empty()) continue;
    std::vector<int> cont;
    bool left = false;
    {
      FeBatch J;
      FE_TRY(subset(ended, J));
      FE_TRY(fe_batch_inner_finish(&J));
      FE_TRY(fe_batch_read(&J));
      for (size_t k = 0; k < ended.size(); ++k) {
        if (J.hsc[2 * k].done) {
          B->active[ended[k]] = 0;
          left = true;
        } else {
          cont.push_back(ended[k]);
        }
      }
    }
    if (!cont.empty()) {
      FeBatch K;
      FE_TRY(subset(cont, K));
      FE_TRY(fe_batch_inner_start(&K));
    }
    if (left) {
      bool any = false;
      for (size_t i = 0; i < B->hp.size(); ++i) any |= B->active[i] != 0;
      if (!any) break;
      FE_TRY(fe_batch_build(B));
    }
  }
  return FE_OK;
}

extern "C" fe_status fe_cg_solve_batched(int nprob, const fe_mesh* const* meshes,
                                         const double* const* b, double* const* x,
                                         const fe_cg_opts* opts, fe_cg_result* res, void* stream) {
  if (nprob < 1 || !meshes || !b || !x || !opts || !res) {
    fe_set_error("fe_cg_solve_batched: null argument or nprob < 1");
    return FE_ERR_INVALID;
  }
  if (opts->maxit < 1 || !(opts->rtol >= 0.0) || (opts->mixed != 0 && opts->mixed != FE_F32)) {
    fe_set_error("fe_cg_solve_batched: invalid options");
    return FE_ERR_INVALID;
  }
  for (int i = 0; i < nprob; ++i) {
    if (!meshes[i] || !b[i] || !x[i] || !fe_aligned(b[i]) || !fe_aligned(x[i])) {
      fe_set_error("fe_cg_solve_batched: problem %d: null or misaligned argument", i);
      return FE_ERR_INVALID;
    }
    if (meshes[i]->d.geom_mode == FE_GEOM_RECOMPUTE || meshes[i]->packed || meshes[i]->mzg > 0 ||
        meshes[i]->d.device != meshes[0]->d.device) {
      fe_set_error("fe_cg_solve_batched: problem %d: needs whole meshes with stored/affine geometry "
                   "on one device", i);
      return FE_ERR_INVALID;
    }
    for (int j = 0; j < i; ++j)
      if (meshes[j] == meshes[i]) {
        fe_set_error("fe_cg_solve_batched: mesh %d appears twice", i);
        return FE_ERR_INVALID;
      }
  }
  FeDeviceGuard device_guard;
  FE_CUDA(device_guard.set(meshes[0]->d.device), "cudaSetDevice");
  FE_CUDA(cudaStreamSynchronize((cudaStream_t)stream), "caller stream");
  const bool mixed = opts->mixed == FE_F32;
  FE_TRY(fe_batch_prepare());
  FeBatch B;
  FE_CUDA(cudaStreamCreateWithFlags(&B.st, cudaStreamNonBlocking), "batch stream");
  B.hp.resize(nprob);
  B.active.assign(nprob, 1);
  FE_CUDA(cudaMallocHost(&B.hsc, 2 * nprob * sizeof(CgScal)), "batch scalars");
  B.cap_hsc = 2 * nprob;
  std::vector<double> sb(nprob, 1.0);
  for (int i = 0; i < nprob; ++i) {
    CgWork* w = nullptr;
    FE_TRY(fe_cg_get_work(meshes[i], mixed, &w));
    FE_TRY(fe_ensure_geometry(meshes[i], FE_F64, false));
    if (mixed) FE_TRY(fe_ensure_geometry(meshes[i], FE_F32, false));
    FE_TRY(fe_cg_ensure_diag(meshes[i], w, FE_LAPLACE));
    // each problem scaled by its own exact power of two (fe_cg_rhs_scale), undone on x at the end
    const long long ncw = meshes[i]->ncw;
    FE_TRY(fe_cg_rhs_scale(w, b[i], ncw, &sb[i]));
    FE_TRY(fe_cg_scale(b[i], w->bs, sb[i], ncw, w->st));
    FE_TRY(fe_cg_scale(x[i], w->x, sb[i], ncw, w->st));
    FE_CUDA(cudaStreamSynchronize(w->st), "workspace set-up");
    FE_TRY(fe_batch_fill(&B, i, meshes[i], w, w->bs, opts));
  }
  B.any_flexible = (!mixed && opts->flexible) ? 1 : 0;
  FE_TRY(fe_batch_build(&B));
  FE_TRY(fe_batch_solve(&B, opts));
  FE_TRY(fe_batch_read(&B));
  fe_status worst = FE_OK;
  for (int i = 0; i < nprob; ++i) {
    FE_TRY(fe_cg_scale(B.hp[i].x64, x[i], 1.0 / sb[i], meshes[i]->ncw, B.st));
    const CgScal& o = B.hsc[2 * i];
    const CgScal& in = B.hsc[2 * i + 1];
    res[i].status = (fe_status)o.status;
    res[i].rel_res = o.relres;
    res[i].iters = mixed ? in.stall_total : o.iter;
    res[i].outer_iters = mixed ? o.iter : 1;
    if (o.status != FE_OK && worst == FE_OK) worst = (fe_status)o.status;
  }
  FE_CUDA(cudaStreamSynchronize(B.st), "batch synchronize");
  if (worst != FE_OK) fe_set_error("fe_cg_solve_batched: some problems did not converge");
  return worst;
}
