// fe_recompute.cuh -- metric terms formed on the fly from cell-wise nodal coordinates
// (FE_GEOM_RECOMPUTE).
//
// Sec. 2.3 defines the isoparametric map of a cell through its GLL-node coordinates; the
// Laplace apply needs G = w detJ J^-1 J^-T and the mass apply w detJ at every Gauss point.
// In the recompute mode only the coordinates are kept in HBM (3 values per cell node).  The apply
// walks the mesh in chunks of cells: k_recompute forms the metric of one chunk into a scratch buffer
// and the stored-metric apply consumes it right away.
//
// The coordinates are stored as offsets from the cell's first node: the derivative sums then
// work on values of the size of the cell rather than of the domain, and do not cancel.
// J is obtained as in a collocated gradient: interpolation to the Gauss points along z, y, x, then the
// Gauss-point derivative along each direction.  The threads own lines (N^2 per cell, or per pair of
// cells in packed double-word arithmetic), so every contraction is the even-odd form of the apply with
// coefficients at compile-time offsets.  One thread per point instead, each with its own row of the
// full matrices, reads two thirds of its coefficients at lane-dependent constant addresses, which are
// served one by one, and cannot use packed instructions.  Laplace, FP64, both in chunks of 48 MB: Q3
// 48^3 0.653 -> 0.496 ms (0.037 of that by the stored-metric apply), Q7 24^3 1.036 -> 0.707; FP32 Q4
// 40^3 0.351 -> 0.205 (0.405, 0.595 and 0.164 ms with the present chunks).  At Q3 the FP32 pipe is 70%
// busy, with about 540 operations per point in the sweeps and 430 in the Laplace metric.
#pragma once
#include "fe_apply_pair.cuh"

// slots (cells, or pairs of cells) per CTA, three threads per line (one per coordinate), and CTAs per SM
// of the register budget
template <int N, class V>
struct RecCfg {
  using P = PairStride<N>;
  static constexpr int N2 = N * N, N3 = N2 * N;
  static constexpr int W = std::is_same<V, dw2>::value ? 2 : 1;  // cells per slot
  static constexpr int NPS[7] = {16, 7, 4, 2, 2, 1, 1}, MINBS[7] = {4, 4, 3, 3, 2, 3, 2};
  static constexpr int NP = NPS[N - 2], MINB = MINBS[N - 2];
  static constexpr int CELLS = W * NP, LINES = NP * N2, THREADS = 3 * LINES, TILE = NP * P::CS;
  static constexpr size_t SMEM = (size_t)9 * TILE * sizeof(V);
  static constexpr size_t POINT_BYTES = sizeof(V) / W;  // a metric value of the scratch
};

// a coordinate's type, per arithmetic
template <class V>
struct RV {
  using GV = typename NT<V>::GV;
};
template <>
struct RV<dw2> {
  using GV = float2;  // the halves of a double-word value side by side
};

// The plain product instead of the even-odd form: in single values (binary64, FP32) its operations cost
// no more and its error is smaller (FP32 Q4, relative l2: 5.1e-7 against 7.8e-7); in double-word
// values at n = 3 and 5, where the even-odd form saves little (Laplace, 64^3 and 40^3, one thread per
// line: 0.471 against 0.486 ms, 0.650 against 0.719) and its error is the larger one (l2 3.6e-14
// against 3.3e-14, 7.0e-14 against 5.7e-14; at n = 6: 1.0e-13 both, 0.677 against 0.830 ms).
template <int N, class V>
__host__ __device__ constexpr bool rec_direct() {
  constexpr bool DW = std::is_same<V, dw2>::value || std::is_same<V, dw>::value;
  return !DW || N == 3 || N == 5;
}
template <int N, class V, bool DIRECT = rec_direct<N, V>()>
struct RecomputeTab {
  EO<N, V> V_, D_;
  V W_[N];
};
template <int N, class V>
struct RecomputeTab<N, V, true> {
  typename NT<V>::CV V_[N][N], D_[N][N];
  V W_[N];
};
template <int N, class V>
struct RecomputeArgs {
  const typename RV<V>::GV* xyz;  // [cell][3][N3] offsets from the cell's first node
  typename NT<V>::GV* geo;        // [cell - cell0][7][N3]; double-word: planes of high and low parts
  long long cell0, cell_end;
  const int* skip;
  RecomputeTab<N, V> tab;
};

template <class V>
__device__ __forceinline__ V tile_get(const V* p) {
  return *p;
}
template <>
__device__ __forceinline__ dw2 tile_get<dw2>(const dw2* p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return {v.x, v.y};
}
template <class V>
__device__ __forceinline__ void tile_put(V* p, V v) {
  *p = v;
}
template <>
__device__ __forceinline__ void tile_put<dw2>(dw2* p, dw2 v) {
  *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.h, v.l);
}

// out = M in, normalised
template <int N, class V, int SIG, class M>
__device__ __forceinline__ void rec_line(const M& m, const V (&in)[N], V (&out)[N]) {
  using T = NT<V>;
  if constexpr (rec_direct<N, V>()) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      auto acc = T::prod(m[q][0], in[0]);
#pragma unroll
      for (int r = 1; r < N; ++r) acc = T::mac(acc, m[q][r], in[r]);
      out[q] = T::fin(T::keep(acc));
    }
  } else {
    eo_regs<N, V, SIG>(m, in, out);
#pragma unroll
    for (int q = 0; q < N; ++q) out[q] = T::fin(out[q]);
  }
}

template <int N, class V, int OP>
__global__ void __launch_bounds__(RecCfg<N, V>::THREADS, RecCfg<N, V>::MINB)
    k_recompute(const __grid_constant__ RecomputeArgs<N, V> a) {
  using G = RecCfg<N, V>;
  using T = NT<V>;
  constexpr int N2 = G::N2, N3 = G::N3, W = G::W;
  constexpr int RS = G::P::RS, PS = G::P::PS;
  extern __shared__ __align__(16) unsigned char smraw[];
  if (a.skip && *(volatile const int*)a.skip) return;
  // coordinate (component) d of the thread's lines; of the tile's arrays: the coordinates, d/dz in the
  // end; d/dx; d/dy
  const int d = threadIdx.x / G::LINES, t = threadIdx.x - d * G::LINES;
  V* const sz = reinterpret_cast<V*>(smraw);
  V* const s = sz + d * G::TILE;
  V* const sx = sz + 3 * G::TILE;
  V* const sy = sz + 6 * G::TILE;
  // warps own whole slots in all three directions
  constexpr bool WARP = warp_tile<N>() && G::LINES % 32 == 0;
  auto sync = [] {
    if constexpr (WARP)
      __syncwarp();
    else
      __syncthreads();
  };

  int bx, by;
  {
    const LineOwner o = xy_owner<N>(t);
    bx = o.pl * G::P::CS + o.lb * PS + o.la * RS;
    by = o.pl * G::P::CS + o.lb * PS + o.la;
  }
  const LineOwner zo = z_owner<N>(t);
  const int lt = zo.lb * N + zo.la;
  const int bz = zo.pl * G::P::CS + zo.lb * RS + zo.la;
  const long long cell = a.cell0 + (long long)blockIdx.x * G::CELLS + (long long)zo.pl * W;
  bool act[W];
#pragma unroll
  for (int c = 0; c < W; ++c) act[c] = cell + c < a.cell_end;

  V in[N], out[N];
  // interpolation to the Gauss points along z, y and x, the x-line's derivative with the last
#pragma unroll
  for (int k = 0; k < N; ++k) {
    typename RV<V>::GV g[W];
#pragma unroll
    for (int c = 0; c < W; ++c) {
      g[c] = {};
      if (act[c]) g[c] = __ldcs(a.xyz + (size_t)(cell + c) * (3 * N3) + d * N3 + k * N2 + lt);
    }
    if constexpr (W == 2)
      in[k] = {f2_pack(g[0].x, g[1].x), f2_pack(g[0].y, g[1].y)};
    else if constexpr (std::is_same<V, dw>::value)
      in[k] = {g[0].x, g[0].y};
    else
      in[k] = g[0];
  }
  rec_line<N, V, 1>(a.tab.V_, in, out);
#pragma unroll
  for (int k = 0; k < N; ++k) tile_put(s + bz + k * PS, out[k]);
  sync();
#pragma unroll
  for (int r = 0; r < N; ++r) in[r] = tile_get(s + by + r * RS);
  rec_line<N, V, 1>(a.tab.V_, in, out);
#pragma unroll
  for (int r = 0; r < N; ++r) tile_put(s + by + r * RS, out[r]);
  sync();
#pragma unroll
  for (int r = 0; r < N; ++r) in[r] = tile_get(s + bx + r);
  rec_line<N, V, 1>(a.tab.V_, in, out);
#pragma unroll
  for (int r = 0; r < N; ++r) tile_put(s + bx + r, out[r]);
  rec_line<N, V, -1>(a.tab.D_, out, in);
#pragma unroll
  for (int r = 0; r < N; ++r) tile_put(sx + d * G::TILE + bx + r, in[r]);
  sync();
#pragma unroll
  for (int r = 0; r < N; ++r) in[r] = tile_get(s + by + r * RS);
  rec_line<N, V, -1>(a.tab.D_, in, out);
#pragma unroll
  for (int r = 0; r < N; ++r) tile_put(sy + d * G::TILE + by + r * RS, out[r]);
#pragma unroll
  for (int k = 0; k < N; ++k) in[k] = tile_get(s + bz + k * PS);
  rec_line<N, V, -1>(a.tab.D_, in, out);
  sync();  // the coordinates have been read
#pragma unroll
  for (int k = 0; k < N; ++k) tile_put(s + bz + k * PS, out[k]);
  __syncthreads();

  const V wij = T::mul(a.tab.W_[zo.la], a.tab.W_[zo.lb]);
  // the metric of the z-line's points, shared between the line's three threads
#pragma unroll 1
  for (int k = d; k < N; k += 3) {
    V J[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      J[c][0] = tile_get(sx + c * G::TILE + bz + k * PS);
      J[c][1] = tile_get(sy + c * G::TILE + bz + k * PS);
      J[c][2] = tile_get(sz + c * G::TILE + bz + k * PS);
    }
    auto put = [&](int comp, V v) {
      const size_t first = (size_t)(cell - a.cell0) * FE_GEO_COMPS + comp;
      float* g = reinterpret_cast<float*>(a.geo) + first * (2 * N3) + k * N2 + lt;
      if constexpr (W == 2) {
        const float2 h = f2_unpack(v.h), l = f2_unpack(v.l);
        if (act[0]) g[0] = h.x, g[N3] = l.x;
        g += FE_GEO_COMPS * 2 * N3;
        if (act[1]) g[0] = h.y, g[N3] = l.y;
      } else if constexpr (std::is_same<V, dw>::value) {
        if (act[0]) g[0] = v.h, g[N3] = v.l;
      } else {
        if (act[0]) a.geo[first * N3 + k * N2 + lt] = v;
      }
    };
    // p q - r s
    auto dp = [](V p, V q, V r, V s) { return T::fin(T::mac(T::prod(p, q), T::neg(r), s)); };
    auto dot = [](V p0, V q0, V p1, V q1, V p2, V q2) {
      return T::fin(T::mac(T::mac(T::prod(p0, q0), p1, q1), p2, q2));
    };
    // first column of the adjugate, enough for the determinant
    const V A00 = dp(J[1][1], J[2][2], J[1][2], J[2][1]);
    const V A10 = dp(J[1][2], J[2][0], J[1][0], J[2][2]);
    const V A20 = dp(J[1][0], J[2][1], J[1][1], J[2][0]);
    const V det = dot(J[0][0], A00, J[0][1], A10, J[0][2], A20);
    const V w3 = T::mul(wij, a.tab.W_[k]);
    if constexpr (OP == FE_MASS) {
      put(6, T::mul(w3, det));
    } else {
      // G = w detJ J^-1 J^-T = (w / detJ) adj(J) adj(J)^T
      const V A01 = dp(J[0][2], J[2][1], J[0][1], J[2][2]);
      const V A11 = dp(J[0][0], J[2][2], J[0][2], J[2][0]);
      const V A21 = dp(J[0][1], J[2][0], J[0][0], J[2][1]);
      const V A02 = dp(J[0][1], J[1][2], J[0][2], J[1][1]);
      const V A12 = dp(J[0][2], J[1][0], J[0][0], J[1][2]);
      const V A22 = dp(J[0][0], J[1][1], J[0][1], J[1][0]);
      const V sc = T::mul(w3, T::recip(det));
      put(0, T::mul(sc, dot(A00, A00, A01, A01, A02, A02)));
      put(1, T::mul(sc, dot(A10, A10, A11, A11, A12, A12)));
      put(2, T::mul(sc, dot(A20, A20, A21, A21, A22, A22)));
      put(3, T::mul(sc, dot(A00, A10, A01, A11, A02, A12)));
      put(4, T::mul(sc, dot(A00, A20, A01, A21, A02, A22)));
      put(5, T::mul(sc, dot(A10, A20, A11, A21, A12, A22)));
    }
  }
}
