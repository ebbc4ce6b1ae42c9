// fe_apply_pair.cuh -- the FP64-accurate apply: double-word arithmetic on pairs of cells.
//
// The operator, its 1D tables and its tile modes are those of fe_apply_kernel.cuh; here a thread owns
// the same 1D line in two neighbouring cells of the tile (a pair: cells 2s and 2s+1 along x in a
// brick or a packed unit, consecutive cells otherwise), and every operation of the sweeps is one
// packed FP32 instruction on both (dw2 in fe_arith.h).  A tile element is 16 bytes, the high parts of
// both cells and then the low parts: one 128-bit shared-memory access moves the pair.
//
// FP64 accuracy.  Inputs stay binary64 until they are differenced (Laplace) or converted (mass);
// the CTA's values are scaled by a power of two (cta_exp_shift) so that every double-word value
// stays inside the float range.  The Laplace gradient is formed from differences of neighbouring
// nodal values: component a is B'_a (the derivative from the differences along axis a) followed by
// V along the two other axes, so every value the sweeps carry has the size of such a difference and
// the rounding of the sweeps does not meet the cancellation of the derivative of a smooth field.
#pragma once
#include "fe_apply_kernel.cuh"

// Launch and code shape per n = 2..8 [Laplace, mass], each the fastest of those measured (stored
// geometry, 7 to 17 million cell-wise DoFs, unassembled; before -> now is the kernel on single cells
// against this one, in ns per 1000 DoFs):
//   Laplace  n = 2 23.3 -> 22.1, 3 25.5 -> 20.2, 4 24.9 -> 19.6, 5 27.2 -> 23.7, 6 35.2 -> 30.4,
//            7 38.4 -> 32.4, 8 35.8 -> 29.6
//   mass     10.2 -> 7.6, 9.8 -> 7.3, 10.4 -> 7.6, 10.9 -> 8.9, 12.1 -> 11.2, 13.1 -> 12.2, 14.1 -> 11.4
// What bounds the Laplace kernels is the FP32 pipe together with what does not overlap it: at n = 4
// the double-word operations alone need 0.239 ms of the 0.328 ms of a 64^3 mesh, the bytes 0.158 ms.
struct PairTune {
  int minb;  // CTAs per SM of the register budget (one-layer kernel on consecutive cells)
  int zreg;  // 1: z-lines stay in registers between the phases; 0: every line through the tile
  int roll;  // output pairs per loop iteration of a contraction (0: unrolled, for the code's size)
  int pts;   // points per loop iteration of the pointwise phases (n where zreg or ahead need it)
  int ahead; // Laplace: load a point's metric one point ahead; mass: all of the z-line's at the start
};
template <int N, int OP>
__host__ __device__ constexpr PairTune pair_tune() {
  constexpr PairTune l[7] = {{4, 1, 0, 2, 0}, {5, 1, 0, 3, 1}, {6, 1, 0, 4, 0}, {5, 0, 2, 2, 0},
                             {2, 0, 1, 2, 0}, {2, 0, 3, 7, 1}, {4, 0, 2, 8, 1}};
  constexpr PairTune m[7] = {{8, 1, 0, 2, 1}, {9, 1, 0, 3, 1}, {8, 1, 0, 4, 1}, {5, 1, 2, 5, 1},
                             {2, 1, 3, 6, 1}, {3, 1, 2, 7, 0}, {6, 1, 1, 8, 0}};
  return OP == FE_LAPLACE ? l[N - 2] : m[N - 2];
}
// the register budget of the bricks and packed units (n = 2..4), whose layer loop and interface sums
// need more registers: at the one-layer budgets of n = 4 they spill (64^3 Laplace, assembled:
// 0.460 ms at 6 CTAs per SM, 0.416 at 5, 0.438 at 4)
template <int N, int OP, int MODE>
__host__ __device__ constexpr int pair_minb() {
  if constexpr (MODE == MODE_CELLS) {
    return pair_tune<N, OP>().minb;
  } else {
    constexpr int l[3] = {4, 5, 5}, m[3] = {8, 8, 6};
    return OP == FE_LAPLACE ? l[N - 2] : m[N - 2];
  }
}

// Tile of the pair kernel: NP pairs per CTA, N^2 threads per pair.  An element is 16 bytes, so a
// quarter warp (8 lanes) covers the 32 banks once; row, plane and pair strides (RS, PS, CS
// elements) are those with the fewest bank conflicts over the x-, y- and z-line accesses of all
// quarter warps (counted for the strides n..n+2, +0..7 of each).  For n = 4 the z-lines are given to
// the threads in another order (z_owner), which with CS = 4 mod 8 leaves no conflict at all.
template <int N>
struct PairStride;
template <> struct PairStride<2> { static constexpr int RS = 2, PS = 5, CS = 12; };
template <> struct PairStride<3> { static constexpr int RS = 3, PS = 12, CS = 41; };
template <> struct PairStride<4> { static constexpr int RS = 5, PS = 20, CS = 84; };
template <> struct PairStride<5> { static constexpr int RS = 5, PS = 29, CS = 145; };
template <> struct PairStride<6> { static constexpr int RS = 6, PS = 37, CS = 228; };
template <> struct PairStride<7> { static constexpr int RS = 7, PS = 49, CS = 343; };
template <> struct PairStride<8> { static constexpr int RS = 9, PS = 72, CS = 576; };
// Tile shapes: pairs of cells; the same with about a warp of threads per CTA; single cells (a
// thread's lines are those of one cell, in scalar double-word arithmetic, the same operations and
// bits).  The last two are for launches that leave the SMs part-empty (pair_shape).
enum { TILE_PAIRS = 0, TILE_PAIRS_SMALL = 1, TILE_SINGLE = 2 };
template <int N, int SHAPE = TILE_PAIRS>
struct PairCfg {
  static constexpr int N2 = N * N;
  static constexpr int N3 = N * N * N;
  static constexpr int RS = PairStride<N>::RS, PS = PairStride<N>::PS, CS = PairStride<N>::CS;
  static constexpr int W = SHAPE == TILE_SINGLE ? 1 : 2;  // cells per slot
  using V = typename std::conditional<W == 2, dw2, dw>::type;
  // slots (pairs or cells) per CTA: nearly whole warps of N^2 threads each
  static constexpr int NPS[3][7] = {{32, 14, 8, 5, 7, 5, 2}, {8, 3, 2, 1, 3, 1, 1}, {16, 7, 4, 5, 3, 5, 2}};
  static constexpr int NP = NPS[SHAPE][N - 2];
  static constexpr int CELLS = W * NP;
  static constexpr int THREADS = NP * N2;
  static constexpr int TILE = NP * CS;
  static constexpr int UPB = NP / 4;  // 2^3-packed storage units per CTA (4 pairs each)
};

// Pair slot and line coordinates of thread t: for the x- and y-lines consecutive threads walk the
// lines of a pair; for the z-lines of n = 4 a quarter warp takes a row of i of two neighbouring pairs.
struct LineOwner {
  int pl, la, lb;
};
template <int N>
__device__ __forceinline__ LineOwner xy_owner(int t) {
  const int pl = t / (N * N), lt = t - pl * (N * N), lb = lt / N;
  return {pl, lt - lb * N, lb};
}
template <int N>
__device__ __forceinline__ LineOwner z_owner(int t) {
  if constexpr (N == 4)
    return {((t >> 2) & 1) | ((t >> 4) & ~1), t & 3, (t >> 3) & 3};
  else
    return xy_owner<N>(t);
}
// bricks of assembled applies: BX x BY = 2 NP cells, BX even
template <int N>
struct PairBrick;
template <> struct PairBrick<2> { static constexpr int BX = 8, BY = 8; };
template <> struct PairBrick<3> { static constexpr int BX = 4, BY = 7; };
template <> struct PairBrick<4> { static constexpr int BX = 4, BY = 4; };

// Arrays of the tile: the three gradient components (Laplace; the binary64 inputs are differenced
// in the place of the first before it is written), or one (mass).
__host__ __device__ constexpr int pair_narr(int op) { return op == FE_LAPLACE ? 3 : 1; }
template <int N, int SHAPE = TILE_PAIRS>
constexpr size_t pair_smem_bytes(int op) {
  return (size_t)pair_narr(op) * PairCfg<N, SHAPE>::TILE * 8 * PairCfg<N, SHAPE>::W;
}

template <>
struct Sm<dw> {  // single cells: hi and lo interleaved, one 64-bit access per value
  float2* p;
  __device__ __forceinline__ Sm(unsigned char* base, int arr, int tile)
      : p(reinterpret_cast<float2*>(base) + (size_t)arr * tile) {}
  __device__ __forceinline__ dw get(int e) const {
    const float2 v = p[e];
    return {v.x, v.y};
  }
  __device__ __forceinline__ void put(int e, dw v) const { p[e] = make_float2(v.h, v.l); }
};

template <>
struct Sm<dw2> {
  ulonglong2* p;
  __device__ __forceinline__ Sm(unsigned char* base, int arr, int tile)
      : p(reinterpret_cast<ulonglong2*>(base) + (size_t)arr * tile) {}
  __device__ __forceinline__ dw2 get(int e) const {
    const ulonglong2 v = p[e];
    return {v.x, v.y};
  }
  __device__ __forceinline__ void put(int e, dw2 v) const { p[e] = make_ulonglong2(v.h, v.l); }
  // one cell's value of an element (lane 0 or 1)
  __device__ __forceinline__ dw get1(int e, int lane) const {
    const float* f = reinterpret_cast<const float*>(p + e) + lane;
    return {f[0], f[2]};
  }
  __device__ __forceinline__ void put1(int e, int lane, dw v) const {
    float* f = reinterpret_cast<float*>(p + e) + lane;
    f[0] = v.h;
    f[2] = v.l;
  }
};

// For n = 2 and 4 a warp owns whole pairs (8 and 2) in all three line directions, so the phases of
// a cell need no CTA barrier; otherwise the CTA's threads share the tile's pairs.
template <int N>
__host__ __device__ constexpr bool warp_tile() {
  return N == 2 || N == 4;
}
template <int N>
__device__ __forceinline__ void tile_sync() {
  if constexpr (warp_tile<N>())
    __syncwarp();
  else
    __syncthreads();
}

// Exponent shift of the FP64 path: the CTA's inputs enter the double-word arithmetic scaled by
// 2^-sh, sh = (binary exponent of the largest finite |x| of the CTA), and every output is scaled
// back by 2^sh.  Powers of two are exact, so the result is the same operator applied to x; the
// scaling keeps every intermediate double-word value (and its low part) inside the float range
// whatever the magnitude of x.  Scaled values below 2^-74 (of the CTA's largest) are flushed to
// zero.  The conversions below are for the exponents of ordinary data: `plain` is set when the CTA
// holds no infinity or NaN and |sh| <= 800, so that no difference overflows and no output leaves
// binary64's normal range; otherwise the general conversions (fe_arith.h) run.
struct ExpShift {
  int sh;
  bool plain;
  unsigned in_add;  // (-896 - sh) << 23: exponent field of a binary64 in the place of a float's
  unsigned in_min;  // high word of the smallest |x| that is not flushed
};
// All threads of the CTA call it; it holds a barrier.  Where a warp owns whole pairs and nothing is
// summed between pairs (WARP) the shift is the warp's own.
template <int N, bool WARP, int W>
__device__ __forceinline__ ExpShift cta_exp_shift(const double (&xr)[W][N]) {
  unsigned em = 0, all = 0;
#pragma unroll
  for (int c = 0; c < W; ++c)
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const unsigned e = ((unsigned)__double2hiint(xr[c][k]) >> 20) & 0x7FFu;
      em = max(em, e == 0x7FFu ? 0u : e);  // infinities and NaNs keep their own value
      all = max(all, e);
    }
  unsigned m, am;
  if constexpr (WARP) {
    __syncwarp();
    m = __reduce_max_sync(0xFFFFFFFFu, em);
    am = __reduce_max_sync(0xFFFFFFFFu, all);
  } else {
    __shared__ uint2 s_wmax[32];
    const unsigned warp = threadIdx.x >> 5;
    const unsigned lanes = min(32u, blockDim.x - warp * 32u);
    const unsigned lmask = lanes == 32u ? 0xFFFFFFFFu : ((1u << lanes) - 1u);
    em = __reduce_max_sync(lmask, em);
    all = __reduce_max_sync(lmask, all);
    if ((threadIdx.x & 31u) == 0u) s_wmax[warp] = make_uint2(em, all);
    __syncthreads();
    m = am = 0;
    const unsigned nw = (blockDim.x + 31u) >> 5;
    for (unsigned w = 0; w < nw; ++w) m = max(m, s_wmax[w].x), am = max(am, s_wmax[w].y);
  }
  ExpShift s;
  s.sh = (int)m - 1023;
  s.plain = am != 0x7FFu && s.sh >= -800 && s.sh <= 800;
  s.in_add = (unsigned)(-896 - s.sh) << 23;
  s.in_min = (unsigned)max(949 + s.sh, 1) << 20;
  return s;
}

// a slot's binary64 values, scaled by 2^-sh, as double-words
__device__ __forceinline__ dw2 lanes_of(const float (&h)[2], const float (&l)[2]) {
  return {f2_pack(h[0], h[1]), f2_pack(l[0], l[1])};
}
__device__ __forceinline__ dw lanes_of(const float (&h)[1], const float (&l)[1]) { return {h[0], l[0]}; }
static __device__ __noinline__ dw2 dw_from_doubles_general(double a, double b, int sh) {
  const dw x = dw_from_double_ftz(a, sh), y = dw_from_double_ftz(b, sh);
  return {f2_pack(x.h, y.h), f2_pack(x.l, y.l)};
}
static __device__ __noinline__ dw dw_from_doubles_general(double a, int sh) {
  return dw_from_double_ftz(a, sh);
}
// The same bits for finite values below 2^(sh + 2) (`plain`): per value, hi is the top 24 significand
// bits under the shifted exponent.  The 29 bits below become a float without an integer conversion
// (which would issue on the FP64 pipe): 6 bits under the exponent of 2^46 and 23 bits under that
// of 2^23, the biases removed by an exact subtraction and the sum, which rounds the 29 bits once;
// then the scale 2^(e-52) with the sign.
template <int W>
struct SplitBits {
  float hi[W], sc[W], m6[W], m23[W];
  __device__ __forceinline__ void set(int c, double v, const ExpShift& s) {
    const unsigned H = (unsigned)__double2hiint(v), L = (unsigned)__double2loint(v);
    const unsigned t = __funnelshift_l(L, H, 3) + s.in_add;
    const bool in = (H & 0x7FFFFFFFu) >= s.in_min;
    const unsigned h = (t & 0x7FFFFFFFu) | (H & 0x80000000u);
    sc[c] = __uint_as_float(in ? (h & 0xFF800000u) - (52u << 23) : 0u);
    hi[c] = __uint_as_float(in ? h : 0u);
    m6[c] = __uint_as_float(((L >> 23) & 0x3Fu) | 0x56800000u);
    m23[c] = __uint_as_float((L & 0x7FFFFFu) | 0x4B000000u);
  }
};
__device__ __forceinline__ dw2 dw_from_doubles(double a, double b, const ExpShift& s) {
  SplitBits<2> v;
  v.set(0, a, s);
  v.set(1, b, s);
  constexpr f2 BIAS = 0x5680000156800001ull;  // 2^46 + 2^23
  auto pack = [](const float (&x)[2]) { return f2_pack(x[0], x[1]); };
  return {pack(v.hi), f2_mul(f2_add(f2_sub(pack(v.m6), BIAS), pack(v.m23)), pack(v.sc))};
}
__device__ __forceinline__ dw dw_from_doubles(double a, const ExpShift& s) {
  SplitBits<1> v;
  v.set(0, a, s);
  const float lo = __fadd_rn(__fsub_rn(v.m6[0], __uint_as_float(0x56800001u)), v.m23[0]);
  return {v.hi[0], __fmul_rn(lo, v.sc[0])};
}

// (h + l) 2^sh as binary64, rounded once.  Where the CTA's inputs are `plain` and the parts finite (in_range)
// both are widened on the integer pipe, subnormal floats to zero, and one FP64 addition rounds; the rest goes
// out of line and gets the same bits wherever both are right, so that a cell's values do not depend on what
// else its tile holds.  Finite inputs can still overflow float on the way, in a metric beyond its range or
// in the sweeps, and an infinity or NaN then has to arrive as one.
__device__ __forceinline__ bool in_range(dw v) {
  const float inf = __uint_as_float(0x7F800000u);
  return fabsf(v.h) < inf && fabsf(v.l) < inf;
}
__device__ __forceinline__ double dw_to_double_plain(dw v, int sh) {
  const unsigned k = (unsigned)(896 + sh) << 20;
  auto wide = [&](float f) {
    const unsigned u = __float_as_uint(f);
    const bool zero = (u & 0x7F800000u) == 0u;
    const unsigned h = ((unsigned)((int)u >> 3) & 0x8FFFFFFFu) + k;
    return __hiloint2double(zero ? 0 : (int)h, zero ? 0 : (int)(u << 29));
  };
  return wide(v.h) + wide(v.l);
}
static __device__ __noinline__ double dw_to_double_general(dw v, int sh) {
  return scalbn(f2d_bits(v.h) + f2d_bits(v.l), sh);
}

// the two cells of pair slot pl of the tile at cell0 (cell_pos's tile modes)
struct PairPos {
  long long cell[2];
  int cx[2], cy[2], cz[2];
  bool act[2];
};
template <int N, int MODE, int W = 2, class A>
__device__ __forceinline__ PairPos pair_pos(const A& a, long long cell0, int pl) {
  using C = PairCfg<N>;
  PairPos c;
  if constexpr (MODE == MODE_PACKED) {
    const int ux_n = a.mx / 2, uy_n = a.my / 2;
    const long long u = cell0 + pl / 4;
    const int sub = pl % 4;  // sy + 2 sz
    c.cx[0] = (int)(u % ux_n) * 2;
    c.cy[0] = c.cy[1] = (int)((u / ux_n) % uy_n) * 2 + (sub & 1);
    c.cz[0] = c.cz[1] = (int)(u / ((long long)ux_n * uy_n)) * 2 + (sub >> 1);
    c.act[0] = c.act[1] = pl / 4 < C::UPB && u < a.ncells / 8;
    c.cx[1] = c.cx[0] + 1;
    c.cell[0] = ((long long)c.cz[0] * a.my + c.cy[0]) * a.mx + c.cx[0];
    c.cell[1] = c.cell[0] + 1;
  } else if constexpr (MODE == MODE_BRICK || MODE == MODE_BRICKZ) {  // brick index < 2^31
    constexpr int BX = PairBrick<N>::BX, BY = PairBrick<N>::BY, BP = BX / 2;
    const unsigned nbx = (unsigned)(a.mx + BX - 1) / BX, nby = (unsigned)(a.my + BY - 1) / BY;
    const unsigned b = (unsigned)cell0, rb = b / nbx;
    c.cx[0] = (int)(b - rb * nbx) * BX + 2 * (pl % BP);
    c.cx[1] = c.cx[0] + 1;
    c.cy[0] = c.cy[1] = (int)(rb % nby) * BY + pl / BP;
    c.cz[0] = c.cz[1] = (int)(rb / nby);
    c.act[0] = c.cx[0] < a.mx && c.cy[0] < a.my;
    c.act[1] = c.cx[1] < a.mx && c.cy[0] < a.my;
    c.cell[0] = ((long long)c.cz[0] * a.my + c.cy[0]) * a.mx + c.cx[0];
    c.cell[1] = c.cell[0] + 1;
  } else {  // cell coordinates only where the Dirichlet masks need them (64-bit divisions)
#pragma unroll
    for (int l = 0; l < W; ++l) {
      c.cell[l] = cell0 + W * pl + l;
      c.act[l] = c.cell[l] < a.ncells;
      c.cx[l] = c.cy[l] = c.cz[l] = 0;
      if (a.dirichlet && c.act[l]) {
        c.cx[l] = (int)(c.cell[l] % a.mx);
        c.cy[l] = (int)((c.cell[l] / a.mx) % a.my);
        c.cz[l] = (int)(c.cell[l] / ((long long)a.mx * a.my));
      }
    }
  }
  return c;
}

// Intra-brick interface sums on the output tile s (all threads of the CTA call it): x-interfaces
// inside a pair (cell 0 | cell 1) and between a pair and the next, at (j, k) = (la, lb); then the
// y-interfaces between pair rows at (i, k) = (la, lb).
template <int N, class A>
__device__ __forceinline__ void pair_brick_sums(const Sm<dw2>& s, const A& a, long long cell0) {
  using C = PairCfg<N>;
  const LineOwner o = xy_owner<N>(threadIdx.x);
  const int pl = o.pl, la = o.la, lb = o.lb, cb = pl * C::CS;
  constexpr int BP = PairBrick<N>::BX / 2, BY = PairBrick<N>::BY;
  const PairPos c = pair_pos<N, MODE_BRICK>(a, cell0, pl);  // recomputed: nothing held across sweeps
  const int e0 = cb + lb * C::PS + la * C::RS, eN = e0 + N - 1;
  if (c.act[1]) {
    const dw v = dw_add(s.get1(eN, 0), s.get1(e0, 1));
    s.put1(eN, 0, v);
    s.put1(e0, 1, v);
    if (pl % BP < BP - 1 && c.cx[1] + 1 < a.mx) {
      const dw w = dw_add(s.get1(eN, 1), s.get1(e0 + C::CS, 0));
      s.put1(eN, 1, w);
      s.put1(e0 + C::CS, 0, w);
    }
  }
  __syncthreads();
  if (c.act[0] && pl / BP < BY - 1 && c.cy[0] + 1 < a.my) {
    const int eL = cb + lb * C::PS + (N - 1) * C::RS + la;
    const int eR = cb + BP * C::CS + lb * C::PS + la;
    const dw2 v = dw2_add(s.get(eL), s.get(eR));
    s.put(eL, v);
    s.put(eR, v);
  }
  __syncthreads();
}

// MODE_BRICKZ state of a pair (ZCarry of both cells)
struct ZCarry2 {
  double top[2];
  bool pending, last;
};

// in-place 1D sweep of the thread's line (base, stride) of s
template <int N, int SIG, int RU, class V>
__device__ __forceinline__ void pair_sweep(const Sm<V>& s, int base, int st, const EO<N, V>& M) {
  V in[N];
#pragma unroll
  for (int r = 0; r < N; ++r) in[r] = s.get(base + r * st);
  eo_line<N, V, SIG, RU>(M, in, [&](int q, V v) { s.put(base + q * st, v); });
}

// The tile at cell0, applied by the CTA's PairCfg<N>::THREADS threads.
template <int N, int OP, int GEOM, int MODE, int SHAPE = TILE_PAIRS, bool CG = false>
__device__ __forceinline__ void apply_pairs(const CellArgs<N, typename PairCfg<N, SHAPE>::V>& a,
                                            const Tab1D<N, typename PairCfg<N, SHAPE>::V>& tab,
                                            long long cell0, unsigned char* smraw,
                                            ZCarry2* zc = nullptr, const CgApply* cg = nullptr) {
  static_assert(SHAPE != TILE_SINGLE || MODE == MODE_CELLS, "single cells: consecutive cells only");
  static_assert(!CG || SHAPE == TILE_SINGLE, "fused CG iteration: where single cells are taken");
  using C = PairCfg<N, SHAPE>;
  using V = typename C::V;
  using T = NT<V>;
  constexpr int W = C::W;
  constexpr int N2 = C::N2, N3 = C::N3, RS = C::RS, PS = C::PS;
  constexpr PairTune TU = pair_tune<N, OP>();
  constexpr bool ZREG = TU.zreg != 0;
  constexpr int RU = TU.roll, MU = TU.pts;
  const Sm<V> s0(smraw, 0, C::TILE);
  const Sm<V> s1(smraw, OP == FE_LAPLACE ? 1 : 0, C::TILE);
  const Sm<V> s2(smraw, OP == FE_LAPLACE ? 2 : 0, C::TILE);

  // line starts in the tile: x-line (j=la, k=lb), y-line (i=la, k=lb) of the thread's xy lines;
  // z-line (i=la, j=lb) of its z-lines, whose pair and coordinates are pl, la, lb from here on
  int bx, by;
  {
    const LineOwner o = xy_owner<N>(threadIdx.x);
    bx = o.pl * C::CS + o.lb * PS + o.la * RS;
    by = o.pl * C::CS + o.lb * PS + o.la;
  }
  const LineOwner zo = z_owner<N>(threadIdx.x);
  const int pl = zo.pl, la = zo.la, lb = zo.lb, lt = lb * N + la;
  const int bz = pl * C::CS + lb * RS + la;

  // masked(c, k): node k of cell c's z-line lies on a Dirichlet face (bits 0-2 per cell: the whole
  // line, its bottom node, its top node); act: cell c exists
  unsigned mask = 0;
  bool act[W];
  long long cell[W];
  {
    const PairPos pos = pair_pos<N, MODE, W>(a, cell0, pl);
#pragma unroll
    for (int c = 0; c < W; ++c) {
      act[c] = pos.act[c];
      cell[c] = pos.cell[c];
      if (a.dirichlet && act[c]) {
        const int cx = pos.cx[c], cy = pos.cy[c], cz = pos.cz[c];
        if ((cx == 0 && la == 0) || (cx == a.mx - 1 && la == N - 1) || (cy == 0 && lb == 0) ||
            (cy == a.my - 1 && lb == N - 1))
          mask |= 1u << (3 * c);
        if ((a.dirichlet & FE_DIR_ZLO) && cz == 0) mask |= 2u << (3 * c);
        if ((a.dirichlet & FE_DIR_ZHI) && cz == a.mz - 1) mask |= 4u << (3 * c);
      }
    }
  }
  auto masked = [&](int c, int k) {
    const unsigned b = mask >> (3 * c);
    return (b & 1u) != 0u || (k == 0 && (b & 2u)) || (k == N - 1 && (b & 4u));
  };

  // ---- inputs (z-line owner, coalesced), binary64
  auto xaddr = [&](int c, int k) -> long long {
    if constexpr (MODE == MODE_PACKED) {
      constexpr int P = Packed<N>::P, NU = Packed<N>::NU;
      const int sub = pl % 4;
      return (cell0 + pl / 4) * Packed<N>::NU3 +
             ((long long)((sub >> 1) * P + k) * NU + (sub & 1) * P + lb) * NU + c * P + la;
    } else {
      return cell[c] * N3 + k * N2 + lt;
    }
  };
  double xr[W][N];
#pragma unroll
  for (int c = 0; c < W; ++c)
#pragma unroll
    for (int k = 0; k < N; ++k)
      xr[c][k] = act[c] && !masked(c, k) ? __ldcs(a.x + xaddr(c, k)) : 0.0;
  if constexpr (CG) {  // fused CG iteration: p := z + beta p on the way in (0 at masked nodes)
    const double beta = cg->sc->beta;
    const double* z = static_cast<const double*>(cg->z);
    double* p = const_cast<double*>(a.x);
#pragma unroll
    for (int c = 0; c < W; ++c)
#pragma unroll
      for (int k = 0; k < N; ++k)
        if (act[c] && !masked(c, k)) {
          xr[c][k] = z[xaddr(c, k)] + beta * xr[c][k];
          p[xaddr(c, k)] = xr[c][k];
        }
  }

  // metric of component comp at point k of the z-lines: planes of high and of low parts per cell; a
  // cell that does not exist reads the tile's first one (its values multiply zeros)
  const float* g[W];
#pragma unroll
  for (int c = 0; c < W; ++c) {
    const long long gc = act[c] ? cell[c] : pair_pos<N, MODE, W>(a, cell0, 0).cell[0];
    g[c] = reinterpret_cast<const float*>(a.geo) + (size_t)(gc - a.geo_cell0) * (FE_GEO_COMPS * 2 * N3) + lt;
  }
  auto metric = [&](int comp, int k) -> V {
    const int o = comp * 2 * N3 + k * N2;
    float h[W], l[W];
#pragma unroll
    for (int c = 0; c < W; ++c) h[c] = __ldcs(g[c] + o), l[c] = __ldcs(g[c] + o + N3);
    return lanes_of(h, l);
  };
  constexpr bool STORED = GEOM == GEOM_STORED_K;
  constexpr bool PREF_M = OP == FE_MASS && STORED && TU.ahead != 0;
  V jpre[PREF_M ? N : 1];
  if constexpr (PREF_M) {
#pragma unroll
    for (int k = 0; k < N; ++k) jpre[k] = metric(6, k);
  }
  // the metric of the next point (the first one's is loaded before the last V sweep)
  constexpr bool AHEAD = OP == FE_LAPLACE && STORED && TU.ahead != 0;
  V next[AHEAD ? 6 : 1];
  ExpShift es = {};
  // v[c][r], a line's values per cell -> out[r]
  auto to_lanes = [&](const auto& v, auto& out) {
    constexpr int M = sizeof(out) / sizeof(out[0]);
    if (es.plain) {  // uniform over the CTA
#pragma unroll
      for (int r = 0; r < M; ++r) {
        if constexpr (W == 2)
          out[r] = dw_from_doubles(v[0][r], v[1][r], es);
        else
          out[r] = dw_from_doubles(v[0][r], es);
      }
    } else {
#pragma unroll
      for (int r = 0; r < M; ++r) {
        if constexpr (W == 2)
          out[r] = dw_from_doubles_general(v[0][r], v[1][r], es.sh);
        else
          out[r] = dw_from_doubles_general(v[0][r], es.sh);
      }
    }
  };
  if constexpr (OP == FE_LAPLACE) {
    // ---- reference gradient at the Gauss points: s1, s2, s0 = d/dx, d/dy, d/dz
    struct alignas(8 * W) Raw {
      double v[W];
    };
    Raw* raw = reinterpret_cast<Raw*>(smraw);  // the inputs, in the place of s0
#pragma unroll
    for (int k = 0; k < N; ++k) {
      Raw r;
#pragma unroll
      for (int c = 0; c < W; ++c) r.v[c] = xr[c][k];
      raw[bz + k * PS] = r;
    }
    es = cta_exp_shift<N, warp_tile<N>() && MODE == MODE_CELLS, W>(xr);  // its barrier publishes raw
    // B' along x, y and z (in place: z-lines are the thread's own, and the others have been read); an
    // axis loop, not unrolled, keeps the code within the instruction cache
#pragma unroll 1
    for (int ax = 0; ax < 3; ++ax) {
      if (ax == 2) tile_sync<N>();
      const int base = ax == 0 ? bx : (ax == 1 ? by : bz), st = ax == 0 ? 1 : (ax == 1 ? RS : PS);
      const Sm<V> o = ax == 0 ? s1 : (ax == 1 ? s2 : s0);
      double dd[W][N - 1];
      Raw prev = raw[base];
#pragma unroll
      for (int r = 0; r < N - 1; ++r) {
        const Raw cur = raw[base + (r + 1) * st];
#pragma unroll
        for (int c = 0; c < W; ++c) dd[c][r] = cur.v[c] - prev.v[c];
        prev = cur;
      }
      V d[N - 1];
      to_lanes(dd, d);
      eob_line<N, V, RU>(tab.eB, d, [&](int q, V v) { o.put(base + q * st, v); });
    }
    // V along the other axes: s1, s2 along z; s0 along x, s1 along y, s2 along x; s0 along y
#pragma unroll 1
    for (int ax = 0; ax < (AHEAD ? 5 : 6); ++ax) {
      if (ax == 2 || ax == 5) tile_sync<N>();
      const Sm<V> o = (ax == 0 || ax == 3) ? s1 : ((ax == 1 || ax == 4) ? s2 : s0);
      const int base = ax < 2 ? bz : ((ax == 2 || ax == 4) ? bx : by);
      const int st = ax < 2 ? PS : ((ax == 2 || ax == 4) ? 1 : RS);
      pair_sweep<N, 1, RU>(o, base, st, tab.eV);
    }
    if constexpr (AHEAD) {
      tile_sync<N>();
#pragma unroll
      for (int c = 0; c < 6; ++c) next[c] = metric(c, 0);
      pair_sweep<N, 1, RU>(s0, by, RS, tab.eV);
    }
    tile_sync<N>();
    // ---- pointwise metric (z-line owner): (gx, gy, gz) = G grad u
    V u[ZREG ? N : 1];
#pragma unroll(MU)
    for (int k = 0; k < N; ++k) {
      const int e = bz + k * PS;
      const V dx = s1.get(e), dy = s2.get(e), dz = s0.get(e);
      V gx, gy, gz;
      if constexpr (STORED) {
        V G[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          G[c] = AHEAD ? next[AHEAD ? c : 0] : metric(c, k);
          if (AHEAD && k + 1 < N) next[AHEAD ? c : 0] = metric(c, k + 1);
        }
        const V xx = G[0], yy = G[1], zz = G[2], xy = G[3], xz = G[4], yz = G[5];
        gx = T::mac(T::mac(T::prod(xx, dx), xy, dy), xz, dz);
        gy = T::mac(T::mac(T::prod(xy, dx), yy, dy), yz, dz);
        gz = T::mac(T::mac(T::prod(xz, dx), yz, dy), zz, dz);
      } else {
        const V wq = T::mul(T::mul(tab.W_[la], tab.W_[lb]), tab.W_[k]);
        gx = T::mul(T::mul(wq, a.aff[0]), dx);
        gy = T::mul(T::mul(wq, a.aff[1]), dy);
        gz = T::mul(T::mul(wq, a.aff[2]), dz);
      }
      s1.put(e, gx);
      s2.put(e, gy);
      if constexpr (ZREG)
        u[k] = gz;
      else
        s0.put(e, gz);
    }
    tile_sync<N>();
    // ---- transposed derivatives, each in place; their sum on the z-lines
#pragma unroll 1
    for (int ax = 0; ax < (ZREG ? 2 : 3); ++ax)
      pair_sweep<N, -1, RU>(ax == 0 ? s1 : (ax == 1 ? s2 : s0), ax == 0 ? bx : (ax == 1 ? by : bz),
                            ax == 0 ? 1 : (ax == 1 ? RS : PS), tab.eDT);
    if constexpr (ZREG) {
      V w[N];
      eo_regs<N, V, -1>(tab.eDT, u, w);
      tile_sync<N>();
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int e = bz + k * PS;
        u[k] = T::add(T::add(w[k], s1.get(e)), s2.get(e));
      }
      eo_line<N, V, 1, RU>(tab.eVT, u, [&](int q, V v) { s0.put(bz + q * PS, v); });
    } else {
      tile_sync<N>();
#pragma unroll(MU)
      for (int k = 0; k < N; ++k) {
        const int e = bz + k * PS;
        s0.put(e, T::add(T::add(s0.get(e), s1.get(e)), s2.get(e)));
      }
    }
  } else {
    // ---- mass: values at the Gauss points, times w detJ
    es = cta_exp_shift<N, warp_tile<N>() && MODE == MODE_CELLS, W>(xr);
    {
      V u[N];
      to_lanes(xr, u);
      eo_line<N, V, 1, RU>(tab.eV, u, [&](int q, V v) { s0.put(bz + q * PS, v); });
    }
#pragma unroll 1
    for (int ax = 0; ax < 2; ++ax) {
      tile_sync<N>();
      pair_sweep<N, 1, RU>(s0, ax == 0 ? bx : by, ax == 0 ? 1 : RS, tab.eV);
    }
    tile_sync<N>();
    V u[ZREG ? N : 1];
#pragma unroll(MU)
    for (int k = 0; k < N; ++k) {
      const int e = bz + k * PS;
      V jw;
      if constexpr (!STORED)
        jw = T::mul(T::mul(T::mul(tab.W_[la], tab.W_[lb]), tab.W_[k]), a.aff[3]);
      else if constexpr (PREF_M)
        jw = jpre[PREF_M ? k : 0];
      else
        jw = metric(6, k);
      const V v = T::mul(jw, s0.get(e));
      if constexpr (ZREG)
        u[k] = v;
      else
        s0.put(e, v);
    }
    if constexpr (ZREG) eo_line<N, V, 1, RU>(tab.eVT, u, [&](int q, V v) { s0.put(bz + q * PS, v); });
  }

  // ---- transposed interpolation: z (done above from registers if ZREG), x and y in the tile
#pragma unroll 1
  for (int ax = ZREG ? 1 : 0; ax < 3; ++ax) {
    if (ax > 0) tile_sync<N>();
    pair_sweep<N, 1, RU>(s0, ax == 0 ? bz : (ax == 1 ? bx : by), ax == 0 ? PS : (ax == 1 ? 1 : RS),
                         tab.eVT);
  }
  tile_sync<N>();

  // ---- outputs, binary64
  auto out = [&](V v, int k, double (&q)[W]) {
    dw x[W];
    if constexpr (W == 2) {
      const float2 h = f2_unpack(v.h), l = f2_unpack(v.l);
      x[0] = {h.x, l.x};
      x[1] = {h.y, l.y};
    } else {
      x[0] = v;
    }
    bool plain = es.plain;
#pragma unroll
    for (int c = 0; c < W; ++c) {
      if (masked(c, k)) x[c] = {0.0f, 0.0f};
      plain = plain && in_range(x[c]);
    }
#pragma unroll
    for (int c = 0; c < W; ++c)
      q[c] = plain ? dw_to_double_plain(x[c], es.sh) : dw_to_double_general(x[c], es.sh);
  };
  if constexpr (MODE != MODE_CELLS && warp_tile<N>()) __syncthreads();
  if constexpr (MODE == MODE_BRICK || MODE == MODE_BRICKZ) pair_brick_sums<N>(s0, a, cell0);
  if constexpr (MODE == MODE_BRICKZ) {
    // The z-interface with the previous layer of the chunk: the structured DSS's z-pass pair sum
    // (lower + upper copy), formed on the stored values, so the result is that of the pass.
    // The x/y sums inside the brick came first, as they do before the pass.
    double qb[W], qt[W];
    out(s0.get(bz), 0, qb);
    out(s0.get(bz + (N - 1) * PS), N - 1, qt);
#pragma unroll
    for (int c = 0; c < W; ++c) {
      if (!act[c]) continue;
      double* y = a.y + cell[c] * N3 + lt;
      double bottom = qb[c];
      if (zc->pending) {
        bottom = zc->top[c] + bottom;
        __stcs(y - (long long)a.mx * a.my * N3 + (N - 1) * N2, bottom);
      }
      __stcs(y, bottom);
      if (zc->last)
        __stcs(y + (N - 1) * N2, qt[c]);
      else
        zc->top[c] = qt[c];
    }
#pragma unroll
    for (int k = 1; k < N - 1; ++k) {
      double q[W];
      out(s0.get(bz + k * PS), k, q);
#pragma unroll
      for (int c = 0; c < W; ++c)
        if (act[c]) __stcs(a.y + cell[c] * N3 + lt + k * N2, q[c]);
    }
    zc->pending = !zc->last;
    return;
  }
  if constexpr (MODE == MODE_PACKED) {
    // unit-internal assembly: sum the copies on the x-, y- and z-interfaces between the unit's
    // sub-cells in the tile (as the structured DSS passes do, z then y then x), then every stored
    // node is written once, by the sub-cell with the lowest index along each axis that holds it
    constexpr int P = Packed<N>::P, NU = Packed<N>::NU;
    const int sub = pl % 4, sy = sub & 1, sz = sub >> 1;
    auto pair_sum = [&](int eL, int eR) {
      const dw2 v = dw2_add(s0.get(eL), s0.get(eR));
      s0.put(eL, v);
      s0.put(eR, v);
    };
    if (act[0] && sz == 0)  // z-interface: (k = P of sz 0) + (k = 0 of sz 1), thread (i, j)
      pair_sum(bz + P * PS, bz + 2 * C::CS);
    __syncthreads();
    const int plx = xy_owner<N>(threadIdx.x).pl;
    const bool actx = pair_pos<N, MODE, W>(a, cell0, plx).act[0];
    if (actx && (plx & 1) == 0)  // y-interface, thread (i, k) = (la, lb)
      pair_sum(by + P * RS, by + C::CS);
    __syncthreads();
    if (actx) {  // x-interface between the pair's cells, thread (j, k) = (la, lb)
      const dw v = dw_add(s0.get1(bx + P, 0), s0.get1(bx, 1));
      s0.put1(bx + P, 0, v);
      s0.put1(bx, 1, v);
    }
    __syncthreads();
    if (act[0] && (sy == 0 || lb > 0)) {
      double* yu = a.y + (cell0 + pl / 4) * Packed<N>::NU3 + (long long)(sy * P + lb) * NU + la;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        if (sz == 1 && k == 0) continue;
        double q[W];
        out(s0.get(bz + k * PS), k, q);
#pragma unroll
        for (int c = 0; c < W; ++c)
          if (c == 0 || la > 0) __stcs(yu + (long long)(sz * P + k) * NU * NU + c * P, q[c]);
      }
    }
    return;
  }
  // two points per iteration from n = 5 on, so that one's conversion covers the other's branch and store: Q4
  // 40^3 mass 73.8 -> 73.1 us, Q5 32^3 82.3 -> 81.4, Q7 32^3 190.1 -> 189.0; at n = 3 and 4 one is faster (Laplace
  // Q2 64^3 145.3 against 146.8, Q3 64^3 328.8 against 331.2)
  constexpr int OUT = N >= 5 ? 2 : 1;
  Acc<double> qp;
#pragma unroll(OUT)
  for (int k = 0; k < N; ++k) {
    double q[W];
    out(s0.get(bz + k * PS), k, q);
#pragma unroll
    for (int c = 0; c < W; ++c) {
      if (!act[c]) continue;
      const long long e = cell[c] * N3 + lt + k * N2;
      __stcs(a.y + e, q[c]);
      if constexpr (CG) qp.add_prod(q[c], *(volatile const double*)(a.x + e));
    }
  }
  if constexpr (CG) cg_finish_apply(*cg, qp);
}

template <int N, int OP, int GEOM, int MODE, int SHAPE, bool CG>
__global__ void __launch_bounds__(PairCfg<N, SHAPE>::THREADS,
                                  (SHAPE == TILE_PAIRS
                                       ? pair_minb<N, OP, MODE>()
                                       : 512 / ((PairCfg<N, SHAPE>::THREADS + 31) / 32 * 32)))
    k_apply_pair(const __grid_constant__ ApplyArgs<N, typename PairCfg<N, SHAPE>::V> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (a.skip && *(volatile const int*)a.skip) return;  // uniform over the grid
  long long cell0;
  if constexpr (MODE == MODE_BRICK)
    cell0 = (long long)blockIdx.x;
  else if constexpr (MODE == MODE_PACKED)
    cell0 = (long long)blockIdx.x * PairCfg<N>::UPB;
  else
    cell0 = a.c.cell_base + (long long)blockIdx.x * PairCfg<N, SHAPE>::CELLS;
  apply_pairs<N, OP, GEOM, MODE, SHAPE, CG>(a.c, a.tab, cell0, smraw, nullptr, &a.cg);
}

// Tile shape of a launch on consecutive cells.  A lone warp on a scheduler runs the packed
// arithmetic at the pace of its issue, two cycles an instruction, and then takes twice as long for two
// cells as for one: up to 16 warps of single cells per SM those are faster (measured, 8^3 cells,
// single against pairs: n = 8 16.2 against 18.7 us, n = 6 12.1 against 13.2, n = 4 7.0 against 7.3;
// 12^3 cells, 37 warps per SM, n = 7: 32.5 against 29.1).  Above, the small pair tile where the busiest
// of the SMs has fewer warps to work through with it, in a launch of at most four ordinary CTAs per SM.
inline bool pair_single(long long cells, int n, int sms) { return cells * n * n <= 16LL * 32 * sms; }
template <int N>
inline int pair_shape(long long cells, int sms) {
  using L = PairCfg<N>;
  using S = PairCfg<N, TILE_PAIRS_SMALL>;
  if (pair_single(cells, N, sms)) return TILE_SINGLE;
  const long long pairs = (cells + 1) / 2;
  auto busiest = [&](int np, int threads) {
    return ((pairs + np - 1) / np + sms - 1) / sms * ((threads + 31) / 32);
  };
  return pairs <= 4LL * sms * L::NP && busiest(S::NP, S::THREADS) < busiest(L::NP, L::THREADS)
             ? TILE_PAIRS_SMALL
             : TILE_PAIRS;
}

// MODE_BRICKZ: blockIdx.x = chunk * (bricks per layer) + brick column; the CTA applies the layers
// [z0, z1) of its column one after the other
template <int N, int OP, int GEOM>
__global__ void __launch_bounds__(PairCfg<N>::THREADS, (pair_minb<N, OP, MODE_BRICKZ>()))
    k_apply_pair_zcarry(const __grid_constant__ ApplyArgs<N, dw2> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (a.skip && *(volatile const int*)a.skip) return;  // uniform over the grid
  constexpr int BX = PairBrick<N>::BX, BY = PairBrick<N>::BY;
  const unsigned per_layer =
      (unsigned)((a.c.mx + BX - 1) / BX) * (unsigned)((a.c.my + BY - 1) / BY);
  const unsigned col = blockIdx.x % per_layer, chunk = blockIdx.x / per_layer;
  const int z0 = (int)chunk * a.zchunk;
  const int z1 = z0 + a.zchunk < a.c.mz ? z0 + a.zchunk : a.c.mz;
  ZCarry2 zc;
  zc.pending = false;
  for (int cz = z0; cz < z1; ++cz) {
    zc.last = cz == z1 - 1;
    apply_pairs<N, OP, GEOM, MODE_BRICKZ>(a.c, a.tab, (long long)cz * per_layer + col, smraw, &zc);
    __syncthreads();  // the next layer refills the tile
  }
}
