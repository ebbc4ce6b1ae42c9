// fe_vec.cuh -- shared pieces of the vector / reduction kernels.
#pragma once
#include "fe_apply_kernel.cuh"

fe_status fe_ensure_reduction(const fe_mesh* m);

// The assembled value of one cell-wise entry, gathered: the copies of its node in the neighbouring
// cells, summed as the structured passes do (z pairs, then y, then x; a pair's sum does not depend on
// its order), so the result is theirs bit for bit.  Cells below 2^32 / max(mx, my) (fe_dss_grid).
struct DssGrid {
  int mx, my, mz;
  unsigned rx, ry;  // floor(2^32 / m) + 1: exact quotients of the cell index by mx and my (0 for m = 1)
};
inline bool fe_dss_grid(const fe_mesh* m, DssGrid* g) {
  *g = {m->d.mx, m->d.my, m->d.mz, 0u, 0u};
  if (m->d.mx > 1) g->rx = (unsigned)((1ull << 32) / (unsigned)m->d.mx + 1);
  if (m->d.my > 1) g->ry = (unsigned)((1ull << 32) / (unsigned)m->d.my + 1);
  const long long big = m->d.mx > m->d.my ? m->d.mx : m->d.my;
  return m->ncells * big < (1ll << 32) && m->ncw < (1ll << 31);
}
template <class S, int N>
__device__ __forceinline__ S dss_gather(const S* v, int e, const DssGrid& g) {
  constexpr int P = N - 1, N2 = N * N, N3 = N2 * N;
  const unsigned cell = (unsigned)e / N3, f = (unsigned)e - cell * N3;
  const int k = f / N2, j = (f / N) % N, i = f % N;
  const unsigned row = g.rx ? __umulhi(cell, g.rx) : cell, cz = g.ry ? __umulhi(row, g.ry) : row;
  const int cx = (int)(cell - row * g.mx), cy = (int)(row - cz * g.my);
  // offset to the other copy of the node along an axis, 0 if there is none
  auto other = [](int c, int m, int l, int cstep, int nstep) {
    return l == 0 && c > 0 ? -cstep + P * nstep : (l == P && c + 1 < m ? cstep - P * nstep : 0);
  };
  const int ox = other(cx, g.mx, i, N3, 1), oy = other(cy, g.my, j, g.mx * N3, N),
            oz = other((int)cz, g.mz, k, g.mx * g.my * N3, N2);
  auto zsum = [&](int o) {
    S s = v[o];
    if (oz) s += v[o + oz];
    return s;
  };
  auto ysum = [&](int o) {
    S s = zsum(o);
    if (oy) s += zsum(o + oy);
    return s;
  };
  S s = ysum(e);
  if (ox) s += ysum(e + ox);
  return s;
}
