// The cells of a local entity and the basis operator's entries, shared by the
// local solvers.
#pragma once

#include "cams_internal.h"

namespace cams {

namespace {

__device__ __forceinline__ double coupling(const Geo& g, const double* Abx, const double* Aby,
                                           const double* Abz, int d, long long i) {
  // A_b entry between i and i - e_d (stored at the upper cell)
  return d == 0 ? Abx[i] : (d == 1 ? Aby[i] : Abz[i]);
}

__device__ __forceinline__ long long gstride(const Geo& g, int d) {
  return d == 0 ? 1 : (d == 1 ? g.sy : g.sz);
}

__device__ __forceinline__ int gextent(const Geo& g, int d) {
  return d == 0 ? g.nx : (d == 1 ? g.ny : g.nz);
}

// global slot (bits over x,y,z) of the entity's r-th right-hand side
__device__ __forceinline__ int slot_of(int r, int free_mask) {
  int s = 0, k = 0;
  for (int d = 0; d < 3; ++d)
    if (free_mask & (1 << d)) {
      if (r & (1 << k)) s |= 1 << d;
      ++k;
    }
  return s;
}

struct Local {
  int c[3];        // coordinates
  long long i;     // global cell
};

__device__ __forceinline__ Local local_cell(const Entity& E, int l) {
  Local L;
  const int L0 = E.L[E.ord[0]], L1 = E.L[E.ord[1]];
  int t[3];
  t[0] = l % L0;
  t[1] = (l / L0) % L1;
  t[2] = l / (L0 * L1);
  for (int k = 0; k < 3; ++k) L.c[E.ord[k]] = E.org[E.ord[k]] + t[k];
  return L;
}

__device__ __forceinline__ int local_stride(const Entity& E, int d) {
  const int L0 = E.L[E.ord[0]], L1 = E.L[E.ord[1]];
  return d == E.ord[0] ? 1 : (d == E.ord[1] ? L0 : L0 * L1);
}

// The row of A_b at cell i, kept for the adaptive update's test.
__device__ __forceinline__ void snapshot_row(const Geo& g, const Local& c, long long i,
                                             const double* Abd, const double* Abx,
                                             const double* Aby, const double* Abz, double* snap) {
  snap[0 * g.N + i] = Abd[i];
  snap[1 * g.N + i] = c.c[0] > 0 ? Abx[i] : 0.0;
  snap[2 * g.N + i] = c.c[0] < g.nx - 1 ? Abx[i + 1] : 0.0;
  snap[3 * g.N + i] = c.c[1] > 0 ? Aby[i] : 0.0;
  snap[4 * g.N + i] = c.c[1] < g.ny - 1 ? Aby[i + g.sy] : 0.0;
  snap[5 * g.N + i] = c.c[2] > 0 ? Abz[i] : 0.0;
  snap[6 * g.N + i] = c.c[2] < g.nz - 1 ? Abz[i + g.sz] : 0.0;
}

}  // namespace

}  // namespace cams
