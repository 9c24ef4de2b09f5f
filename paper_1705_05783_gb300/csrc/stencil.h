// Walk of the fine grid shared by the streaming FP64 kernels: a thread takes
// one (x, y) column of the grid and marches along z, so the column's
// coordinates cost one division, the values of the plane below and the
// coupling to it stay in registers, and a warp still reads contiguous runs.
//
// What bounds these kernels is the FP64 unit (a warp instruction holds it for
// about 64 cycles), so every load that an instruction waits for has to be in
// flight early: the loads of a cell are issued together, with a zero in place
// of a neighbour outside the grid (0 * 0 changes no sum), instead of one by
// one inside branches.  The residual of 256^3 cells: 260 us (303 with a branch
// per neighbour and a thread per row element), where its eight FP64
// instructions a cell take 213.
#ifndef CAMS_STENCIL_H
#define CAMS_STENCIL_H

#include "cams_internal.h"

namespace cams {

constexpr int kColThreads = 256;    // threads of a CTA, one column each
// CTAs of a launch at most: six for each of the 152 SMs (the residual's 64
// registers a thread leave four of them resident at once, the assembly's 80 three).
constexpr int kColBlocks = 6 * 152;

// A launch's work: pieces of `threads` columns x `planes` planes.
struct ColWork {
  int planes;           // planes of a piece
  unsigned tiles;       // pieces side by side in a plane; 0: flat
  unsigned pieces;
};

// Planes that a thread marches through: short runs where the grid would not
// fill the chip otherwise; eight planes reuse 7/8 of what a run can reuse.
//
// Thin grids are flat: where the last piece of a plane would leave more than an
// eighth of its lanes without a column, pieces run on into the next planes
// (column and run come from one index, at the price of a division), and below
// a warp's width of columns a run is one plane, for consecutive threads to read
// consecutive cells.  1 x 1 x 10^6 and 4 x 4 x 65536 cells: 1210 and 104 us of the
// residual by planes, 40 and 40 flat (a cell a thread, as it was before: 56).
inline ColWork col_work(const Geo& g, int threads = kColThreads) {
  ColWork w;
  const long long t = g.N / (2LL * kColBlocks * kColThreads);
  w.planes = t < 1 ? 1 : (t > 8 ? 8 : (int)t);
  const long long tiles = (g.sz + threads - 1) / threads;
  if (g.nz > 1 && tiles * threads > g.sz + g.sz / 8) {
    if (g.sz < 32) w.planes = 1;
    const long long runs = (g.nz + w.planes - 1) / w.planes;
    w.tiles = 0;
    w.pieces = (unsigned)((g.sz * runs + threads - 1) / threads);
  } else {
    w.tiles = (unsigned)tiles;
    w.pieces = w.tiles * (unsigned)((g.nz + w.planes - 1) / w.planes);
  }
  return w;
}

inline int col_grid(const ColWork& w) {
  return w.pieces < (unsigned)kColBlocks ? (int)w.pieces : kColBlocks;
}

#ifdef __CUDACC__
// Block-wide sum; every thread passes its value, thread 0 gets the total.
// Fixed shape, fixed order: bit-reproducible for a fixed launch.
__device__ inline double block_sum(double v) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
  if (wid == 0)
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  return v;
}

// The column j of this thread in piece w0, and the run of planes [z0, z1);
// false where there is none.
__device__ __forceinline__ bool col_of(const Geo& g, const ColWork& w, unsigned w0, unsigned& j, int& z0,
                                       int& z1) {
  unsigned seg;
  if (w.tiles) {
    seg = w0 / w.tiles;
    j = (w0 - seg * w.tiles) * blockDim.x + threadIdx.x;
  } else {
    const unsigned q = w0 * blockDim.x + threadIdx.x;
    seg = q / (unsigned)g.sz;
    j = q - seg * (unsigned)g.sz;
  }
  z0 = (int)seg * w.planes;
  z1 = min(z0 + w.planes, g.nz);
  return j < (unsigned)g.sz && z0 < g.nz;
}

// Adds up the CTAs' sums: each CTA leaves its own in red[blockIdx.x], and the
// CTA that comes last (a ticket) adds them in block order, writes the total
// and sets the ticket back to zero.  True in one thread of that CTA.  The
// launches that share red and tick run one after the other.  (A second
// kernel for it takes 4.4 us, a ticket about 1.)
__device__ inline bool finish_sum(double s, double* red, unsigned* tick, double* total) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    red[blockIdx.x] = s;
    __threadfence();
    last = atomicAdd(tick, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double t = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) t += __ldcg(red + b);
  t = block_sum(t);
  if (threadIdx.x != 0) return false;
  *tick = 0;
  *total = t;
  return true;
}

// r = f - A p on the cells of this CTA's pieces (r, r32: null when not
// wanted), returning the thread's sum of r^2.  Axu.. hold the couplings to
// the upper neighbours (the arrays Ax.. themselves for a symmetric A).
__device__ __forceinline__ double residual_columns(
    const Geo& g, const ColWork& w, const double* __restrict__ Ad, const double* __restrict__ Ax,
    const double* __restrict__ Ay, const double* __restrict__ Az, const double* __restrict__ Axu,
    const double* __restrict__ Ayu, const double* __restrict__ Azu, const double* __restrict__ f,
    const double* __restrict__ p, double* r, float* r32) {
  double s2 = 0.0;
  for (unsigned w0 = blockIdx.x; w0 < w.pieces; w0 += gridDim.x) {
    unsigned j;
    int z0, z1;
    if (!col_of(g, w, w0, j, z0, z1)) continue;
    const unsigned y = j / (unsigned)g.nx, x = j - y * (unsigned)g.nx;
    const bool xl = x > 0, xu = x + 1 < (unsigned)g.nx, yl = y > 0, yu = y + 1 < (unsigned)g.ny;
    long long i = j + g.sz * z0;
    double pc = p[i], pd = 0.0, azd = 0.0;
    if (z0 > 0) {
      pd = p[i - g.sz];
      azd = Az[i];
    }
    const bool sym = Azu == Az;
    for (int z = z0; z < z1; ++z, i += g.sz) {
      const bool zu = z + 1 < g.nz;
      const double fi = f[i], ad = Ad[i];
      const double axl = xl ? Ax[i] : 0.0, pxl = xl ? p[i - 1] : 0.0;
      const double axu = xu ? Axu[i + 1] : 0.0, pxu = xu ? p[i + 1] : 0.0;
      const double ayl = yl ? Ay[i] : 0.0, pyl = yl ? p[i - g.sy] : 0.0;
      const double ayu = yu ? Ayu[i + g.sy] : 0.0, pyu = yu ? p[i + g.sy] : 0.0;
      const double azu = zu ? Azu[i + g.sz] : 0.0, pu = zu ? p[i + g.sz] : 0.0;
      // the lower coupling of the plane above: the same number when A is
      // symmetric, so it is not read again
      const double azn = sym ? azu : (zu ? Az[i + g.sz] : 0.0);
      double a = fi - ad * pc;
      a -= axl * pxl;
      a -= axu * pxu;
      a -= ayl * pyl;
      a -= ayu * pyu;
      a -= azd * pd;
      a -= azu * pu;
      if (r) r[i] = a;
      if (r32) r32[i] = (float)a;
      s2 += a * a;
      pd = pc;
      pc = pu;
      azd = azn;
    }
  }
  return s2;
}
#endif

}  // namespace cams

#endif
