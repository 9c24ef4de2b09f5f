// Local basis solves in panels (the entities of k_basis.cu: banded SPD
// systems M P = B of n cells, half-width m, up to 8 right-hand sides).
//
// One CTA solves one entity by a left-looking banded L D L^T, kPB columns at a
// time.  A panel is the rows k .. k + m + kPB - 1 of its columns plus 8 rows
// for the right-hand sides (eliminated like rows of the matrix: their entries
// divided by the pivots are D^{-1} L^{-1} B).  Four lanes hold a row, lane pt
// the columns 4 j + pt, in registers from the first product to the last:
//   1. the entries of M (at most four a column, kept per cell);
//   2. minus the products with the previous m columns, from a ring of columns
//      of L in shared memory (a load of the row's entry and one 16-byte load
//      of the panel rows' entries, times d, for four FMAs); a tile of 8 rows
//      starts at the first column that reaches it, so the band's empty
//      triangle costs nothing;
//   3. the panel's own pivots, one barrier each: the 16 diagonal rows publish
//      the next column and its reciprocal pivot, every row scales its entry,
//      hands it to its four lanes and updates its later columns.
// The columns go to the ring and, panel by panel, to the CTA's slice of global
// scratch (L2) for the backward substitution, which takes kPB rows at a time:
// 16 columns x 8 right-hand sides, one thread each, the next panel copied
// ahead (cp.async).
//
// What bounds it: in FP64 the FP64 unit (91% busy on 9^3 interiors, 73% on 9 x 9 x 4;
// a warp instruction holds it for about 64 cycles, so lanes without work cost as much as others), in FP32
// the instructions issued (66% of the cycles).  The right-looking kernel
// (k_basis.cu) reads and writes the whole trailing window in shared memory for
// every 8 pivots, divides in the pivots' chain, and leaves half of the FP64
// units without lanes.  All levels of a build, right-looking -> panels:
//   FP32: 10^6 cells, 10^3 blocks 3.36 -> 1.71 ms; 80^3, 8^3 1.29 -> 0.63;
//         100x100x50, 10x10x5 1.24 -> 0.50; 64^3, 2x8x8 0.56 -> 0.25;
//         flat 100x100, 5x5 0.040 -> 0.031
//   FP64: 14.1 -> 9.5; 4.03 -> 2.77; 2.83 -> 1.89
// In FP64 a level whose half-widths are all below 16 stays with the per-pivot
// kernel: 16 columns a panel are mostly outside such a band, and the faces of
// 10x10x5 blocks (half-width 9) took 360 us here.
#include "cams_internal.h"
#include "entity.h"
#include "rcp64.h"

namespace cams {

namespace {

constexpr int kPB = 16;       // columns of a panel
constexpr int kRhs = 8;       // rows for the right-hand sides
constexpr int kPanelWarps = 8;

__host__ __device__ inline int round16(int x) { return (x + 15) & ~15; }
// columns the ring holds; rows of a column (the right-hand sides' after the
// m + kPB band rows), with a stride that puts 4 columns x 8 rows on different
// banks; rows of the ring of solutions
__host__ __device__ inline int ring_cols(int m) { return m < 16 ? 16 : round16(m); }
__host__ __device__ inline int ring_stride(int m) {
  const int rows = m + kPB + kRhs;
  return rows + ((8 - rows) & 15);
}
__host__ __device__ inline int panel_tiles(int m) { return 1 + (kPB + m + 7) / 8; }
__host__ __device__ inline int panel_elems(int m) {
  const int R = ring_cols(m);
  const int fwd = R * (ring_stride(m) + kPB);
  const int bwd = 2 * (m + kPB) * kPB + (R + kPB) * kRhs;
  return (fwd > bwd ? fwd : bwd) + R + kPB * kPB + kPB * 4 + 2 * kPB * kRhs;
}

// the place of panel column c among the four lanes' registers: lane c & 3,
// register c >> 2
__device__ __forceinline__ int perm16(int c) { return (c & 3) * 4 + (c >> 2); }

__device__ __forceinline__ float pivot_inverse(float d, bool& bad) {
  bad = !(d > 0.f) || !isfinite(d);
  return bad ? 1.f : __frcp_rn(d);
}
__device__ __forceinline__ double pivot_inverse(double d, bool& bad) {
  const long long b = __double_as_longlong(d);
  bad = !(b > 0 && b < 0x7FF0000000000000LL);
  return rcp_halley(bad ? 1.0 : d);
}

__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void load4(const double* p, double (&v)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void store4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(double* p, const double (&v)[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src) : "memory");
}

// Cell l's part of M and B: the diagonal, the couplings to the upper
// neighbours inside the box, and one right-hand side per corner vertex.
template <class T>
__device__ void build_cell(const Geo& g, const Entity& E, int l, T* cell, T* y, const double* Abd,
                           const double* Abx, const double* Aby, const double* Abz, const T* P) {
  const Local c = local_cell(E, l);
  const long long i = c.c[0] + g.sy * c.c[1] + g.sz * c.c[2];
  T rhs[kRhs];
#pragma unroll
  for (int r = 0; r < kRhs; ++r) rhs[r] = T(0);
  double diag = Abd[i];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int n_d = gextent(g, d);
    T upper = T(0);
    if (n_d > 1) {
      const long long sd = gstride(g, d);
      const bool has_lo = c.c[d] > 0, has_up = c.c[d] < n_d - 1;
      if (!(E.free_mask & (1 << d))) {
        // lattice direction: neighbours are one level higher -> lumped
        diag += has_lo ? coupling(g, Abx, Aby, Abz, d, i) : 0.0;
        diag += has_up ? coupling(g, Abx, Aby, Abz, d, i + sd) : 0.0;
      } else {
        // free direction: inside the box -> band entry; outside -> known data
        if (c.c[d] < E.org[d] + E.L[d] - 1) {
          upper = T(coupling(g, Abx, Aby, Abz, d, i + sd));
        } else if (has_up) {
          const T a = T(coupling(g, Abx, Aby, Abz, d, i + sd));
#pragma unroll
          for (int r = 0; r < kRhs; ++r) {
            const int s = slot_of(r, E.free_mask);
            if (r < E.nrhs && (s & (1 << d))) rhs[r] -= a * P[(long long)(s & ~(1 << d)) * g.N + i + sd];
          }
        }
        if (c.c[d] == E.org[d] && has_lo) {
          const T a = T(coupling(g, Abx, Aby, Abz, d, i));
#pragma unroll
          for (int r = 0; r < kRhs; ++r) {
            const int s = slot_of(r, E.free_mask);
            if (r < E.nrhs && !(s & (1 << d))) rhs[r] -= a * P[(long long)s * g.N + i - sd];
          }
        }
      }
    }
    cell[1 + d] = upper;
  }
  cell[0] = T(diag);
#pragma unroll
  for (int r = 0; r < kRhs; ++r) y[r] = rhs[r];
}

// NT: tiles of 8 rows a warp holds at most.
template <class T, int NT>
constexpr int kPanelCtas = NT == 4 ? 1 : (sizeof(T) == 4 ? 4 : (NT == 1 ? 3 : 2));
template <class T, int NT>
__global__ void __launch_bounds__(32 * kPanelWarps, kPanelCtas<T, NT>) k_entity_panel(
    Geo g, const Entity* __restrict__ ents, int count, const unsigned char* __restrict__ flag,
    int adaptive, const double* __restrict__ Abd, const double* __restrict__ Abx,
    const double* __restrict__ Aby, const double* __restrict__ Abz, T* P, double* snap, T* lscratch,
    long long lstride, int* status, unsigned* next) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ T rinv[kPB];
  __shared__ unsigned s_e;
  const int tid = threadIdx.x, nt = blockDim.x, nw = nt >> 5, lane = tid & 31, warp = tid >> 5;
  const int rl = lane >> 2, pt = lane & 3;
  T* const Lp = lscratch + (long long)blockIdx.x * lstride;
  // entities in the order that CTAs come free (their sizes differ by up to
  // eight); who solves an entity makes no difference to its result.  The last
  // draw sets the counter back.
  for (;;) {
    if (tid == 0) s_e = atomicAdd(next, 1u);
    __syncthreads();
    const unsigned e = s_e;
    __syncthreads();
    if (e >= (unsigned)count) {
      if (tid == 0 && e == (unsigned)count + gridDim.x - 1) *next = 0;
      break;
    }
    if (flag && !flag[e]) continue;
    const Entity E = ents[e];
    const int n = E.n, m = E.m, np = (n + kPB - 1) / kPB, n16 = np * kPB;
    const int R = ring_cols(m), CS = ring_stride(m), rows = m + kPB, tiles = panel_tiles(m);
    T* const ab = reinterpret_cast<T*>(sm_raw);   // 4 entries of M a panel column
    T* const yb = ab + 4 * kPB;                   // the panel's right-hand sides
    T* const ps = yb + kPB * kRhs;                // partial sums (backward)
    T* const colb = ps + kPB * kRhs;              // published pivot columns
    T* const dcol = colb + kPB * kPB;             // pivots of the ring's columns
    T* const ring = dcol + R;                     // R columns of L, stride CS
    T* const Tc = ring + R * CS;                  // d_j l_{k+c,j}, 16 a ring column
    T* const Yg = Lp + (long long)n16 * rows;     // global: right-hand sides, then solutions
    T* const Mg = Yg + (long long)n16 * kRhs;     // global: M's entries, 4 a cell
    int st[3];                                    // distance in l of the upper neighbour
#pragma unroll
    for (int d = 0; d < 3; ++d) st[d] = E.L[d] > 1 ? local_stride(E, d) : -1 - rows;
    for (int l = tid; l < n16; l += nt) {
      if (l < n) {
        build_cell<T>(g, E, l, Mg + 4 * l, Yg + (long long)kRhs * l, Abd, Abx, Aby, Abz, P);
      } else {                                    // rows past the end: the identity
        for (int q = 0; q < 4; ++q) Mg[4 * l + q] = q == 0 ? T(1) : T(0);
        for (int r = 0; r < kRhs; ++r) Yg[(long long)kRhs * l + r] = T(0);
      }
    }
    for (int t = tid; t < R * CS; t += nt) ring[t] = T(0);
    for (int t = tid; t < R; t += nt) dcol[t] = T(0);
    __syncthreads();
    // the panel's inputs: 64 entries of M and 128 of B, at most 2 a thread
    auto input = [&](int k, int t) { return t < 4 * kPB ? Mg[4 * k + t] : Yg[(long long)kRhs * k + t - 4 * kPB]; };
    for (int t = tid; t < kPB * (4 + kRhs); t += nt) ab[t] = input(0, t);
    int kslot = 0, kpos = 0;                      // k modulo the ring's columns and rows
    for (int k = 0; k < n; k += kPB) {
      // --- d_j l_{k+c,j} of the ring's columns j ---
      for (int t = tid; t < R * kPB; t += nt) {
        const int s = t / kPB, c = t % kPB;
        int pos = kpos + c, back = kslot - s;     // column j = k - back
        if (pos >= rows) pos -= rows;
        if (back <= 0) back += R;
        // (past the band's edge the place may hold another row)
        Tc[s * kPB + perm16(c)] = back + c <= m ? dcol[s] * ring[s * CS + pos] : T(0);
      }
      __syncthreads();
      // --- my tiles: entries of M (or B) minus the previous columns' products ---
      T v[NT][4];
      int row[NT];                                // first row of the tile; < 0: the right-hand sides
#pragma unroll
      for (int it = 0; it < NT; ++it) {
        // long and short tiles in turn, so that the warps' sums are alike
        const int t = it % 2 == 0 ? it * nw + warp : (it + 1) * nw - 1 - warp;
        row[it] = t == 0 ? -1 : (t < tiles ? 8 * (t - 1) : rows + 8);
        if (t >= tiles) continue;
        const int r = row[it] + rl;
        int pos;
        if (t == 0) {
          pos = rows + rl;
#pragma unroll
          for (int j = 0; j < 4; ++j) v[it][j] = yb[(4 * j + pt) * kRhs + rl];
        } else {
          pos = kpos + r;
          if (pos >= rows) pos -= rows;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int c = 4 * j + pt, df = r - c;
            T a[4];
            load4(ab + 4 * c, a);
            v[it][j] = df == 0 ? a[0] : (df == st[0] ? a[1] : (df == st[1] ? a[2] : (df == st[2] ? a[3] : T(0))));
          }
        }
        // columns j0 .. k - 1 (j0 a multiple of 4: the ring never wraps inside
        // four; what it adds below the band's edge is zero)
        int j0 = k - m + (t == 0 ? 0 : row[it]);
        j0 = j0 < 0 ? 0 : j0 & ~3;
        int s = j0 % R;
        for (int j = j0; j < k; j += 4) {
          const T* rp = ring + s * CS + pos;
          const T* tp = Tc + s * kPB + 4 * pt;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const T l = rp[u * CS];
            T cv[4];
            load4(tp + u * kPB, cv);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) v[it][jj] -= l * cv[jj];
          }
          s += 4;
          if (s == R) s = 0;
        }
      }
      T pre[2] = {T(0), T(0)};
      if (k + kPB < n) {
        pre[0] = tid < kPB * (4 + kRhs) ? input(k + kPB, tid) : T(0);
        pre[1] = tid + nt < kPB * (4 + kRhs) ? input(k + kPB, tid + nt) : T(0);
      }
      // --- the panel's pivots ---
      // column q of the diagonal rows, a = this lane's entry of it, and the
      // pivot's inverse, for step q
      auto publish = [&](int q, int it, T a) {
        const int r = row[it] + rl;
        if (pt != (q & 3) || r < q) return;
        colb[q * kPB + perm16(r)] = a;
        if (r == q) {
          bool bad;
          rinv[q] = pivot_inverse(a, bad);
          dcol[kslot + q] = bad ? T(1) : a;
          if (bad) atomicOr(status, kStatSingular);
        }
      };
#pragma unroll
      for (int it = 0; it < NT; ++it)
        if (row[it] >= 0 && row[it] < kPB) publish(0, it, v[it][0]);
      // (with several tiles a warp four steps share a body, the register of
      // column q being q / 4: unrolled, the sixteen miss the instruction cache)
#pragma unroll
      for (int jq = 0; jq < 4; ++jq) {
#pragma unroll(NT == 1 ? 4 : 1)
        for (int ql = 0; ql < 4; ++ql) {
          const int q = 4 * jq + ql;
          __syncthreads();
          const T ri = rinv[q];
          T cv[4], lq[NT];
          load4(colb + q * kPB + 4 * pt, cv);
#pragma unroll
          for (int it = 0; it < NT; ++it) {
            lq[it] = T(0);
            // (uniform) no tile; below the band's edge in this column; rows of
            // the diagonal block above the pivot
            const int r0 = row[it];
            if (r0 >= kPB ? r0 > m + q : (r0 >= 0 && r0 + 7 <= q)) continue;
            T l = v[it][jq] * ri;
            l = __shfl_sync(0xffffffffu, l, (lane & ~3) | ql);
            if (r0 >= 0 && r0 + rl <= q) l = T(0);               // this row is final
            else if (pt == ql) v[it][jq] = l;
            lq[it] = l;
            // the next pivot's column first
            if (pt > ql) v[it][jq] -= l * cv[jq];
            if (jq < 3 && ql == 3) v[it][(jq + 1) & 3] -= l * cv[(jq + 1) & 3];
            if (r0 >= 0 && r0 < kPB && q + 1 < kPB)
              publish(q + 1, it, ql == 3 ? v[it][(jq + 1) & 3] : v[it][jq]);
          }
#pragma unroll
          for (int it = 0; it < NT; ++it) {
            if (row[it] >= kPB ? row[it] > m + q : (row[it] >= 0 && row[it] + 7 <= q)) continue;
#pragma unroll
            for (int j = jq + 1; j < 4; ++j)
              if (j > jq + 1 || ql < 3) v[it][j] -= lq[it] * cv[j];
          }
        }
      }
      // --- to the ring, and the scratch of the backward substitution ---
#pragma unroll
      for (int it = 0; it < NT; ++it) {
        if (row[it] > rows) continue;
        const int r = row[it] + rl;
        if (row[it] < 0) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            ring[(kslot + 4 * j + pt) * CS + rows + rl] = v[it][j];
            Yg[(long long)(k + 4 * j + pt) * kRhs + rl] = v[it][j];
          }
        } else if (r < rows) {
          int pos = kpos + r;
          if (pos >= rows) pos -= rows;
          // no later panel needs the diagonal rows: their places are the
          // zeros past the band of the rows to come
#pragma unroll
          for (int j = 0; j < 4; ++j) ring[(kslot + 4 * j + pt) * CS + pos] = r < kPB ? T(0) : v[it][j];
          store4(Lp + ((long long)k * rows + (long long)r * kPB + 4 * pt), v[it]);
        }
      }
      if (tid < kPB * (4 + kRhs)) ab[tid] = pre[0];
      if (tid + nt < kPB * (4 + kRhs)) ab[tid + nt] = pre[1];
      kslot += kPB;
      if (kslot == R) kslot = 0;
      kpos += kPB;
      if (kpos >= rows) kpos -= rows;
      __syncthreads();
    }
    // --- backward substitution with L^T, a panel at a time ---
    T* const LB = ring;                           // two panels of L
    T* const X = LB + 2 * rows * kPB;             // ring of solutions, Rx rows
    const int Rx = R + kPB, pv = rows * kPB * (int)sizeof(T) / 16;
    for (int t = tid; t < Rx * kRhs; t += nt) X[t] = T(0);
    auto fetch = [&](int p) {
      unsigned char* dst = reinterpret_cast<unsigned char*>(LB + (p & 1) * rows * kPB);
      const unsigned char* src = reinterpret_cast<const unsigned char*>(Lp + (long long)p * rows * kPB);
      for (int t = tid; t < pv; t += nt) copy16(dst + 16 * t, src + 16 * t);
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(np - 1);
    // thread: column c of the panel, right-hand side rh, every parts-th row
    const int c = tid & 15, rh = (tid >> 4) & 7, part = tid >> 7, parts = nt >> 7;
    const int pc = perm16(c);
    for (int p = np - 1; p >= 0; --p) {
      const int k = p * kPB, kx = k % Rx;
      const T* L = LB + (p & 1) * rows * kPB;
      T x = T(0);
      if (part == 0) x = Yg[(long long)(k + c) * kRhs + rh];
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (p > 0) fetch(p - 1);
      T s = T(0);
      if (part < parts) {
#pragma unroll 4
        for (int r = kPB + part; r < rows; r += parts) {
          int pos = kx + r;
          if (pos >= Rx) pos -= Rx;
          s += L[r * kPB + pc] * X[pos * kRhs + rh];
        }
      }
      if (parts > 1) {
        if (part == 1) ps[tid - 128] = s;
        __syncthreads();
        if (part == 0) s += ps[tid];
      }
      if (part == 0) {
        x -= s;
#pragma unroll
        for (int q = kPB - 1; q > 0; --q) {
          const T xq = __shfl_sync(0xffffffffu, x, (lane & 16) | q);
          if (c < q) x -= L[q * kPB + pc] * xq;
        }
        int pos = kx + c;
        if (pos >= Rx) pos -= Rx;
        X[pos * kRhs + rh] = x;
        Yg[(long long)(k + c) * kRhs + rh] = x;
      }
    }
    __syncthreads();
    // write the basis values (slots on lattice bits stay zero)
    for (int l = tid; l < n; l += nt) {
      const Local lc = local_cell(E, l);
      const long long i = lc.c[0] + g.sy * lc.c[1] + g.sz * lc.c[2];
      for (int s = 0; s < 8; ++s) {
        const bool on = !(s & ~E.free_mask);
        int r = 0, b = 0;                         // the slot's right-hand side
        for (int d = 0; d < 3; ++d)
          if (E.free_mask & (1 << d)) r |= ((s >> d) & 1) << b++;
        P[(long long)s * g.N + i] = on ? Yg[(long long)kRhs * l + r] : T(0);
      }
      if (adaptive) snapshot_row(g, lc, i, Abd, Abx, Aby, Abz, snap);
    }
    __syncthreads();
  }
}

}  // namespace

// Elements of a CTA's global scratch slice for one entity.
long long entity_panel_scratch(const Entity& E) {
  const long long n16 = round16(E.n);
  return (n16 * (E.m + kPB + kRhs + 4) + 31) / 32 * 32;
}

int entity_panel_smem(int m, bool single) {
  return panel_elems(m) * (int)(single ? sizeof(float) : sizeof(double));
}

// 0: the half-width is beyond the kernel's tiles
int entity_panel_threads(int m) {
  const int tiles = panel_tiles(m);
  if (tiles > 4 * kPanelWarps) return 0;
  const int per = tiles <= kPanelWarps ? 1 : (tiles <= 2 * kPanelWarps ? 2 : 4);
  const int w = (tiles + per - 1) / per;
  return 32 * (w < 4 ? 4 : w);
}

template <class T>
static auto panel_kernel(int tiles) {
  return tiles <= kPanelWarps ? k_entity_panel<T, 1>
                              : (tiles <= 2 * kPanelWarps ? k_entity_panel<T, 2> : k_entity_panel<T, 4>);
}

cudaError_t set_entity_panel_smem(int m, bool single) {
  const int tiles = panel_tiles(m), smem = entity_panel_smem(m, single);
  return single ? raise_smem_limit(panel_kernel<float>(tiles), smem)
                : raise_smem_limit(panel_kernel<double>(tiles), smem);
}

template <class T>
static cudaError_t panel_launch(const Geo& g, const Entity* ents, const unsigned char* flag, int count,
                                int m, int grid, long long lstride, int adaptive, T* P, Buffers& b,
                                cudaStream_t s) {
  const int tiles = panel_tiles(m), threads = entity_panel_threads(m);
  const int smem = entity_panel_smem(m, sizeof(T) == 4);
  panel_kernel<T>(tiles)<<<grid < count ? grid : count, threads, smem, s>>>(
      g, ents, count, flag, adaptive, b.Abd, b.Abx, b.Aby, b.Abz, P, b.snap,
      reinterpret_cast<T*>(b.lscratch), lstride, b.status,
      b.tick + 1);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_entity_panel(const Geo& g, const Entity* ents, const unsigned char* flag, int count,
                                int m, int grid, long long lstride, int adaptive, bool single,
                                Buffers& b, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  return single ? panel_launch<float>(g, ents, flag, count, m, grid, lstride, adaptive, b.f32.P, b, s)
                : panel_launch<double>(g, ents, flag, count, m, grid, lstride, adaptive, b.P, b, s);
}

}  // namespace cams
