// The ILU(0) smoother's sweeps (Sec. 3, Table 1 step 6).  One smoothing step
// x <- x + M^{-1}(b - A x) is
//   rd = D^{-1} (b - A x)                         (parallel)
//   w_i = rd_i - sum_{j<i} (a_ij / d_i) w_j       (forward wavefront)
//   z_i = w_i  - sum_{j>i} (a_ij / d_i) z_j       (backward wavefront)
//   x += z
// with the couplings pre-scaled by the row pivot (k_ilu.cu), so every cell of
// a sweep is a chain of three FMAs.  In FP64 (b, x) = (f, p); in the
// mixed-precision preconditioner the smoother runs in FP32 on the correction
// equation, (b, x) = (r, delta).
//
// What bounds a sweep: not its bytes (20 or 40 a cell) but the chain of
// nx + ny + nz dependent cells and, along it, the hand-overs between tiles.
// The layout and the schedule are made for that chain.
//
// Layout.  A lane owns an x-row and works on chunks of G consecutive cells
// (G = 4 in FP32: one 16-byte access per operand, and what a step costs apart
// from its FMAs - the neighbour exchange, the operand loads, the barrier - is
// paid once for four cells; G = 1 in FP64, where a warp's three FMAs hold its
// FP64 unit for about 190 cycles a cell, so that longer chunks would lengthen
// the path of nx/G + ny + nz steps of G cells each).  The (y, z) cross-section
// is cut into tiles of 32 rows: 8 x 4, or 32 x 1 on a 2D grid.  Row (ty, tz)
// works on chunk X = s - ty - tz at step s, and the 32 chunks of a step are
// contiguous: a sweep's operands are stored [tile][step][operand][lane][G],
// operand 0 the input vector and 1-3 the scaled couplings, so a step's four
// operands are one record; the backward sweep's output z has records of its
// own.  Slots that hold no cell (the pipeline's fill and drain, the tail of a
// row's last chunk, rows beyond the grid) are zero in the input and in the
// couplings, so a step is branch-free; the values computed there never reach a
// cell with a nonzero coupling.
//
// Schedules of the same arithmetic (bitwise identical results):
//  * level-scheduled: one launch per hyperplane x+y+z = L (reference);
//  * pipelined: one tile per CTA, run by a team of four warps in lock step, the
//    CTAs of a thread-block cluster on a block of neighbouring tiles.
//    - Inside the tile a row's neighbours are one step behind; their chunks pass
//      through a two-deep shared-memory exchange buffer.
//    - Edge chunks from other tiles arrive in shared-memory rings (one per edge
//      row): pushed through distributed shared memory by the upstream tile's
//      CTA when it belongs to the same cluster, otherwise fetched by helper
//      warps that poll the upstream tile's published chunks in L2.  Measured
//      one way, CTA to CTA: 350 cycles through distributed shared memory, 550
//      (same die) or 890 (other die) through L2 in a tight ping-pong.
//    - A slot not written yet holds a signalling-NaN sentinel that no
//      arithmetic produces, in global memory as in the rings, so a value is its
//      own ready flag and no fences are needed (aligned 4- and 8-byte words are
//      written and read with single-copy atomicity; a chunk is ready when all
//      its words are).  The forward sweep re-marks the edge rows of z and the
//      backward sweep those of w behind them.
//    - Blocks are claimed through an atomic ticket in anti-diagonal order, so a
//      cluster only waits on blocks already claimed by running clusters: no
//      co-residency assumption, no deadlock.  Every wait has an iteration
//      limit; on expiry an abort flag and the status word are set and all warps
//      run on to their end.
//    Measured at 200 x 200 x 100 (us a sweep): FP32 150 -> 98, FP64 230 -> 145
//    against one warp a tile with per-cell steps and every hand-over through
//    L2; 64^3 FP64 86 -> 49, 40 x 40 x 1 FP64 35 -> 24.
//  The backward sweep runs the same schedule on the mirrored grid: its steps
//  read the same records in reverse order.
#include "cams_internal.h"
#include "launch.h"

namespace cams {

namespace {

constexpr int kStep = 4;                     // steps of the unrolled loop body (even)
constexpr int kSlots = 8;                    // operand slots: steps staged ahead (a power of two)
constexpr int kTeam = 4;                     // warps per tile
constexpr long long kPollLimit = 1LL << 22;  // helper polls without progress before a wait gives up
constexpr long long kSpinLimit = 1LL << 26;  // shared-memory polls before a wait gives up
constexpr int kSweepCtas = 8;                // CTAs of a cluster
constexpr int kSpare = kStep;                // spare records at both ends of a vector

// A chunk of G cells of one row, and the "not computed yet" sentinel: a
// signalling NaN.  IEEE arithmetic never produces one, so no computed value
// carries its pattern.
template <class T>
struct Chunk;
template <>
struct Chunk<float> {
  static constexpr int G = 4, kRing = 128;   // kRing: chunks per edge-row ring (a power of two)
  static constexpr unsigned kUnset = 0x7FA5A5A1u;
  struct alignas(16) V {
    float v[4];
  };
  static __device__ __forceinline__ V splat(float x) { return V{{x, x, x, x}}; }
  static __device__ __forceinline__ V get(const V* p) {
    const float4 f = *reinterpret_cast<const float4*>(p);
    return V{{f.x, f.y, f.z, f.w}};
  }
  static __device__ __forceinline__ void put(V* p, const V& a) {
    *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
  }
  static __device__ __forceinline__ float unset_value() { return __uint_as_float(kUnset); }
  static __device__ __forceinline__ bool unset(const V& a) {
    return __float_as_uint(a.v[0]) == kUnset || __float_as_uint(a.v[1]) == kUnset ||
           __float_as_uint(a.v[2]) == kUnset || __float_as_uint(a.v[3]) == kUnset;
  }
  static __device__ __forceinline__ V load_relaxed(const float* p) {
    V a;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(a.v[0]), "=f"(a.v[1]), "=f"(a.v[2]), "=f"(a.v[3])
                 : "l"(p));
    return a;
  }
  static __device__ __forceinline__ void store_cluster(unsigned p, const V& a) {
    asm volatile("st.relaxed.cluster.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p),
                 "f"(a.v[0]), "f"(a.v[1]), "f"(a.v[2]), "f"(a.v[3]));
  }
  static __device__ __forceinline__ void copy_async(unsigned dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
  static __device__ __forceinline__ void publish(float* p, const V& a) {
    asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a.v[0]),
                 "f"(a.v[1]), "f"(a.v[2]), "f"(a.v[3]));
  }
  static __device__ __forceinline__ V load_shared(unsigned p) {
    V a;
    asm volatile("ld.volatile.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(a.v[0]), "=f"(a.v[1]), "=f"(a.v[2]), "=f"(a.v[3])
                 : "r"(p));
    return a;
  }
  static __device__ __forceinline__ void store_shared(unsigned p, const V& a) {
    asm volatile("st.volatile.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(a.v[0]),
                 "f"(a.v[1]), "f"(a.v[2]), "f"(a.v[3]));
  }
};
template <>
struct Chunk<double> {
  static constexpr int G = 1, kRing = 256;
  static constexpr unsigned long long kUnset = 0x7FF4DEADBEEF0001ull;
  struct alignas(8) V {
    double v[1];
  };
  static __device__ __forceinline__ V splat(double x) { return V{{x}}; }
  static __device__ __forceinline__ V get(const V* p) { return *p; }
  static __device__ __forceinline__ void put(V* p, const V& a) { *p = a; }
  static __device__ __forceinline__ double unset_value() {
    return __longlong_as_double((long long)kUnset);
  }
  static __device__ __forceinline__ bool unset(const V& a) {
    return (unsigned long long)__double_as_longlong(a.v[0]) == kUnset;
  }
  // (values travel as 64-bit words: no floating-point move touches them)
  static __device__ __forceinline__ V load_relaxed(const double* p) {
    long long u;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(u) : "l"(p));
    return V{{__longlong_as_double(u)}};
  }
  static __device__ __forceinline__ void store_cluster(unsigned p, const V& a) {
    asm volatile("st.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(p),
                 "l"(__double_as_longlong(a.v[0])));
  }
  static __device__ __forceinline__ void copy_async(unsigned dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
  }
  static __device__ __forceinline__ void publish(double* p, const V& a) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(__double_as_longlong(a.v[0])));
  }
  static __device__ __forceinline__ V load_shared(unsigned p) {
    long long u;
    asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(u) : "r"(p));
    return V{{__longlong_as_double(u)}};
  }
  static __device__ __forceinline__ void store_shared(unsigned p, const V& a) {
    asm volatile("st.volatile.shared.b64 [%0], %1;" ::"r"(p), "l"(__double_as_longlong(a.v[0])));
  }
};

__device__ __forceinline__ int ld_relaxed_int(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Rows of a tile, one a lane: 8 x 4, or 32 x 1 on a 2D grid (nz = 1), where
// 8 x 4 would leave three quarters of every warp idle.
template <class T, bool kFlat>
struct Tile {
  static constexpr int TY = kFlat ? 32 : 8, TZ = kFlat ? 1 : 4;
  static constexpr int EY = TZ, EZ = kFlat ? 0 : TY, E = EY + EZ;    // edge rows: y, z
  static constexpr int G = Chunk<T>::G;
  static constexpr int kVec = 32 * G, kRec = 4 * kVec;               // elements of a record
  static_assert(TY * TZ == 32 && E <= 32, "a tile is one warp; a lane carries one edge row");
};

struct Shape {
  int nty, ntz;   // tiles in y and z
  int nxc, ns;    // chunks per row, records per tile (a multiple of kStep)
};

template <class T, bool kFlat>
Shape shape_of(const Geo& g) {
  using L = Tile<T, kFlat>;
  const int nxc = (g.nx + L::G - 1) / L::G;
  const int ns = (nxc + L::TY + L::TZ - 2 + kStep - 1) / kStep * kStep;
  return Shape{(g.ny + L::TY - 1) / L::TY, (g.nz + L::TZ - 1) / L::TZ, nxc, ns};
}

// Record and element within a record's operand of cell (x, y, z).
template <class T, bool kFlat>
__device__ __forceinline__ void sweep_index(const Shape& s, int x, int y, int z, long long& rec,
                                            int& el) {
  using L = Tile<T, kFlat>;
  const int Y = y / L::TY, ty = y - Y * L::TY, Z = z / L::TZ, tz = z - Z * L::TZ;
  const int X = x / L::G, u = x - X * L::G;
  rec = kSpare + (long long)(Y + s.nty * Z) * s.ns + X + ty + tz;
  el = (ty + L::TY * tz) * L::G + u;
}

// ------------------------------------------------------ parallel parts ---

// The conversions between the natural and the sweep layout run as tile
// transposes: one CTA per (tile, kXC positions along x).  Rows are read or
// written in the natural layout by warps along x (coalesced); records are
// written or read by warps whose lanes are the tile's lanes, one chunk each;
// shared memory holds the block in between.  FP64 takes 32 positions a CTA: the
// FP64 unit bounds the residual there, and with 64 a grid of 500k cells gave
// some SMs three CTAs of work and others two (19.5 against 18.4 us).
template <class T>
constexpr int kXC = sizeof(T) == 8 ? 32 : 64;
// row stride of that block: in a record, lane ty + 1 sits one row down and one
// chunk to the left; this stride keeps the chunks of a record on different banks
template <class T>
constexpr int kRow = kXC<T> + 2 * Chunk<T>::G;

// Row-pivot-scaled couplings in the sweep layout: L_d = a_{i,i-e_d} / d_i into
// operands 1-3 of lo, U_d = a_{i,i+e_d} / d_i into those of up.
template <class T, bool kFlat>
__global__ void k_ilu_scale(Geo g, Shape s, const T* __restrict__ Ax, const T* __restrict__ Ay,
                            const T* __restrict__ Az, const T* __restrict__ Axu,
                            const T* __restrict__ Ayu, const T* __restrict__ Azu,
                            const T* __restrict__ dinv, T* lo, T* up) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  int x, y, z;
  xyz_of(g, i, x, y, z);
  long long rec;
  int el;
  sweep_index<T, kFlat>(s, x, y, z, rec, el);
  constexpr int kOp = Tile<T, kFlat>::kVec;
  const long long j = rec * Tile<T, kFlat>::kRec + el;
  const T di = dinv[i];
  lo[j + kOp] = Ax[i] * di;
  lo[j + 2 * kOp] = Ay[i] * di;
  lo[j + 3 * kOp] = Az[i] * di;
  up[j + kOp] = x < g.nx - 1 ? Axu[i + 1] * di : T(0);
  up[j + 2 * kOp] = y < g.ny - 1 ? Ayu[i + g.sy] * di : T(0);
  up[j + 3 * kOp] = z < g.nz - 1 ? Azu[i + g.sz] * di : T(0);
}

// rd = D^{-1} (b - A x) into operand 0 of lo.  kNS: Axu.. hold the couplings
// to the upper neighbours (A not symmetric); otherwise Ax.. serve both.
// The first CTA resets the tickets of the two sweeps that follow.
template <class T, bool kNS, bool kFlat>
__global__ void __launch_bounds__(256) k_resid_scaled(Geo g, Shape s, const T* __restrict__ Ad,
                                                      const T* __restrict__ Ax,
                                                      const T* __restrict__ Ay,
                                                      const T* __restrict__ Az,
                                                      const T* __restrict__ Axu,
                                                      const T* __restrict__ Ayu,
                                                      const T* __restrict__ Azu,
                                                      const T* __restrict__ bv,
                                                      const T* __restrict__ xv,
                                                      const T* __restrict__ dinv, T* lo,
                                                      int* ctrl) {
  using L = Tile<T, kFlat>;
  using Ch = Chunk<T>;
  using V = typename Ch::V;
  constexpr int G = L::G, kRows = 32, kC = kXC<T>;
  __shared__ alignas(16) T blk[kRows][kRow<T>];
  const int piece = (int)blockIdx.x / (s.nty * s.ntz), tile = (int)blockIdx.x - piece * (s.nty * s.ntz);
  const int x0 = piece * kC;
  pdl_enter();
  if (blockIdx.x == 0 && threadIdx.x < 3) ctrl[threadIdx.x] = 0;
  const int Y = tile % s.nty, Z = tile / s.nty;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // (unrolled, with predicates instead of early exits, so that a thread's
  // loads of several cells are in flight together; 256 threads)
#pragma unroll 4
  for (int rr = 0; rr < kRows / 8; ++rr) {
    const int r = warp + rr * 8;
    const int y = Y * L::TY + r % L::TY, z = Z * L::TZ + r / L::TY;
#pragma unroll
    for (int hh = 0; hh < kC / 32; ++hh) {
      const int h = lane + 32 * hh;
      const int x = x0 + h;
      T v = T(0);                            // the tail of the row's last chunk
      if (y < g.ny && z < g.nz && x < g.nx) {
        const long long i = x + g.sy * y + g.sz * z;
        T a;
        if constexpr (sizeof(T) == 4) {
          // every load before the first use, with a zero in place of a
          // neighbour outside the grid (0 * 0 changes no sum): behind branches
          // each neighbour's loads wait for the ones before.  (4M cells: 40.6
          // against 38.4 us; FP64, which waits for its unit, gains nothing.)
          const bool xl = x > 0, xu = x < g.nx - 1, yl = y > 0, yu = y < g.ny - 1, zl = z > 0, zu = z < g.nz - 1;
          const T cb = bv[i], cd = Ad[i], xc = xv[i];
          const T c0 = xl ? Ax[i] : T(0), v0 = xl ? xv[i - 1] : T(0);
          const T c1 = xu ? (kNS ? Axu : Ax)[i + 1] : T(0), v1 = xu ? xv[i + 1] : T(0);
          const T c2 = yl ? Ay[i] : T(0), v2 = yl ? xv[i - g.sy] : T(0);
          const T c3 = yu ? (kNS ? Ayu : Ay)[i + g.sy] : T(0), v3 = yu ? xv[i + g.sy] : T(0);
          const T c4 = zl ? Az[i] : T(0), v4 = zl ? xv[i - g.sz] : T(0);
          const T c5 = zu ? (kNS ? Azu : Az)[i + g.sz] : T(0), v5 = zu ? xv[i + g.sz] : T(0);
          a = cb - cd * xc;
          a -= c0 * v0;
          a -= c1 * v1;
          a -= c2 * v2;
          a -= c3 * v3;
          a -= c4 * v4;
          a -= c5 * v5;
        } else {
          a = bv[i] - Ad[i] * xv[i];
          if (x > 0) a -= Ax[i] * xv[i - 1];
          if (x < g.nx - 1) a -= (kNS ? Axu : Ax)[i + 1] * xv[i + 1];
          if (y > 0) a -= Ay[i] * xv[i - g.sy];
          if (y < g.ny - 1) a -= (kNS ? Ayu : Ay)[i + g.sy] * xv[i + g.sy];
          if (z > 0) a -= Az[i] * xv[i - g.sz];
          if (z < g.nz - 1) a -= (kNS ? Azu : Az)[i + g.sz] * xv[i + g.sz];
        }
        v = a * dinv[i];
      }
      blk[r][h] = v;
    }
  }
  __syncthreads();
  // record q holds lane (ty, tz)'s rows at chunk X = q - ty - tz
  const int ty = lane % L::TY, tz = lane / L::TY, X0 = x0 / G;
  constexpr int kQ = kC / G + L::TY + L::TZ - 2;
  for (int q = X0 + warp; q < X0 + kQ; q += 8) {
    const int X = q - ty - tz;
    if (Y * L::TY + ty < g.ny && Z * L::TZ + tz < g.nz && X >= X0 && X < X0 + kC / G && X < s.nxc)
      Ch::put(reinterpret_cast<V*>(lo + (kSpare + (long long)tile * s.ns + q) * L::kRec + lane * G),
              Ch::get(reinterpret_cast<const V*>(&blk[lane][(X - X0) * G])));
  }
}

// x += z (the correction of one smoothing step), z in the sweep layout.
template <class T, bool kFlat>
__global__ void __launch_bounds__(256) k_apply_z(Geo g, Shape s, const T* __restrict__ zs, T* xv) {
  using L = Tile<T, kFlat>;
  using Ch = Chunk<T>;
  using V = typename Ch::V;
  constexpr int G = L::G, kRows = 32, kC = kXC<T>;
  __shared__ alignas(16) T blk[kRows][kRow<T>];
  const int piece = (int)blockIdx.x / (s.nty * s.ntz), tile = (int)blockIdx.x - piece * (s.nty * s.ntz);
  const int x0 = piece * kC;
  pdl_enter();
  const int Y = tile % s.nty, Z = tile / s.nty;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ty = lane % L::TY, tz = lane / L::TY, X0 = x0 / G;
  constexpr int kQ = kC / G + L::TY + L::TZ - 2;
#pragma unroll 4
  for (int q = X0 + warp; q < X0 + kQ; q += 8) {
    const int X = q - ty - tz;
    if (Y * L::TY + ty < g.ny && Z * L::TZ + tz < g.nz && X >= X0 && X < X0 + kC / G && X < s.nxc)
      Ch::put(reinterpret_cast<V*>(&blk[lane][(X - X0) * G]),
              Ch::get(reinterpret_cast<const V*>(
                  zs + (kSpare + (long long)tile * s.ns + q) * L::kVec + lane * G)));
  }
  __syncthreads();
  // several x values of a thread are loaded before any is written back (the
  // stores through xv would otherwise order every later load after them);
  // 256 threads
  constexpr int kB = 4;
#pragma unroll 1
  for (int r0 = 0; r0 < kRows / 8; r0 += kB) {
    T xo[kB][kC / 32];
#pragma unroll
    for (int rr = 0; rr < kB; ++rr) {
      const int r = warp + (r0 + rr) * 8;
      const int y = Y * L::TY + r % L::TY, z = Z * L::TZ + r / L::TY;
#pragma unroll
      for (int hh = 0; hh < kC / 32; ++hh) {
        const int x = x0 + lane + 32 * hh;
        xo[rr][hh] = (y < g.ny && z < g.nz && x < g.nx) ? xv[x + g.sy * y + g.sz * z] : T(0);
      }
    }
#pragma unroll
    for (int rr = 0; rr < kB; ++rr) {
      const int r = warp + (r0 + rr) * 8;
      const int y = Y * L::TY + r % L::TY, z = Z * L::TZ + r / L::TY;
#pragma unroll
      for (int hh = 0; hh < kC / 32; ++hh) {
        const int h = lane + 32 * hh, x = x0 + h;
        if (y < g.ny && z < g.nz && x < g.nx) xv[x + g.sy * y + g.sz * z] = xo[rr][hh] + blk[r][h];
      }
    }
  }
}

// operand 0 of every record of `a` (kRec elements each): n = records x kVec
template <class T>
__global__ void k_fill_unset(long long n, int kVec, int kRec, T* a) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) a[i / kVec * kRec + i % kVec] = Chunk<T>::unset_value();
}

// ---------------------------------------------------- level schedule ---

// value = in - Cx v_x - Cy v_y - Cz v_z over the upstream neighbours
template <class T>
__device__ __forceinline__ T cell_value(T in, T cx, T cy, T cz, T vx, T vy, T vz) {
  return fma(-cx, vx, fma(-cy, vy, fma(-cz, vz, in)));
}

template <class T, bool kBackward, bool kFlat>
__global__ void k_sweep_level(Geo g, Shape sh, int Lv, const T* ops, T* out, int out_rec) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)g.ny * g.nz) return;
  const int y = (int)(t % g.ny), z = (int)(t / g.ny);
  const int xf = Lv - y - z;                 // position along the sweep
  if (xf < 0 || xf >= g.nx) return;
  // the backward sweep visits hyperplane Lv of the mirrored grid
  const int x = kBackward ? g.nx - 1 - xf : xf;
  const int yy = kBackward ? g.ny - 1 - y : y;
  const int zz = kBackward ? g.nz - 1 - z : z;
  using L = Tile<T, kFlat>;
  constexpr int kOp = L::kVec, e = kBackward ? 1 : -1;
  auto at = [&](int dx, int dy, int dz) {
    long long rec;
    int el;
    sweep_index<T, kFlat>(sh, x + dx, yy + dy, zz + dz, rec, el);
    return out[rec * out_rec + el];
  };
  const bool hx = kBackward ? x < g.nx - 1 : x > 0;
  const bool hy = kBackward ? yy < g.ny - 1 : yy > 0;
  const bool hz = kBackward ? zz < g.nz - 1 : zz > 0;
  long long rec;
  int el;
  sweep_index<T, kFlat>(sh, x, yy, zz, rec, el);
  const T* c = ops + rec * L::kRec + el;
  out[rec * out_rec + el] =
      cell_value(c[0], c[kOp], c[2 * kOp], c[3 * kOp], hx ? at(e, 0, 0) : T(0),
                 hy ? at(0, e, 0) : T(0), hz ? at(0, 0, e) : T(0));
}

// ------------------------------------------------ pipelined schedule ---

// Block (Y, Z) of ticket t: anti-diagonals Y + Z in increasing order, Y
// ascending within one.
__device__ __forceinline__ void block_of_ticket(int t, int ny, int nz, int& Y, int& Z) {
  for (int d = 0;; ++d) {
    const int ylo = d - (nz - 1) > 0 ? d - (nz - 1) : 0;
    const int yhi = d < ny - 1 ? d : ny - 1;
    const int cnt = yhi - ylo + 1;
    if (t < cnt) {
      Y = ylo + t;
      Z = d - Y;
      return;
    }
    t -= cnt;
  }
}

// Shared memory of a CTA: operand slots [kSlots][4][32], exchange buffers
// [2]{[32], [E], zero}, edge rings [E][kRing], then control words.
template <class T, bool kFlat>
struct Plan {
  using L = Tile<T, kFlat>;
  static constexpr int XS = 32 + L::E + 1, kV = (int)sizeof(typename Chunk<T>::V);
  static constexpr int kRing = Chunk<T>::kRing;
  // A main warp's progress matters only to rows that wrap around the rings, and
  // a report needs a fence, which costs half a microsecond: a report every
  // quarter of a ring, and none for shorter rows.
  static constexpr int kReport = kRing / 4, kNoWrap = kRing - 32;
  static constexpr int kLanes = 8;                            // helper lanes per edge row
  static constexpr int kRows = 32 / kLanes;                   // edge rows per helper warp
  static constexpr int H = (L::E + kRows - 1) / kRows;
  static constexpr int kThreads = 32 * (kTeam + H);           // the team, the helpers
  static constexpr int kOpsB = kSlots * 128 * kV, kXchB = 2 * XS * kV, kRingsB = L::E * kRing * kV;
  static constexpr int kRings = kOpsB + kXchB, kCtrl = (kRings + kRingsB + 15) / 16 * 16;
  // control words: progress of the y and the z downstream tile and of this
  // one (every edge chunk of steps <= it has been taken), two ticket slots
  static constexpr int kBytes = kCtrl + 5 * 4;
  // record stride of the vector a sweep publishes: the forward sweep's w is
  // operand 0 of the backward sweep's records, z is a vector of its own
  static constexpr int rec_out(bool backward) { return backward ? L::kVec : L::kRec; }
};

// ---- thread-block cluster ----
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the address of a shared-memory word of this CTA in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_rank(unsigned p, unsigned rank) {
  unsigned q;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(q) : "r"(p), "r"(rank));
  return q;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ void store_cluster(unsigned p, int v) {
  asm volatile("st.relaxed.cluster.shared::cluster.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int load_ctrl(unsigned p) {
  int v;
  asm volatile("ld.volatile.shared.b32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
  return v;
}

__device__ __forceinline__ void give_up(int* abort_flag, int* status) {
  atomicOr(status, kStatTimeout);
  atomicExch(abort_flag, 1);
}

// A chunk that has not arrived in its ring yet: polls until it has.  After an
// abort or a timeout (flagged) it returns zeros: the tile then runs on to its
// end with wrong values, and the caller of the sweep reports the status.
template <class T>
__device__ __noinline__ typename Chunk<T>::V wait_edge(unsigned p, int* abort_flag, int* status) {
  using Ch = Chunk<T>;
  for (long long it = 0; it < kSpinLimit; ++it) {
    const typename Ch::V e = Ch::load_shared(p);
    if (!Ch::unset(e)) return e;
    if ((it & 255) == 255) {
      if (ld_relaxed_int(abort_flag)) return Ch::splat(T(0));
      if (it > 65536) __nanosleep(40);
    }
  }
  give_up(abort_flag, status);
  return Ch::splat(T(0));
}

// Waits until the consumer's progress reaches `need` (ring room) and returns
// it; after an abort or a timeout it returns a progress that never waits.
__device__ __noinline__ int wait_room(unsigned prog, int need, int* abort_flag, int* status) {
  for (long long it = 0; it < kSpinLimit; ++it) {
    const int p = load_ctrl(prog);
    if (p >= need) return p;
    if ((it & 255) == 255) {
      if (ld_relaxed_int(abort_flag)) return 1 << 30;
      if (it > 65536) __nanosleep(40);
    }
  }
  give_up(abort_flag, status);
  return 1 << 30;
}

// A tile is run by a team of four warps in lock step, a named barrier a step.
// A warp alone issues an instruction every four cycles or so (each waits for
// the one before), so a step is kept short by giving every warp little to do:
//  * the main warp has the dependent chain: neighbours' chunks from the
//    exchange buffer, the FMAs, its chunk into the exchange buffer and out;
//  * the stager copies the operands (cp.async) kSlots steps ahead;
//  * the edge warp takes the next step's edge chunks from their rings to the
//    exchange buffer;
//  * the feeder passes the last step's chunks to the rings of the downstream
//    tiles of this CTA and marks the rows that the next sweep polls.
// Barrier s (from -1) ends step s.  Before it, the edge chunks of step s + 1
// are in the exchange buffer and the operands of steps <= s + 2 in their slots.
__device__ __forceinline__ void team_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kTeam) : "memory");
}

// What the warps of a CTA know of its tile: (Ym, Zm) is its place in the sweep
// frame (mirrored for the backward sweep).  A block of tiles belongs to the
// CTAs of a cluster, nby x nbz of them, tile (Ym, Zm) at place (by, bz).
struct Place {
  int Ym, Zm, by, bz, nby, nbz;
};

template <class T, bool kBackward, bool kFlat>
struct Team {
  using Ch = Chunk<T>;
  using V = typename Ch::V;
  using L = Tile<T, kFlat>;
  using Pl = Plan<T, kFlat>;
  static constexpr int G = L::G, kDir = kBackward ? -1 : 1;
  static constexpr int kRing = Pl::kRing;
  static constexpr unsigned kV = Pl::kV, kXB = Pl::XS * kV, kRingB = kRing * kV;
  static constexpr int kIn = kDir * L::kRec;                           // per step
  static constexpr int kOut = kDir * Pl::rec_out(kBackward), kMark = kDir * Pl::rec_out(!kBackward);
  int tym, tzm, lane_m, pad, lag;
  long long rec0;
  unsigned base, ops, xch, rings, ctrl;
  __device__ __forceinline__ Team(const Shape& sh, unsigned char* smem, int lane, const Place& p) {
    base = (unsigned)__cvta_generic_to_shared(smem);
    tym = lane % L::TY;
    tzm = lane / L::TY;
    lane_m = kBackward ? 31 - lane : lane;                             // in a record
    const int Y = kBackward ? sh.nty - 1 - p.Ym : p.Ym, Z = kBackward ? sh.ntz - 1 - p.Zm : p.Zm;
    rec0 = kSpare + (long long)(Y + sh.nty * Z) * sh.ns + (kBackward ? sh.ns - 1 : 0);
    // my chunk of step s is s - lag (the backward sweep starts in the padding)
    pad = kBackward ? sh.ns - (sh.nxc + L::TY + L::TZ - 2) : 0;
    lag = tym + tzm + pad;
    ops = base + (unsigned)lane * kV;
    xch = base + Pl::kOpsB;
    rings = base + Pl::kRings;
    ctrl = base + Pl::kCtrl;
  }
};

// The main warp.  It runs kStep dry steps first (no barriers, global
// stores into the spare records): a CTA reaches its tile with a cold
// instruction cache, and fetching the loop's code only when the upstream
// chunks have arrived would add its misses to every hand-over.
template <class T, bool kBackward, bool kFlat>
__device__ __forceinline__ void main_warp(const Shape& sh, T* out, unsigned char* smem, int lane,
                                          const Place& pc) {
  using P = Team<T, kBackward, kFlat>;
  using Ch = typename P::Ch;
  using V = typename P::V;
  using L = typename P::L;
  using Pl = typename P::Pl;
  constexpr int G = P::G;
  constexpr unsigned kV = P::kV, kXB = P::kXB;
  const P t(sh, smem, lane, pc);
  const unsigned xo = t.xch + (unsigned)lane * kV;   // my place in the exchange buffer
  const unsigned xy = t.tym > 0 ? xo - kV : t.xch + (unsigned)(32 + t.tzm) * kV;
  const unsigned xz = kFlat        ? t.xch + (unsigned)(32 + L::E) * kV
                      : t.tzm > 0 ? xo - L::TY * kV
                                  : t.xch + (unsigned)(32 + L::EY + t.tym) * kV;
  const long long spare = kSpare + (long long)sh.nty * sh.ntz * sh.ns + (kBackward ? kSpare - 1 : 0);
  T* po = out + spare * Pl::rec_out(kBackward) + t.lane_m * G;         // of step s0
  const V zero = Ch::splat(T(0));
  V o[4];
  T vprev = T(0);
  auto operands = [&](int s, V* v) {
    const unsigned d = t.ops + (unsigned)(s & (kSlots - 1)) * (128 * kV);
#pragma unroll
    for (int a = 0; a < 4; ++a) v[a] = Ch::load_shared(d + a * 32 * kV);
  };
#pragma unroll
  for (int a = 0; a < 4; ++a) o[a] = zero;
#pragma unroll 1
  for (int s0 = -kStep; s0 < sh.ns; s0 += kStep) {
    const bool live = s0 >= 0;
    if (s0 == 0) {
      po = out + t.rec0 * Pl::rec_out(kBackward) + t.lane_m * G;
      Ch::store_shared(xo, zero);
      Ch::store_shared(xo + kXB, zero);
      vprev = T(0);
    }
#pragma unroll
    for (int k = 0; k < kStep; ++k) {
      const int s = s0 + k;
      const unsigned xr = (k & 1) ? 0u : kXB, xw = (k & 1) ? kXB : 0u;   // kStep is even
      if (live) team_sync();
      const V vy = Ch::load_shared(xy + xr);
      const V vz = Ch::load_shared(xz + xr);
      if (s0 == 0 && k == 0) operands(0, o);
      V on[4];
      operands(s + 1, on);                         // (past the tile: not used)
      if (s == t.lag) vprev = T(0);                // my row starts here
      V v;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const int u = kBackward ? G - 1 - q : q;
        vprev = cell_value(o[0].v[u], o[1].v[u], o[2].v[u], o[3].v[u], vprev, vy.v[u], vz.v[u]);
        v.v[u] = vprev;
      }
      Ch::store_shared(xo + xw, v);
      Ch::publish(po + k * P::kOut, v);
#pragma unroll
      for (int a = 0; a < 4; ++a) o[a] = on[a];
    }
    po += kStep * P::kOut;
  }
  team_sync();
}

template <class T, bool kBackward, bool kFlat>
__device__ __forceinline__ void stager_warp(const Shape& sh, const T* ops, unsigned char* smem,
                                            int lane, const Place& pc) {
  using P = Team<T, kBackward, kFlat>;
  using Ch = typename P::Ch;
  using L = typename P::L;
  constexpr unsigned kV = P::kV;
  const P t(sh, smem, lane, pc);
  const T* pi = ops + t.rec0 * L::kRec + t.lane_m * P::G;              // of the step being staged
  auto stage = [&](int s) {
    if (s < sh.ns) {
      const unsigned d = t.ops + (unsigned)(s & (kSlots - 1)) * (128 * kV);
#pragma unroll
      for (int a = 0; a < 4; ++a) Ch::copy_async(d + a * 32 * kV, pi + a * L::kVec);
      pi += P::kIn;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 1
  for (int s = 0; s < kSlots; ++s) stage(s);
#pragma unroll 1
  for (int s = -1; s < sh.ns; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSlots - 3) : "memory");
    team_sync();
    if (s >= 0) stage(s + kSlots);                 // into the slot of step s
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Lane e < E carries edge row e.
template <class T, bool kBackward, bool kFlat>
__device__ __forceinline__ void edge_warp(const Shape& sh, int* abort_flag, int* status,
                                          unsigned char* smem, int lane, const Place& pc) {
  using P = Team<T, kBackward, kFlat>;
  using Ch = typename P::Ch;
  using V = typename P::V;
  using L = typename P::L;
  using Pl = typename P::Pl;
  constexpr int kRing = P::kRing;
  constexpr unsigned kV = P::kV, kXB = P::kXB;
  const P t(sh, smem, lane, pc);
  const bool has_edge = lane < L::E && (lane < L::EY ? pc.Ym > 0 : pc.Zm > 0);
  const int elag = (lane < L::EY ? lane : lane - L::EY) + t.pad;
  const int first = elag, last = has_edge ? elag + sh.nxc : 0;         // steps that need my chunk
  const unsigned ring = t.rings + (unsigned)(lane < L::E ? lane : 0) * P::kRingB;
  const unsigned xe = t.xch + (unsigned)(32 + lane) * kV;
  const V unset = Ch::splat(Ch::unset_value());
  // who is told of the progress: lane 0 this CTA's helpers, lanes 1 and 2 the
  // y and z upstream tiles of the cluster
  unsigned tell = t.ctrl + 8;
  if (lane == 1 && pc.by > 0) tell = map_rank(t.ctrl, (unsigned)(pc.by - 1 + pc.nby * pc.bz));
  if (lane == 2 && pc.bz > 0) tell = map_rank(t.ctrl + 4, (unsigned)(pc.by + pc.nby * (pc.bz - 1)));
  if (lane == 0) tell = map_rank(tell, (unsigned)(pc.by + pc.nby * pc.bz));
  const bool teller = sh.nxc > Pl::kNoWrap && (lane == 0 || (lane == 1 && pc.by > 0) || (lane == 2 && pc.bz > 0));
  for (int k = lane; k < L::E + 1; k += 32) {
    Ch::store_shared(t.xch + (unsigned)(32 + k) * kV, Ch::splat(T(0)));
    Ch::store_shared(t.xch + (unsigned)(32 + k) * kV + kXB, Ch::splat(T(0)));
  }
  __syncwarp();
  // (a chunk is loaded from its ring before the barrier and looked at after it)
  V e = unset;
  if (0 >= first && 0 < last) e = Ch::load_shared(ring);
#pragma unroll 2
  for (int s = -1; s < sh.ns; ++s) {
    if (s + 1 >= first && s + 1 < last) {
      const unsigned re = ring + (unsigned)((s + 1) & (kRing - 1)) * kV;
      if (Ch::unset(e)) e = wait_edge<T>(re, abort_flag, status);
      Ch::store_shared(xe + ((s & 1) ? kXB : 0u), e);
      Ch::store_shared(re, unset);
    }
    if (has_edge) e = Ch::load_shared(ring + (unsigned)((s + 2) & (kRing - 1)) * kV);
    team_sync();
    if (teller && s >= 0 && (s & (Pl::kReport - 1)) == Pl::kReport - 1) {
      asm volatile("fence.acq_rel.cluster;" ::: "memory");   // the ring slots that were reset come first
      store_cluster(tell, s - t.pad);
    }
  }
}

template <class T, bool kBackward, bool kFlat>
__device__ __forceinline__ void feeder_warp(const Shape& sh, T* mark, int* abort_flag, int* status,
                                            unsigned char* smem, int lane, const Place& pc) {
  using P = Team<T, kBackward, kFlat>;
  using Ch = typename P::Ch;
  using V = typename P::V;
  using L = typename P::L;
  using Pl = typename P::Pl;
  constexpr int kRing = P::kRing;
  constexpr unsigned kV = P::kV, kXB = P::kXB, kRingB = P::kRingB;
  const P t(sh, smem, lane, pc);
  const bool fy = pc.by + 1 < pc.nby && pc.Ym + 1 < sh.nty;            // fed through the cluster
  const bool fz = !kFlat && pc.bz + 1 < pc.nbz && pc.Zm + 1 < sh.ntz;
  const bool put_y = fy && t.tym == L::TY - 1, put_z = fz && t.tzm == L::TZ - 1;
  unsigned oy = t.rings + (unsigned)t.tzm * kRingB, oz = t.rings + (unsigned)(L::EY + t.tym) * kRingB;
  if (fy) oy = map_rank(oy, (unsigned)(pc.by + 1 + pc.nby * pc.bz));
  if (fz) oz = map_rank(oz, (unsigned)(pc.by + pc.nby * (pc.bz + 1)));
  const unsigned xo = t.xch + (unsigned)lane * kV;
  const bool mark_lane = t.tym == 0 || (!kFlat && t.tzm == 0);
  const V unset = Ch::splat(Ch::unset_value());
  T* pm = mark + t.rec0 * Pl::rec_out(!kBackward) + t.lane_m * P::G;
  int seen_y = -1, seen_z = -1;
  team_sync();
#pragma unroll 2
  for (int s = 0; s < sh.ns; ++s) {
    // room downstream: the ring slot of chunk X is free once its consumer has
    // taken chunk X - kRing (progress p: every edge chunk of steps <= p)
    if (fy && s - t.pad > seen_y + kRing + L::TY - 1)
      seen_y = wait_room(t.ctrl, s - t.pad - kRing - (L::TY - 1), abort_flag, status);
    if (fz && s - t.pad > seen_z + kRing + L::TZ - 1)
      seen_z = wait_room(t.ctrl + 4, s - t.pad - kRing - (L::TZ - 1), abort_flag, status);
    const bool row = (unsigned)(s - t.lag) < (unsigned)sh.nxc;
    team_sync();
    if (row && (put_y || put_z)) {
      // (ring slots go by the consumer's step)
      const V v = Ch::load_shared(xo + ((s & 1) ? kXB : 0u));
      if (put_y) Ch::store_cluster(oy + (unsigned)((s - (L::TY - 1)) & (kRing - 1)) * kV, v);
      if (put_z) Ch::store_cluster(oz + (unsigned)((s - (L::TZ - 1)) & (kRing - 1)) * kV, v);
    }
    if (mark_lane) Ch::publish(pm, unset);
    pm += P::kMark;
  }
}

// Helper warp hw of a CTA: fetches edge rows from upstream tiles outside the
// cluster, kLanes lanes a row; lane j polls chunks j, j + kLanes, ... in turn
// (a ring slot is its own ready flag, so the lanes of a row need no order
// among them).  Until the first chunk of any of its rows arrives, only the
// rows' first lanes poll.  One loop for both, and no lane leaves it or takes a
// path of its own before the others are done: lanes that spin must not keep
// the others from running.
template <class T, bool kBackward, bool kFlat>
__device__ __forceinline__ void helper_warp(const Shape& sh, const T* out, int* abort_flag,
                                            int* status, unsigned char* smem, int hw, int lane,
                                            const Place& pc) {
  using P = Team<T, kBackward, kFlat>;
  using Ch = typename P::Ch;
  using V = typename P::V;
  using L = typename P::L;
  using Pl = typename P::Pl;
  constexpr int kRing = P::kRing;
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int kN = Pl::kLanes;
  const P t(sh, smem, lane, pc);
  const int j = lane % kN, e = hw * Pl::kRows + lane / kN;             // my edge row
  const bool y_row = e < L::EY;
  const int lag = y_row ? e : e - L::EY;
  const bool active = e < L::E && (y_row ? pc.by == 0 && pc.Ym > 0 : pc.bz == 0 && pc.Zm > 0);
  // the upstream tile, its lane and step of chunk 0
  const int lane_u = y_row ? L::TY - 1 + L::TY * lag : lag + L::TY * (L::TZ - 1);
  const int s_u = t.pad + lag + (y_row ? L::TY : L::TZ) - 1;
  const int Yu = pc.Ym - (y_row ? 1 : 0), Zu = pc.Zm - (y_row ? 0 : 1);
  const int Y = kBackward ? sh.nty - 1 - Yu : Yu, Z = kBackward ? sh.ntz - 1 - Zu : Zu;
  const long long rec =
      kSpare + (long long)(Y + sh.nty * Z) * sh.ns + (kBackward ? sh.ns - 1 - s_u : s_u);
  constexpr int dv = P::kOut;
  const int el = (kBackward ? 31 - lane_u : lane_u) * L::G;
  const T* src = out + (active ? rec * Pl::rec_out(kBackward) + el + (long long)j * dv : 0);
  const unsigned rg = t.rings + (active ? (unsigned)(e * kRing) * P::kV : 0u);
  const int end = active ? sh.nxc : 0;
  int X = j;                                       // my next chunk
  bool begun = false;
  long long idle = 0;
  while (__any_sync(kAll, X < end)) {
    // the ring slot of chunk X is free once the consumer has taken chunk X - kRing
    const bool want = X < end && (begun || j == 0) && X < load_ctrl(t.ctrl + 8) + kRing + 1 - lag;
    V v = Ch::splat(T(0));
    if (want) v = Ch::load_relaxed(src);
    const bool got = want && !Ch::unset(v);
    if (got) {
      Ch::store_shared(rg + (unsigned)((X + lag + t.pad) & (kRing - 1)) * P::kV, v);
      X += kN;
      src += kN * dv;
    }
    begun = begun || __any_sync(kAll, got);
    idle = got ? 0 : idle + 1;
    if ((idle & 255) == 255 && X < end) {
      if (idle >= kPollLimit) give_up(abort_flag, status);
      if (ld_relaxed_int(abort_flag)) X = end;
    }
  }
}

// ctrl: [0] forward ticket, [1] backward ticket, [2] abort flag.  ops: the
// sweep's operand records; `out` is the vector it publishes into (its edge
// rows hold the sentinel), `mark` the one whose edge rows it marks unset for
// the next sweep.  nby x nbz: the CTAs of a cluster, one tile each.
template <class T, bool kBackward, bool kFlat>
__global__ void __launch_bounds__(Plan<T, kFlat>::kThreads)
    k_sweep(Shape sh, const T* ops, T* out, T* mark, int* ctrl, int* status, int nby, int nbz) {
  using Ch = Chunk<T>;
  using L = Tile<T, kFlat>;
  using Pl = Plan<T, kFlat>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const unsigned base = (unsigned)__cvta_generic_to_shared(smem_raw), words = base + Pl::kCtrl;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned rank = cluster_rank();
  cluster_arrive();
  pdl_enter();
  // (a ring slot is reset when its chunk is taken, so the rings are unset
  // again after every tile)
  for (int k = threadIdx.x; k < Pl::kRingsB / Pl::kV; k += blockDim.x)
    Ch::store_shared(base + Pl::kRings + (unsigned)k * Pl::kV, Ch::splat(Ch::unset_value()));
  // no CTA's shared memory is written from another one before all have started
  cluster_wait();
  const int ncy = (sh.nty + nby - 1) / nby, ncz = (sh.ntz + nbz - 1) / nbz, nblocks = ncy * ncz;
  Place pc{0, 0, (int)rank % nby, (int)rank / nby, nby, nbz};
  for (unsigned turn = 0;; turn ^= 1u) {
    // the cluster's block: its first CTA claims it and tells the others.  (The
    // barrier at the end of a block keeps the control words of the next one
    // apart; the tickets alternate between two words.)
    if (threadIdx.x < 3) store_cluster(map_rank(words + 4u * threadIdx.x, rank), -1);
    if (rank == 0 && warp == 0) {
      int t = 0;
      if (lane == 0) {
        t = atomicAdd(&ctrl[kBackward ? 1 : 0], 1);
        // after an abort, in this sweep or an earlier one of the call: stop
        if (ld_relaxed_int(ctrl + 2) || (ld_relaxed_int(status) & kStatTimeout)) t = nblocks;
      }
      t = __shfl_sync(0xffffffffu, t, 0);
      if (lane < nby * nbz) store_cluster(map_rank(words + 12 + 4 * turn, (unsigned)lane), t);
    }
    cluster_sync();
    const int t = load_ctrl(words + 12 + 4 * turn);
    if (t >= nblocks) return;
    int CY, CZ;
    block_of_ticket(t, ncy, ncz, CY, CZ);
    pc.Ym = CY * nby + pc.by;
    pc.Zm = CZ * nbz + pc.bz;
    if (pc.Ym < sh.nty && pc.Zm < sh.ntz) {
      if (warp == 0) {
        main_warp<T, kBackward, kFlat>(sh, out, smem_raw, lane, pc);
      } else if (warp == 1) {
        edge_warp<T, kBackward, kFlat>(sh, ctrl + 2, status, smem_raw, lane, pc);
      } else if (warp == 2) {
        stager_warp<T, kBackward, kFlat>(sh, ops, smem_raw, lane, pc);
      } else if (warp == 3) {
        feeder_warp<T, kBackward, kFlat>(sh, mark, ctrl + 2, status, smem_raw, lane, pc);
      } else {
        if (warp == kTeam && lane == 0) {
          // the tile's operands into L2 while it waits for its turn
          const int Y = kBackward ? sh.nty - 1 - pc.Ym : pc.Ym, Z = kBackward ? sh.ntz - 1 - pc.Zm : pc.Zm;
          const T* src = ops + (kSpare + (long long)(Y + sh.nty * Z) * sh.ns) * L::kRec;
          for (int r = 0; r < sh.ns; r += 16)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src + (long long)r * L::kRec),
                         "r"((unsigned)((sh.ns - r < 16 ? sh.ns - r : 16) * L::kRec * (int)sizeof(T))));
        }
        __syncwarp();
        helper_warp<T, kBackward, kFlat>(sh, out, ctrl + 2, status, smem_raw, warp - kTeam, lane, pc);
      }
    }
    // (a warp that gave up comes here too: the others see the abort flag in
    // their waits, and the next claim ends the cluster)
    cluster_sync();
  }
}

inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }

// Clusters of a sweep.  A tile is at work for ns steps; the next anti-diagonal
// of blocks starts a block's skew and one hand-over later, so only that many
// anti-diagonals are ever active.  Launching no more keeps the rest of the GPU
// free for other streams.
template <class T, bool kFlat>
int sweep_clusters(const Shape& sh, int nby, int nbz) {
  using L = Tile<T, kFlat>;
  const int ncy = (sh.nty + nby - 1) / nby, ncz = (sh.ntz + nbz - 1) / nbz;
  const int width = ncy < ncz ? ncy : ncz;
  const int hop = (kFlat ? nby * L::TY : nbz * L::TZ) + 4;
  const long long want = (long long)width * (sh.ns / hop + 3), n = (long long)ncy * ncz;
  return (int)(want < n ? want : n);
}

// The vectors of one precision's smoother.
template <class T>
struct IluSet {
  const T *Ad, *Ax, *Ay, *Az;
  const T *Axu, *Ayu, *Azu;
  const T* dinv;
  T *lo, *up, *z;
  T *b, *x;
};

IluSet<double> set_of(Buffers& b, double*) {
  return IluSet<double>{b.Ad, b.Ax, b.Ay, b.Az, b.Axu, b.Ayu, b.Azu, b.dinv,
                        b.lo, b.up, b.z, b.f, b.p};
}
// b = the outer residual's FP32 copy (written with it by launch_residual)
IluSet<float> set_of(Buffers& b, float*) {
  const SingleBuffers& f = b.f32;
  return IluSet<float>{f.Ad, f.Ax, f.Ay, f.Az, f.Axu, f.Ayu, f.Azu, f.dinv,
                       f.lo, f.up, f.z, f.r, f.d};
}

// cta: blocks of kBlock tiles per cluster, else one tile per CTA on its own.
template <class T, bool kBackward, bool kFlat>
cudaError_t run_sweep(const Geo& g, const Shape& sh, const IluSet<T>& v, bool cta, int* ctrl, int* status,
                      cudaStream_t s) {
  using Pl = Plan<T, kFlat>;
  // 8 CTAs a cluster (the portable limit).  Measured at 200 x 200 x 100, FP32 /
  // FP64: 2 x 4 tiles 98 / 145 us, 4 x 2 98 / 147, 8 x 1 118 / 159, 1 x 8
  // 159 / 199, no clusters 122 / 188 (hand-overs through L2 only).
  // A grid of one row of tiles takes its clusters along it: half of their CTAs
  // would have no tile, and be counted in the hand-overs (1 x 1 x 20000, FP32: a
  // sweep of 8.7 ms with 2 x 4, 4.4 with 1 x 8; 300 x 300 x 3: 74 and 70 us).
  const int nbz = !cta || kFlat || sh.ntz == 1 ? 1 : sh.nty == 1 ? 8 : sh.ntz >= 4 ? 4 : 2;
  const int nby = cta ? kSweepCtas / nbz : 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)(sweep_clusters<T, kFlat>(sh, nby, nbz) * nby * nbz));
  c.blockDim = dim3(Pl::kThreads);
  c.dynamicSmemBytes = Pl::kBytes;
  c.stream = s;
  cudaLaunchAttribute a[2];
  a[0].id = cudaLaunchAttributeClusterDimension;
  a[0].val.clusterDim.x = (unsigned)(nby * nbz);
  a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
  a[1] = pdl_attribute();
  c.attrs = a;
  c.numAttrs = pdl_grid(g) ? 2 : 1;
  return cudaLaunchKernelEx(&c, k_sweep<T, kBackward, kFlat>, sh, (const T*)(kBackward ? v.up : v.lo),
                            kBackward ? v.z : v.up, kBackward ? v.up : v.z, ctrl, status, nby, nbz);
}

template <class T, bool kFlat>
cudaError_t sweep_impl(const Geo& g, Buffers& b, bool backward, bool pipelined, bool cta, cudaStream_t s) {
  const Shape sh = shape_of<T, kFlat>(g);
  const IluSet<T> v = set_of(b, (T*)nullptr);
  if (!pipelined) {
    const int blocks = blocks_for((long long)g.ny * g.nz, 256);
    const int levels = g.nx + g.ny + g.nz - 2;
    for (int L = 0; L < levels; ++L) {
      if (!backward) k_sweep_level<T, false, kFlat><<<blocks, 256, 0, s>>>(g, sh, L, v.lo, v.up, Tile<T, kFlat>::kRec);
      else k_sweep_level<T, true, kFlat><<<blocks, 256, 0, s>>>(g, sh, L, v.up, v.z, Tile<T, kFlat>::kVec);
    }
    count_launches(levels);
    return cudaGetLastError();
  }
  count_launches(1);
  return backward ? run_sweep<T, true, kFlat>(g, sh, v, cta, b.ctrl, b.status, s)
                  : run_sweep<T, false, kFlat>(g, sh, v, cta, b.ctrl, b.status, s);
}

// The CTAs of a layout conversion, the tiles of one piece of x after another (in
// one dimension of the grid: a second one would end at 65535 pieces).
template <class T>
dim3 layout_grid(const Geo& g, const Shape& sh) {
  return dim3((unsigned)(sh.nty * sh.ntz) * (unsigned)((g.nx + kXC<T> - 1) / kXC<T>));
}

template <class T, bool kFlat>
cudaError_t resid_impl(const Geo& g, Buffers& b, cudaStream_t s) {
  const Shape sh = shape_of<T, kFlat>(g);
  const IluSet<T> v = set_of(b, (T*)nullptr);
  const dim3 grid = layout_grid<T>(g, sh);
  count_launches(1);
  return launch_after(pdl_grid(g), v.Axu != v.Ax ? k_resid_scaled<T, true, kFlat> : k_resid_scaled<T, false, kFlat>,
                      grid, 256, 0, s, g, sh, v.Ad, v.Ax, v.Ay, v.Az, v.Axu, v.Ayu, v.Azu, v.b, v.x,
                      v.dinv, v.lo, b.ctrl);
}

template <class T, bool kFlat>
cudaError_t apply_impl(const Geo& g, Buffers& b, cudaStream_t s) {
  const Shape sh = shape_of<T, kFlat>(g);
  const IluSet<T> v = set_of(b, (T*)nullptr);
  const dim3 grid = layout_grid<T>(g, sh);
  count_launches(1);
  return launch_after(pdl_grid(g), k_apply_z<T, kFlat>, grid, 256, 0, s, g, sh, v.z, v.x);
}

template <class T, bool kFlat>
cudaError_t prepare_impl(const Geo& g, Buffers& b, bool pipelined, cudaStream_t s) {
  const Shape sh = shape_of<T, kFlat>(g);
  const IluSet<T> v = set_of(b, (T*)nullptr);
  int n = 1;
  if (pipelined) {
    // w (operand 0 of up) starts "not computed" (the sweeps keep its edge rows
    // and z's so from here on; z is marked by the first forward sweep)
    using L = Tile<T, kFlat>;
    const long long len = ilu_sweep_len(g, sizeof(T) == 4);
    k_fill_unset<T><<<blocks_for(len, 256), 256, 0, s>>>(len, L::kVec, L::kRec, v.up);
    ++n;
  }
  k_ilu_scale<T, kFlat><<<blocks_for(g.N, 256), 256, 0, s>>>(g, sh, v.Ax, v.Ay, v.Az, v.Axu, v.Ayu,
                                                            v.Azu, v.dinv, v.lo, v.up);
  count_launches(n);
  return cudaGetLastError();
}

template <class T, bool kFlat>
bool allow_smem(int max_smem) {
  constexpr int bytes = Plan<T, kFlat>::kBytes;
  return bytes <= max_smem && raise_smem_limit(k_sweep<T, false, kFlat>, bytes) == cudaSuccess &&
         raise_smem_limit(k_sweep<T, true, kFlat>, bytes) == cudaSuccess;
}

template <class T, bool kFlat>
bool cluster_ok() {
  return cluster_fits(k_sweep<T, false, kFlat>, kSweepCtas, Plan<T, kFlat>::kThreads, Plan<T, kFlat>::kBytes) &&
         cluster_fits(k_sweep<T, true, kFlat>, kSweepCtas, Plan<T, kFlat>::kThreads, Plan<T, kFlat>::kBytes);
}

}  // namespace

namespace {
template <class T, bool kFlat>
long long sweep_len(const Geo& g) {
  const Shape s = shape_of<T, kFlat>(g);
  return ((long long)s.nty * s.ntz * s.ns + 2 * kSpare) * Tile<T, kFlat>::kVec;
}
}  // namespace

bool ilu_sweep_smem(int max_smem) {
  const bool ok = allow_smem<float, false>(max_smem) && allow_smem<double, false>(max_smem) &&
                  allow_smem<float, true>(max_smem) && allow_smem<double, true>(max_smem);
  if (!ok) cudaGetLastError();
  return ok;
}

#define CAMS_BY_SHAPE(fn, ...)                                                       \
  (single ? (g.nz == 1 ? fn<float, true>(__VA_ARGS__) : fn<float, false>(__VA_ARGS__)) \
          : (g.nz == 1 ? fn<double, true>(__VA_ARGS__) : fn<double, false>(__VA_ARGS__)))

bool ilu_cluster_ok(const Geo& g, bool single) { return CAMS_BY_SHAPE(cluster_ok); }

long long ilu_sweep_len(const Geo& g, bool single) { return CAMS_BY_SHAPE(sweep_len, g); }

cudaError_t launch_ilu_prepare(const Geo& g, Buffers& b, bool pipelined, bool single,
                               cudaStream_t s) {
  return CAMS_BY_SHAPE(prepare_impl, g, b, pipelined, s);
}

cudaError_t launch_ilu_resid(const Geo& g, Buffers& b, bool single, cudaStream_t s) {
  return CAMS_BY_SHAPE(resid_impl, g, b, s);
}

cudaError_t launch_ilu_sweep(const Geo& g, Buffers& b, bool backward, bool pipelined, bool cta,
                             bool single, cudaStream_t s) {
  return CAMS_BY_SHAPE(sweep_impl, g, b, backward, pipelined, cta, s);
}

cudaError_t launch_ilu_apply(const Geo& g, Buffers& b, bool single, cudaStream_t s) {
  return CAMS_BY_SHAPE(apply_impl, g, b, s);
}

}  // namespace cams
