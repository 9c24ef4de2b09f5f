// ILU(0) factorisation of the second-stage smoother (Sec. 3, Table 1 step 6)
// for the 7-point matrix in natural order.  For this stencil ILU(0) only
// changes the diagonal: d_i = a_ii - sum_{j in {i-1, i-nx, i-nx*ny}} a_ij a_ji / d_j,
// and M = (D + L_A) D^{-1} (D + U_A) with L_A, U_A the strict triangles of A
// (the solves with M are in k_sweep.cu).  For a nonsymmetric A (the
// full-Jacobian step) the recurrence takes the products a_{i,j} a_{j,i},
// formed once per factorisation.  In mixed precision it is the factorisation
// of an FP32 copy of A.  Operands and pivots are in the natural layout.
//
// Two schedules of the same arithmetic (bitwise identical results):
//  * level-scheduled: one launch per hyperplane x+y+z = L (reference);
//  * pipelined: one persistent launch.  The (y, z) cross-section is cut into
//    tiles of kIluTY x kIluTZ = 32 x-rows; each warp takes a whole tile and
//    steps through it, row (ty, tz) working on x = s - ty - tz at step s.
//    The values a row needs from rows y-1 and z-1 of its own tile were
//    produced by the neighbouring lanes one step earlier and arrive by warp
//    shuffle.  Operands are staged by cp.async into a shared-memory ring
//    kG - 1 groups of kU steps ahead.  Values from another tile are read from
//    the output vector itself, which is pre-filled with a signalling-NaN
//    sentinel that no arithmetic produces: a value is ready once it differs
//    from the sentinel, so no flags or fences are needed (values are written
//    and read with single-copy atomic relaxed accesses at device scope); they
//    are fetched one group ahead and re-polled only when still unset.  Tiles
//    are claimed through an atomic ticket in anti-diagonal order, so a warp
//    only ever waits on tiles already claimed by running warps: no
//    co-residency assumption, no deadlock.  Every wait has an iteration
//    limit; on expiry the kernel sets an abort flag and the status word and
//    all warps leave.  One CTA of four warps per SM keeps one sweeping warp
//    per FP64 pipe.
#include "cams_internal.h"

namespace cams {

namespace {

constexpr int kTY = kIluTY, kTZ = kIluTZ, kR = kIluR;
static_assert(kR == 32, "a tile is one warp");
constexpr int kWarps = 4;                    // tiles in flight per CTA (one per FP64 pipe)
constexpr int kU = 4;                        // steps per group (straight-line code)
constexpr int kG = 3;                        // operand ring slots (groups staged kG - 1 ahead)
constexpr long long kSpinLimit = 1LL << 22;  // polls before a wait gives up (~ a second)
constexpr int kFastPolls = 64;               // in-loop polls before a wait starts to sleep

// Bit pattern of a value and the "not computed yet" sentinel: a signalling
// NaN.  IEEE arithmetic never produces a signalling NaN, so no computed
// value carries this pattern.
template <class T>
struct Word;
template <>
struct Word<double> {
  using U = unsigned long long;
  static constexpr U kNotReady = 0x7FF4DEADBEEF0001ull;
  static __device__ __forceinline__ double value(U u) { return __longlong_as_double((long long)u); }
};
template <>
struct Word<float> {
  using U = unsigned;
  static constexpr U kNotReady = 0x7FA5A5A1u;
  static __device__ __forceinline__ float value(U u) { return __uint_as_float(u); }
};

template <class T>
__device__ __forceinline__ T not_ready() {
  return Word<T>::value(Word<T>::kNotReady);
}

constexpr int kFactorCtrl = 4;               // control words: 4 of the sweeps', then the factorisation's

struct Skew {
  int nty, ntz, ns;   // tiles in y and z, steps per tile (a multiple of kU)
};

inline Skew make_skew(const Geo& g) {
  const int ns = g.nx + kTY + kTZ - 2;
  return Skew{(g.ny + kTY - 1) / kTY, (g.nz + kTZ - 1) / kTZ, (ns + kU - 1) / kU * kU};
}

// ---- relaxed device-scope accesses, copies (8- or 4-byte values) ----
__device__ __forceinline__ unsigned long long ld_relaxed(const double* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ unsigned ld_relaxed(const float* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// ld_relaxed when `pred` holds, else 0 (a predicated load: no branch).
__device__ __forceinline__ unsigned long long ld_relaxed_if(bool pred, const double* p) {
  unsigned long long v = 0ull;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.relaxed.gpu.global.b64 %0, [%1];\n\t}"
      : "+l"(v)
      : "l"(p), "r"((unsigned)pred));
  return v;
}
__device__ __forceinline__ unsigned ld_relaxed_if(bool pred, const float* p) {
  unsigned v = 0u;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.relaxed.gpu.global.b32 %0, [%1];\n\t}"
      : "+r"(v)
      : "l"(p), "r"((unsigned)pred));
  return v;
}

__device__ __forceinline__ int ld_relaxed_int(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ void publish(double* p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v));
}
__device__ __forceinline__ void publish(float* p, float v) {
  asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v));
}

__device__ __forceinline__ void cp_async(double* smem_dst, const double* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async(float* smem_dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------------------ parallel parts ---

template <class T>
__global__ void k_fill_not_ready(long long n, T* a) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) a[i] = not_ready<T>();
}

// FP32 copy of the 7-point matrix (mixed precision)
__global__ void k_matrix_to_single(long long n, const double* __restrict__ Ad,
                                   const double* __restrict__ Ax, const double* __restrict__ Ay,
                                   const double* __restrict__ Az, float* sd, float* sx, float* sy,
                                   float* sz) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  sd[i] = (float)Ad[i];
  sx[i] = (float)Ax[i];
  sy[i] = (float)Ay[i];
  sz[i] = (float)Az[i];
}

// FP32 copies of three arrays (the transposed couplings of a nonsymmetric A)
__global__ void k_three_to_single(long long n, const double* __restrict__ a,
                                  const double* __restrict__ b, const double* __restrict__ c,
                                  float* sa, float* sb, float* sc) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  sa[i] = (float)a[i];
  sb[i] = (float)b[i];
  sc[i] = (float)c[i];
}

// Q_d[i] = a_{i,i-e_d} a_{i-e_d,i}: the pivot recurrence's products
template <class T>
__global__ void k_pivot_products(long long n, const T* __restrict__ Ax, const T* __restrict__ Ay,
                                 const T* __restrict__ Az, const T* __restrict__ Axu,
                                 const T* __restrict__ Ayu, const T* __restrict__ Azu, T* Qx,
                                 T* Qy, T* Qz) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  Qx[i] = Ax[i] * Axu[i];
  Qy[i] = Ay[i] * Ayu[i];
  Qz[i] = Az[i] * Azu[i];
}

// p += delta (mixed precision: the FP32 correction enters the FP64 iterate)
__global__ void k_add_correction(long long n, const float* __restrict__ d, double* p) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  p[i] += (double)d[i];
}

// -------------------------------------------------- per-cell operator ---
// "value = op(cell, operands, values of the three upstream neighbours)", with
// 0 standing for a neighbour outside the grid (its coupling is 0 as well).
// src(a, i) is the address of operand a of cell i; apply() combines the
// operands with the upstream values and publishes the result.  `cell` is
// false on the pipeline's fill/drain slots and on rows beyond the grid:
// there the result is discarded and nothing is written.

// d = a_ii - a_{i,x-1}^2 / d_{x-1} - a_{i,y-1}^2 / d_{y-1} - a_{i,z-1}^2 / d_{z-1};
// kProd: the operands are the products a_{i,i-e} a_{i-e,i} (nonsymmetric A)
template <class T, bool kProd = false>
struct Factor {
  using Scalar = T;
  static constexpr int kN = 4;
  const T *Ad, *Ax, *Ay, *Az;
  T* dinv;
  int* status;
  __device__ __forceinline__ const T* src(int a, long long i) const {
    return (a == 0 ? Ad : a == 1 ? Ax : a == 2 ? Ay : Az) + i;
  }
  __device__ __forceinline__ T apply(const T* in, long long i, bool cell, T vx, T vy,
                                     T vz) const {
    T d = in[0];
    if constexpr (kProd) {
      d -= in[1] * vx;
      d -= in[2] * vy;
      d -= in[3] * vz;
    } else {
      d -= in[1] * in[1] * vx;
      d -= in[2] * in[2] * vy;
      d -= in[3] * in[3] * vz;
    }
    if (cell && (!(d != T(0)) || !isfinite(d))) {
      atomicOr(status, kStatSingular);
      d = T(1);
    }
    const T v = T(1) / d;
    if (cell) publish(dinv + i, v);
    return v;
  }
};

// ---------------------------------------------------- level schedule ---

template <class Op>
__global__ void k_factor_level(Geo g, int L, Op op, const typename Op::Scalar* vals) {
  using T = typename Op::Scalar;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)g.ny * g.nz) return;
  const int y = (int)(t % g.ny), z = (int)(t / g.ny);
  const int x = L - y - z;
  if (x < 0 || x >= g.nx) return;
  const long long i = x + g.sy * y + g.sz * z;
  T in[Op::kN];
#pragma unroll
  for (int a = 0; a < Op::kN; ++a) in[a] = *op.src(a, i);
  op.apply(in, i, true, x > 0 ? vals[i - 1] : T(0), y > 0 ? vals[i - g.sy] : T(0),
           z > 0 ? vals[i - g.sz] : T(0));
}

// ------------------------------------------------ pipelined schedule ---

__device__ __forceinline__ void tile_of_ticket(int t, int nty, int ntz, int& Y, int& Z) {
  // anti-diagonals d = Y + Z in increasing order, Y ascending within one
  for (int d = 0;; ++d) {
    const int ylo = d - (ntz - 1) > 0 ? d - (ntz - 1) : 0;
    const int yhi = d < nty - 1 ? d : nty - 1;
    const int cnt = yhi - ylo + 1;
    if (t < cnt) {
      Y = ylo + t;
      Z = d - Y;
      return;
    }
    t -= cnt;
  }
}

// Polls *p until it holds a published value; returns its bits, or the
// sentinel after an abort or a timeout (the status word and the abort flag
// are then set).  A light loop (one address, a short sleep between polls)
// for the long wait before a tile's first step: heavy polling there slows
// the tile's first steps and every tile downstream of it.
template <class T>
__device__ __forceinline__ typename Word<T>::U wait_bits(const T* p, int* abort_flag, int* status) {
  unsigned nap = 32;
  for (long long it = 0; it < kSpinLimit; ++it) {
    const typename Word<T>::U b = ld_relaxed(p);
    if (b != Word<T>::kNotReady) return b;
    if ((it & 63) == 63 && ld_relaxed_int(abort_flag)) return Word<T>::kNotReady;
    __nanosleep(nap);
    nap = nap < 256 ? 2 * nap : 256;      // back off while the upstream tile is far away
  }
  atomicOr(status, kStatTimeout);
  atomicExch(abort_flag, 1);
  return Word<T>::kNotReady;
}

// One tile of the factorisation, run by one warp: the tile at (Y, Z), ring:
// this warp's operand ring.  Values from other tiles are read from `out`.
// Before its first step the tile waits (lightly) for the upstream values of
// its first group; steps then run in groups of kU: a group's prologue
// prefetches the next group's cross-tile values (they sit on the critical
// path, so they go ahead of the copies) and stages the operands of the group
// kG - 1 ahead; values still unset are re-polled together; the kU steps
// themselves are straight-line code.  Returns false after an abort or a
// timeout (the warp's copies drained).  kOwnEnd: the end of the tile's copies
// takes a path of its own (own_end; the arithmetic is the same).
template <class Op, bool kOwnEnd>
__device__ __forceinline__ bool factor_tile(const Geo& g, const Skew& sk, const Op& op,
                                            const typename Op::Scalar* out, int* abort_flag,
                                            int* status, typename Op::Scalar* ringw, int lane,
                                            int Y, int Z) {
  using T = typename Op::Scalar;
  using U = typename Word<T>::U;
  constexpr U kNR = Word<T>::kNotReady;
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int kN = Op::kN;
  const int ty = lane % kTY, tz = lane / kTY;       // row within the tile
  const int y = Y * kTY + ty, z = Z * kTZ + tz;
  const bool valid = y < g.ny && z < g.nz;
  const bool hy = valid && y > 0, hz = valid && z > 0;            // upstream rows exist
  const bool gy = hy && ty == 0, gz = hz && tz == 0;              // ... in another tile
  const int xoff = ty + tz;                                       // x is step - xoff
  const int yc = valid ? y : 0, zc = valid ? z : 0;               // rows beyond the grid read row 0
  const long long row = (long long)yc * g.sy + (long long)zc * g.sz;
  const long long i0 = row - xoff;
  const long long oy0 = i0 - g.sy, oz0 = i0 - g.sz;
  // Operands of steps gs .. gs+kU-1 into ring slot q, laid out
  // [slot][operand][step][lane], clamped to my row (read, then discarded).
  T* const ring = ringw + lane;
  auto stage = [&](int gs, int q) {
    if (kOwnEnd && gs >= sk.ns) {
      cp_async_commit();
      return;
    }
    if (kOwnEnd || gs < sk.ns) {
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        long long i = i0 + (gs + u);
        i = i < row ? row : i;
        i = i > row + g.nx - 1 ? row + g.nx - 1 : i;
#pragma unroll
        for (int a = 0; a < kN; ++a) cp_async(ring + ((q * kN + a) * kU + u) * kR, op.src(a, i));
      }
    }
    cp_async_commit();
  };
  // values of steps gs .. gs+kU-1 read from `out` (0 where none is needed)
  auto fetch = [&](int gs, U* cy, U* cz) {
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int xq = gs + u - xoff;
      const bool in_row = xq >= 0 && xq < g.nx;
      cy[u] = ld_relaxed_if(gy && in_row, out + oy0 + (gs + u));
      cz[u] = ld_relaxed_if(gz && in_row, out + oz0 + (gs + u));
    }
  };
  // the operands of the first kG - 1 groups do not depend on other tiles:
  // their copies overlap the first wait
#pragma unroll 1
  for (int gq = 0; gq < kG - 1; ++gq) stage(gq * kU, gq);
  {
    // The first group's upstream values (the first wait is the long one).
    // A tile publishes in step order, and among my edge lanes the one with
    // the largest skew needs the latest value, so that lane alone polls for
    // each direction (tz = 3 in y, ty = 7 in z): few pollers keep L2 quiet
    // for the tiles that are running.
    // (Every lane takes part in both shuffles.)
    const int xq = kU - 1 - xoff;
    bool ok = true;
    const bool in_row = xq >= 0 && xq < g.nx;
    const bool need_y = gy && in_row, need_z = gz && in_row;
    const bool des_y = __shfl_sync(kAll, need_y, ty + (kTZ - 1) * kTY);   // tz = 3 of my column
    const bool des_z = __shfl_sync(kAll, need_z, (kTY - 1) + tz * kTY);   // ty = 7 of my row
    const bool last_y = tz == kTZ - 1 || !des_y;
    const bool last_z = ty == kTY - 1 || !des_z;
    if (need_y && last_y) ok &= wait_bits(out + oy0 + (kU - 1), abort_flag, status) != kNR;
    if (need_z && last_z) ok &= wait_bits(out + oz0 + (kU - 1), abort_flag, status) != kNR;
    if (__any_sync(kAll, !ok)) {
      cp_async_wait<0>();
      return false;
    }
  }
  U cy[kU], cz[kU];
  fetch(0, cy, cz);
  T vprev = T(0), from_y = T(0), from_z = T(0);
  int q = 0;
  for (int s0 = 0; s0 < sk.ns; s0 += kU) {
    U ny_[kU], nz_[kU];
    fetch(s0 + kU, ny_, nz_);
    stage(s0 + (kG - 1) * kU, q == 0 ? kG - 1 : q - 1);
    // values still unset: re-poll them together (one round trip per poll)
    bool pending = false;
#pragma unroll
    for (int u = 0; u < kU; ++u) pending |= (cy[u] == kNR) | (cz[u] == kNR);
    if (__any_sync(kAll, pending)) {
      bool fail = false;
      for (long long it = 0; pending && !fail; ++it) {
        pending = false;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          if (cy[u] == kNR) {
            cy[u] = ld_relaxed(out + oy0 + (s0 + u));
            pending |= cy[u] == kNR;
          }
          if (cz[u] == kNR) {
            cz[u] = ld_relaxed(out + oz0 + (s0 + u));
            pending |= cz[u] == kNR;
          }
        }
        if (pending && it >= kFastPolls) {
          if (it >= kSpinLimit) {
            atomicOr(status, kStatTimeout);
            atomicExch(abort_flag, 1);
            fail = true;
          } else if ((it & 15) == 0 && ld_relaxed_int(abort_flag)) {
            fail = true;
          } else {
            __nanosleep(100);
          }
        }
      }
      if (__any_sync(kAll, fail)) {
        cp_async_wait<0>();
        return false;
      }
    }
    cp_async_wait<kG - 1>();
    T in[kU][kN];
#pragma unroll
    for (int u = 0; u < kU; ++u)
#pragma unroll
      for (int a = 0; a < kN; ++a) in[u][a] = ring[((q * kN + a) * kU + u) * kR];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int xs = s0 + u - xoff;
      const bool cell = valid && xs >= 0 && xs < g.nx;
      const T vy = hy ? (ty > 0 ? from_y : Word<T>::value(cy[u])) : T(0);
      const T vz = hz ? (tz > 0 ? from_z : Word<T>::value(cz[u])) : T(0);
      const T vx = xs > 0 ? vprev : T(0);
      const T v = op.apply(in[u], i0 + (s0 + u), cell, vx, vy, vz);
      // rows y-1 / z-1 of my tile computed my next neighbours just now
      from_y = __shfl_up_sync(kAll, v, 1);
      from_z = __shfl_up_sync(kAll, v, kTY);
      vprev = v;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      cy[u] = ny_[u];
      cz[u] = nz_[u];
    }
    q = q == kG - 1 ? 0 : q + 1;
  }
  cp_async_wait<0>();
  return true;
}

// Operand rings of a CTA's warps: [kWarps][kG][Op::kN][kU][32].
template <class Op>
constexpr int ring_bytes() {
  return (int)sizeof(typename Op::Scalar) * kWarps * kG * Op::kN * kU * kR;
}

// ctrl: [0] ticket, [1] abort flag.  `out` is the vector the operator
// publishes into (pre-filled with the sentinel on every cell).  Each warp
// claims tiles on its own.
template <class Op, bool kOwnEnd>
__global__ void __launch_bounds__(32 * kWarps, 1) k_factor(Geo g, Skew sk, Op op,
                                                            const typename Op::Scalar* out,
                                                            int* ctrl, int* status) {
  using T = typename Op::Scalar;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T* ringw = reinterpret_cast<T*>(smem_raw) + warp * (kG * Op::kN * kU * kR);
  const int ntiles = sk.nty * sk.ntz;
  for (;;) {
    int t = 0;
    if (lane == 0) t = atomicAdd(&ctrl[0], 1);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= ntiles) return;
    int Y, Z;
    tile_of_ticket(t, sk.nty, sk.ntz, Y, Z);
    if (!factor_tile<Op, kOwnEnd>(g, sk, op, out, ctrl + 1, status, ringw, lane, Y, Z)) return;
  }
}

// Bounded wait used by the self-test: polls a counter that nothing sets.
__device__ __forceinline__ bool wait_at_least(int* ctr, int need, int* abort_flag, int* status) {
  for (long long it = 0; it < kSpinLimit; ++it) {
    if (ld_relaxed_int(ctr) >= need) return true;
    if (ld_relaxed_int(abort_flag)) return false;
    __nanosleep(64);
  }
  atomicOr(status, kStatTimeout);
  atomicExch(abort_flag, 1);
  return false;
}

__global__ void k_wait_selftest(int* ctrl, int* status) {
  if (threadIdx.x == 0) wait_at_least(&ctrl[2], 1, &ctrl[1], status);
}

inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }

// The vectors of one precision's factorisation.
template <class T>
struct IluSet {
  const T *Ad, *Ax, *Ay, *Az;
  const T *Axu, *Ayu, *Azu;
  T *Qx, *Qy, *Qz;
  T* dinv;
};

IluSet<double> set_of(Buffers& b, double*) {
  return IluSet<double>{b.Ad, b.Ax, b.Ay, b.Az, b.Axu, b.Ayu, b.Azu, b.Qx, b.Qy, b.Qz, b.dinv};
}
IluSet<float> set_of(Buffers& b, float*) {
  const SingleBuffers& f = b.f32;
  return IluSet<float>{f.Ad, f.Ax, f.Ay, f.Az, f.Axu, f.Ayu, f.Azu, f.Qx, f.Qy, f.Qz, f.dinv};
}

// Which of the two forms of a tile's copies (the compiler schedules the step
// differently): with one commit for both cases an FP32 step takes 8% longer where a
// tile has an SM's issue slots nearly to itself (a row of 10^5 cells 23.9 against
// 22.2 ms, 4 x 4 x 16384 11.6 against 10.6, 1000 x 1000 839 against 803 us), and 1
// to 8% less where many tiles of both directions run (200 x 200 x 100 496 against
// 537 us, 128^3 323 against 334; 64^3, 8 tiles wide, 139.4 against 138.6).  FP64
// takes up to 2% less with a path of its own everywhere.
template <class T>
bool own_end(const Skew& sk) {
  return sizeof(T) == 8 || sk.nty <= 8 || sk.ntz <= 8;
}

// The pivot wavefront (level-scheduled or pipelined); returns the launch count.
template <class Op>
int factor_sweep(const Geo& g, Buffers& b, bool pipelined, int sms, const Op& fa,
                 typename Op::Scalar* dinv, cudaStream_t s, cudaError_t& e) {
  using T = typename Op::Scalar;
  e = cudaSuccess;
  if (!pipelined) {
    const int blocks = blocks_for((long long)g.ny * g.nz, 256);
    const int levels = g.nx + g.ny + g.nz - 2;
    for (int L = 0; L < levels; ++L) k_factor_level<Op><<<blocks, 256, 0, s>>>(g, L, fa, dinv);
    return levels;
  }
  const Skew sk = make_skew(g);
  int* ctrl = b.ctrl + kFactorCtrl;
  k_fill_not_ready<T><<<blocks_for(g.N, 256), 256, 0, s>>>(g.N, dinv);
  e = cudaMemsetAsync(ctrl, 0, 4 * sizeof(int), s);
  if (e != cudaSuccess) return 1;
  const int ctas = (sk.nty * sk.ntz + kWarps - 1) / kWarps;
  auto* kern = own_end<T>(sk) ? k_factor<Op, true> : k_factor<Op, false>;
  kern<<<ctas < sms ? ctas : sms, 32 * kWarps, ring_bytes<Op>(), s>>>(g, sk, fa, dinv, ctrl,
                                                                             b.status);
  e = cudaGetLastError();
  return 2;
}

template <class T>
cudaError_t factor_impl(const Geo& g, Buffers& b, bool pipelined, int sms, bool nonsym,
                        cudaStream_t s) {
  const IluSet<T> v = set_of(b, (T*)nullptr);
  int n = 0;
  cudaError_t e;
  if (nonsym) {
    k_pivot_products<T><<<blocks_for(g.N, 256), 256, 0, s>>>(g.N, v.Ax, v.Ay, v.Az, v.Axu, v.Ayu,
                                                             v.Azu, v.Qx, v.Qy, v.Qz);
    ++n;
    Factor<T, true> fa{v.Ad, v.Qx, v.Qy, v.Qz, v.dinv, b.status};
    n += factor_sweep(g, b, pipelined, sms, fa, v.dinv, s, e);
  } else {
    Factor<T> fa{v.Ad, v.Ax, v.Ay, v.Az, v.dinv, b.status};
    n += factor_sweep(g, b, pipelined, sms, fa, v.dinv, s, e);
  }
  if (e != cudaSuccess) return e;
  count_launches(n);
  return launch_ilu_prepare(g, b, pipelined, sizeof(T) == 4, s);
}

}  // namespace

int ilu_ctrl_ints(const Geo& g) {
  (void)g;
  return kFactorCtrl + 4;
}

bool ilu_set_smem() {
  auto allow = [](auto* kern, int bytes) { return raise_smem_limit(kern, bytes) == cudaSuccess; };
  return allow(k_factor<Factor<double>, true>, ring_bytes<Factor<double>>()) &&
         allow(k_factor<Factor<float>, true>, ring_bytes<Factor<float>>()) &&
         allow(k_factor<Factor<float>, false>, ring_bytes<Factor<float>>()) &&
         allow(k_factor<Factor<double, true>, true>, ring_bytes<Factor<double, true>>()) &&
         allow(k_factor<Factor<float, true>, true>, ring_bytes<Factor<float, true>>()) &&
         allow(k_factor<Factor<float, true>, false>, ring_bytes<Factor<float, true>>());
}

cudaError_t launch_ilu_factor(const Geo& g, Buffers& b, bool pipelined, int sms, bool single,
                              bool nonsym, cudaStream_t s) {
  if (single) {
    k_matrix_to_single<<<blocks_for(g.N, 256), 256, 0, s>>>(g.N, b.Ad, b.Ax, b.Ay, b.Az, b.f32.Ad,
                                                            b.f32.Ax, b.f32.Ay, b.f32.Az);
    count_launches(1);
    if (nonsym) {
      k_three_to_single<<<blocks_for(g.N, 256), 256, 0, s>>>(g.N, b.Axu, b.Ayu, b.Azu, b.f32.Axu,
                                                             b.f32.Ayu, b.f32.Azu);
      count_launches(1);
    }
    return factor_impl<float>(g, b, pipelined, sms, nonsym, s);
  }
  return factor_impl<double>(g, b, pipelined, sms, nonsym, s);
}

cudaError_t launch_add_correction(const Geo& g, Buffers& b, cudaStream_t s) {
  k_add_correction<<<blocks_for(g.N, 256), 256, 0, s>>>(g.N, b.f32.d, b.p);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_wait_selftest(const Geo& g, Buffers& b, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(b.ctrl, 0, sizeof(int) * (size_t)ilu_ctrl_ints(g), s);
  if (e != cudaSuccess) return e;
  k_wait_selftest<<<1, 32, 0, s>>>(b.ctrl + kFactorCtrl, b.status);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace cams
