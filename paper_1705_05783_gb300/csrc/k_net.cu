// Kernels of the learned basis surrogate: a small 3D convolutional network
// trained and evaluated on the GPU by these kernels alone.
//
// Layout: activations [B][C][S][S][S] (x fastest), FP32; weights
// [co][ci][27] with tap t = (dx+1) + 3 (dy+1) + 9 (dz+1) for the offsets
// d in {-1, 0, 1}^3; biases [co].  Every convolution is a 3x3x3
// cross-correlation with zero padding, output size = input size:
//   y[b][co][v] = bias[co] + sum_ci sum_t w[co][ci][t] x[b][ci][v + d(t)].
// Reductions run in a fixed order (no atomics), so results are
// bit-reproducible for a given launch.
#include <algorithm>
#include <map>
#include <mutex>

#include "cams_internal.h"

namespace cams {

namespace {

constexpr int kCoB = 8;        // output (or input) channels per thread
constexpr int kNetThreads = 256;

__device__ __forceinline__ void tap_offset(int t, int& dx, int& dy, int& dz) {
  dx = t % 3 - 1;
  dy = (t / 3) % 3 - 1;
  dz = t / 9 - 1;
}

// y = conv(x) + bias, optionally ReLU.  Each thread takes kVox voxels
// (kNetThreads apart) and kCoB output channels, so a weight read from shared
// memory feeds kVox FMAs and an input read kCoB.
// grid (ceil(S^3/(256 kVox)), ceil(co/8), B).
constexpr int kVox = 1;   // measured: 4 voxels a thread ran slower (fewer, fuller blocks)

__global__ void __launch_bounds__(kNetThreads) k_conv_fwd(int S, int ci, int co,
                                                          const float* __restrict__ x,
                                                          const float* __restrict__ w,
                                                          const float* __restrict__ bias,
                                                          int relu, float* __restrict__ y) {
  extern __shared__ float ws[];                 // [kCoB][ci][27]
  const int S3 = S * S * S;
  const int co0 = blockIdx.y * kCoB, b = blockIdx.z;
  const int nco = min(kCoB, co - co0);
  for (int e = threadIdx.x; e < kCoB * ci * 27; e += blockDim.x) {
    const int c = e / (ci * 27);
    ws[e] = c < nco ? w[(long long)(co0 + c) * ci * 27 + (e - c * ci * 27)] : 0.0f;
  }
  __syncthreads();
  int vv[kVox], vx[kVox], vy[kVox], vz[kVox];
#pragma unroll
  for (int k = 0; k < kVox; ++k) {
    vv[k] = blockIdx.x * (kNetThreads * kVox) + k * kNetThreads + threadIdx.x;
    const int v = min(vv[k], S3 - 1);
    vx[k] = v % S; vy[k] = (v / S) % S; vz[k] = v / (S * S);
  }
  if (vv[0] >= S3) return;
  float acc[kVox][kCoB];
#pragma unroll
  for (int k = 0; k < kVox; ++k)
#pragma unroll
    for (int c = 0; c < kCoB; ++c) acc[k][c] = c < nco ? bias[co0 + c] : 0.0f;
  const float* xb = x + (long long)b * ci * S3;
  for (int i = 0; i < ci; ++i) {
    const float* xc = xb + (long long)i * S3;
    for (int t = 0; t < 27; ++t) {
      int dx, dy, dz;
      tap_offset(t, dx, dy, dz);
      float xv[kVox];
#pragma unroll
      for (int k = 0; k < kVox; ++k) {
        const int ux = vx[k] + dx, uy = vy[k] + dy, uz = vz[k] + dz;
        xv[k] = (ux < 0 || ux >= S || uy < 0 || uy >= S || uz < 0 || uz >= S) ? 0.0f
                                                                               : xc[ux + S * (uy + S * uz)];
      }
#pragma unroll
      for (int c = 0; c < kCoB; ++c) {
        const float wv = ws[(c * ci + i) * 27 + t];
#pragma unroll
        for (int k = 0; k < kVox; ++k) acc[k][c] += wv * xv[k];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < kVox; ++k) {
    if (vv[k] >= S3) continue;
    float* yb = y + ((long long)b * co + co0) * S3 + vv[k];
#pragma unroll
    for (int c = 0; c < kCoB; ++c)
      if (c < nco) yb[(long long)c * S3] = relu ? fmaxf(acc[k][c], 0.0f) : acc[k][c];
  }
}

// gx[b][i][v] = sum_co sum_t w[co][i][t] gy[b][co][v - d(t)], times the ReLU
// mask (xact > 0) of the layer input when xact is given.
// grid (ceil(S^3/256), ceil(ci/8), B).
__global__ void __launch_bounds__(kNetThreads) k_conv_bwd_data(int S, int ci, int co,
                                                               const float* __restrict__ gy,
                                                               const float* __restrict__ w,
                                                               const float* __restrict__ xact,
                                                               float* __restrict__ gx) {
  extern __shared__ float ws[];                 // [kCoB][co][27]: w[c][i0 + k][t] at (k*co + c)*27 + t
  const int S3 = S * S * S;
  const int ci0 = blockIdx.y * kCoB, b = blockIdx.z;
  const int nci = min(kCoB, ci - ci0);
  for (int e = threadIdx.x; e < kCoB * co * 27; e += blockDim.x) {
    const int k = e / (co * 27), rem = e - k * co * 27, c = rem / 27, t = rem - c * 27;
    ws[e] = k < nci ? w[((long long)c * ci + ci0 + k) * 27 + t] : 0.0f;
  }
  __syncthreads();
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= S3) return;
  const int vx = v % S, vy = (v / S) % S, vz = v / (S * S);
  float acc[kCoB];
#pragma unroll
  for (int k = 0; k < kCoB; ++k) acc[k] = 0.0f;
  const float* gb = gy + (long long)b * co * S3;
  for (int c = 0; c < co; ++c) {
    const float* gc = gb + (long long)c * S3;
    for (int t = 0; t < 27; ++t) {
      int dx, dy, dz;
      tap_offset(t, dx, dy, dz);
      const int ux = vx - dx, uy = vy - dy, uz = vz - dz;
      if (ux < 0 || ux >= S || uy < 0 || uy >= S || uz < 0 || uz >= S) continue;
      const float g = gc[ux + S * (uy + S * uz)];
#pragma unroll
      for (int k = 0; k < kCoB; ++k) acc[k] += ws[(k * co + c) * 27 + t] * g;
    }
  }
  const long long o = ((long long)b * ci + ci0) * S3 + v;
#pragma unroll
  for (int k = 0; k < kCoB; ++k) {
    if (k >= nci) continue;
    float val = acc[k];
    if (xact && !(xact[o + (long long)k * S3] > 0.0f)) val = 0.0f;
    gx[o + (long long)k * S3] = val;
  }
}

// gw[o][i][t] = sum_b sum_v gy[b][o][v] x[b][i][v + d(t)]; gbias[o] = sum gy[b][o][v].
// One CTA per (o, i): grid (ci, co).
__global__ void __launch_bounds__(kNetThreads) k_conv_bwd_w(int B, int S, int ci, int co,
                                                            const float* __restrict__ x,
                                                            const float* __restrict__ gy,
                                                            float* __restrict__ gw,
                                                            float* __restrict__ gbias) {
  __shared__ float red[28][kNetThreads / 32];
  const int i = blockIdx.x, o = blockIdx.y;
  const int S3 = S * S * S;
  float acc[28];
#pragma unroll
  for (int t = 0; t < 28; ++t) acc[t] = 0.0f;
  for (int b = 0; b < B; ++b) {
    const float* xc = x + ((long long)b * ci + i) * S3;
    const float* gc = gy + ((long long)b * co + o) * S3;
    for (int v = threadIdx.x; v < S3; v += blockDim.x) {
      const float g = gc[v];
      if (g == 0.0f) continue;
      const int vx = v % S, vy = (v / S) % S, vz = v / (S * S);
      acc[27] += g;
#pragma unroll
      for (int t = 0; t < 27; ++t) {
        const int dx = t % 3 - 1, dy = (t / 3) % 3 - 1, dz = t / 9 - 1;
        const int ux = vx + dx, uy = vy + dy, uz = vz + dz;
        if (ux < 0 || ux >= S || uy < 0 || uy >= S || uz < 0 || uz >= S) continue;
        acc[t] += g * xc[ux + S * (uy + S * uz)];
      }
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int t = 0; t < 28; ++t) {
    float s = acc[t];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) red[t][wid] = s;
  }
  __syncthreads();
  if (threadIdx.x < 28) {
    float s = 0.0f;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[threadIdx.x][k];
    if (threadIdx.x < 27) gw[((long long)o * ci + i) * 27 + threadIdx.x] = s;
    else if (i == 0) gbias[o] = s;
  }
}

// ---- register-tiled convolutions ----
// The kernels above issue a shared-memory read and a predicated load per eight
// FMAs, and the weight gradient one load per FMA.  Here a thread holds a tile
// of results and every value read from shared memory feeds several of them;
// inputs are staged zero-padded, rows cut into strips of 4 voxels, so the inner
// loops have no conditions, and two FMAs go in one instruction.  What bounds
// them then is how many warps a CTA's registers and staging leave (9 an SM in the
// convolutions, which issue in 0.40 to 0.42 of the cycles, 13 in the weight
// gradient, 0.57), next the FP32 rate: 2.4e9
// FMAs of 32 x 32 channels on 64 patches of 11^3 take 60 us at it.
constexpr int kStrip = 4;      // voxels of a strip (one 16-byte read)
constexpr int kCiB = 4;        // input channels staged at a time (two stages in flight)
// staged values per thread and channel (fewer output channels a thread leave
// registers for more)
constexpr int slots_of(int ko) { return ko == 8 ? 12 : 20; }

// Asynchronous 4-byte copy into shared memory; zero when !in (src is not read).
__device__ __forceinline__ void copy4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(in ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Two FP32 values in a register pair, and two FMAs in one instruction (each
// rounded as a single one is).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

struct ConvTile {
  int NS, P;                   // strips per row, pitch of a staged row (floats)
  int NYP, PR;                 // row pairs per plane, staged rows per plane
  int ko, ncg, ST;             // output channels a thread, groups of them; strip pairs of a CTA
  int planes;                  // staged planes, halo included
  int smem;
};

ConvTile conv_tile(int B, int S, int co, int sms) {
  ConvTile t;
  t.NS = (S + kStrip - 1) / kStrip;
  t.P = kStrip * t.NS + 4;     // x = -1 .. 4 NS, and the rest of the last 16 bytes
  t.NYP = (S + 1) / 2;
  t.PR = 2 * t.NYP + 2;
  t.ko = co > 8 ? 8 : 4;
  t.ncg = co > 16 ? 4 : co > 4 ? 2 : 1;
  const int per = t.NYP * t.NS, q = 32 / t.ncg;
  const long long n = (long long)S * per, groups = (co + 31) / 32;
  // whole warps, 64 to 256 threads: the size that gives the busiest SM the
  // least to do (an SM works on several CTAs at once, a larger one stages less
  // per strip)
  t.ST = 0;
  long long best = 0;
  for (int st = 256 / t.ncg; st >= 64 / t.ncg; st -= q) {
    const long long load = (B * groups * ((n + st - 1) / st) + sms - 1) / sms * st;
    if (t.ST == 0 || load < best) {
      t.ST = st;
      best = load;
    }
  }
  const int span = (t.ST - 1 + per - 1) / per + 1;
  t.planes = (span < S ? span : S) + 2;
  const long long chan = (long long)t.planes * t.PR * t.P;
  const long long bytes = 2 * kCiB * (chan + 27 * (t.ncg * t.ko + 4)) * 4;
  // (too large to stage: no tile)
  t.smem = chan > (long long)slots_of(t.ko) * t.ST * t.ncg || bytes > (1 << 30) ? 1 << 30 : (int)bytes;
  return t;
}

// y = conv(x) over `ci` input and `co` output channels.  A thread has two rows'
// strips (y, y + 1) and KO output channels: 8 KO sums, and per input plane 44
// shared reads (4 rows, each tap's weights for the row pair; KO = 8) feed 576
// FMAs.  A warp's lanes are strip pairs x channel groups, so that its reads of
// the weights and of the rows each touch few addresses.
// kBwd: the data gradient, the same sum with the taps reversed and the weights
// transposed (w is [ci][co][27] then), masked by xact > 0 instead of bias and
// ReLU.  grid (strip blocks, output channels / 32, B).
template <bool kBwd, int KO>
__global__ void __launch_bounds__(kNetThreads) k_conv_tile(int S, int ci, int co, ConvTile t,
                                                           const float* __restrict__ x,
                                                           const float* __restrict__ w,
                                                           const float* __restrict__ bias, int relu,
                                                           const float* __restrict__ xact,
                                                           float* __restrict__ y) {
  extern __shared__ __align__(16) float sm[];
  const int S3 = S * S * S, chan = t.planes * t.PR * t.P, nco = t.ncg * KO;
  constexpr int kSlots = slots_of(KO);
  const int wp = nco + 4;                       // pitch of a tap's weights
  const int stage = kCiB * (chan + 27 * wp);    // [2]{[kCiB][planes][PR][P], [kCiB][27][wp]}
  const int o0 = blockIdx.y * 32, b = blockIdx.z;
  const int first = blockIdx.x * t.ST, per = t.NYP * t.NS;
  const int z_lo = first / per - 1;             // plane of staged plane 0
  const int strip = first + threadIdx.x / t.ncg, cg = threadIdx.x % t.ncg;
  const int z = strip / per, y0 = strip % per / t.NS * 2, x0 = strip % t.NS * kStrip;
  const bool on = z < S;
  f32x2 acc[KO / 2][2][kStrip];                 // pairs of output channels
#pragma unroll
  for (int c = 0; c < KO / 2; ++c) {
    const int o = o0 + cg * KO + 2 * c;
    const f32x2 v = pack2(!kBwd && o < co ? bias[o] : 0.0f, !kBwd && o + 1 < co ? bias[o + 1] : 0.0f);
#pragma unroll
    for (int u = 0; u < kStrip; ++u) acc[c][0][u] = acc[c][1][u] = v;
  }
  const float* xb = x + (long long)b * ci * S3;
  // where my staged values come from (the same in every channel; -1: zero)
  int off[kSlots];
#pragma unroll
  for (int k = 0; k < kSlots; ++k) {
    const int e = threadIdx.x + k * blockDim.x;
    const int px = e % t.P - 1, r = e / t.P, py = r % t.PR - 1, pz = r / t.PR + z_lo;
    const bool in = (unsigned)px < (unsigned)S && (unsigned)py < (unsigned)S && (unsigned)pz < (unsigned)S;
    off[k] = in ? px + S * (py + S * pz) : -1;
  }
  auto fetch = [&](int i0, float* xs, float* ws) {
    const int nci = min(kCiB, ci - i0);
    for (int c = 0; c < nci; ++c) {
      const float* src = xb + (long long)(i0 + c) * S3;
#pragma unroll
      for (int k = 0; k < kSlots; ++k) {
        const int e = threadIdx.x + k * blockDim.x;
        if (e < chan) copy4(xs + c * chan + e, src + max(off[k], 0), off[k] >= 0);
      }
    }
    // a warp copies one tap's weights of all its channels (32 rows of memory, but
    // the next taps' values are in the same lines)
    const int o = threadIdx.x & 31;
    if (o < nco)
      for (int q = threadIdx.x >> 5; q < nci * 27; q += blockDim.x >> 5) {
        const int i = q / 27, tap = q - i * 27;
        const long long at = kBwd ? ((long long)(i0 + i) * co + o0 + o) * 27 + 26 - tap
                                  : ((long long)(o0 + o) * ci + i0 + i) * 27 + tap;
        copy4(ws + q * wp + o, w + (o0 + o < co ? at : 0), o0 + o < co);
      }
    copies_commit();
  };
  fetch(0, sm, sm + kCiB * chan);
  for (int i0 = 0, buf = 0; i0 < ci; i0 += kCiB, buf ^= 1) {
    const int nci = min(kCiB, ci - i0);
    const float* xs = sm + buf * stage;
    const float* ws = xs + kCiB * chan;
    if (i0 + kCiB < ci) {
      float* nx = sm + (buf ^ 1) * stage;
      fetch(i0 + kCiB, nx, nx + kCiB * chan);
      copies_wait<1>();
    } else {
      copies_wait<0>();
    }
    __syncthreads();
    if (on) {
      const float* xr0 = xs + ((z - 1 - z_lo) * t.PR + y0) * t.P + x0;
      const float* wr = ws + cg * KO;
      for (int c = 0; c < nci; ++c)
#pragma unroll 1
        for (int dz = 0; dz < 3; ++dz) {
          const float* xr = xr0 + c * chan + dz * t.PR * t.P;
          const float* wz = wr + (c * 27 + dz * 9) * wp;
          // row r of the four feeds output row 0 as dy = r and row 1 as dy = r - 1
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float4 a = *reinterpret_cast<const float4*>(xr + r * t.P);
            const float2 a2 = *reinterpret_cast<const float2*>(xr + r * t.P + 4);
            const f32x2 xv[6] = {pack2(a.x, a.x), pack2(a.y, a.y),   pack2(a.z, a.z),
                                 pack2(a.w, a.w), pack2(a2.x, a2.x), pack2(a2.y, a2.y)};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int dy = r - h;
              if (dy < 0 || dy > 2) continue;
#pragma unroll
              for (int dx = 0; dx < 3; ++dx) {
                const float* wq = wz + (dy * 3 + dx) * wp;
                f32x2 wv[KO / 2];
#pragma unroll
                for (int k = 0; k < KO / 4; ++k) {
                  const ulonglong2 w2 = *reinterpret_cast<const ulonglong2*>(wq + 4 * k);
                  wv[2 * k] = w2.x;
                  wv[2 * k + 1] = w2.y;
                }
#pragma unroll
                for (int k = 0; k < KO / 2; ++k)
#pragma unroll
                  for (int u = 0; u < kStrip; ++u)
                    acc[k][h][u] = fma2(wv[k], xv[u + dx], acc[k][h][u]);
              }
            }
          }
        }
    }
    __syncthreads();                            // the buffer is free for the copies after next
  }
  if (!on) return;
#pragma unroll
  for (int k = 0; k < KO; ++k) {
    const int o = o0 + cg * KO + k;
    if (o >= co) continue;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int yy = y0 + r;
      if (yy >= S) continue;
      const long long at = ((long long)b * co + o) * S3 + x0 + S * (yy + S * z);
#pragma unroll
      for (int u = 0; u < kStrip; ++u) {
        if (x0 + u >= S) continue;
        const float2 both = unpack2(acc[k / 2][r][u]);
        float v = k % 2 ? both.y : both.x;
        if constexpr (kBwd) {
          const bool edge = x0 + u == 0 || x0 + u == S - 1 || yy == 0 || yy == S - 1 || z == 0 || z == S - 1;
          if (!isfinite(v) && edge) {
            // a non-finite weight times the zero padding: the sum over the taps
            // inside the patch alone (over once it is NaN)
            v = 0.0f;
            for (int i = 0; i < ci && !isnan(v); ++i)
              for (int tap = 0; tap < 27 && !isnan(v); ++tap) {
                int dx, dy, dz;
                tap_offset(tap, dx, dy, dz);
                const int ux = x0 + u - dx, uy = yy - dy, uz = z - dz;
                if (ux < 0 || ux >= S || uy < 0 || uy >= S || uz < 0 || uz >= S) continue;
                v += w[((long long)i * co + o) * 27 + tap] * xb[(long long)i * S3 + ux + S * (uy + S * uz)];
              }
          }
          if (xact && !(xact[at + u] > 0.0f)) v = 0.0f;
        } else if (relu) {
          v = fmaxf(v, 0.0f);
        }
        y[at + u] = v;
      }
    }
  }
}

// Weight gradient, split over the planes (b, z) of the batch into nk chunks:
// part[chunk][o][i][27], and the bias gradient part_b[chunk][o].  A warp has 8
// output channels, its lanes 32 input channels, the CTA one dz: 72 sums a
// thread, and per strip 14 shared reads feed 288 FMAs.  The channels' staged
// planes start 16 bytes apart modulo the banks.  Lanes and warps that the
// channels leave over (nsl lane groups, nsw warp groups) take rows of their
// own, added up at the end.  grid (3, nk, tiles of 32 x 32).
__global__ void __launch_bounds__(kNetThreads, 2) k_conv_bwd_w_tile(int B, int S, int ci, int co,
                                                                    int NS, int P, int CP, int nk,
                                                                    int nsl, int nsw,
                                                                    const float* __restrict__ x,
                                                                    const float* __restrict__ gy,
                                                                    float* __restrict__ part,
                                                                    float* __restrict__ part_b) {
  extern __shared__ __align__(16) float sm[];
  const int S3 = S * S * S, Q = kStrip * NS;
  const int wpg = 8 / nsw, lpg = 32 / nsl;      // warps and lanes of a group
  // [2]{x: [lpg][CP], rows -1 .. S of plane z + dz, pitch P; gy: [4 wpg][S][Q][2]}
  const int stage = lpg * CP + wpg * 8 * S * Q;
  const int wl = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int lane = wl % lpg, warp = wi % wpg;
  const int sub = wi / wpg * nsl + wl / lpg, nsub = nsw * nsl;
  const int dz = (int)blockIdx.x - 1, chunk = blockIdx.y;
  const int nib = (ci + 31) / 32, i0 = blockIdx.z % nib * 32, o0 = blockIdx.z / nib * 32;
  const int nci = min(32, ci - i0), nco = min(32, co - o0);
  const bool with_bias = dz == 0 && i0 == 0;
  f32x2 acc[4][9];                              // pairs of output channels
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int q = 0; q < 9; ++q) acc[k][q] = 0ull;
  float accb = 0.0f;                            // bias: thread t sums every 8th voxel of channel t / 8
  // my units (b, z) with plane z + dz inside the patch
  const long long units = (long long)B * S, un0 = units * chunk / nk, un1 = units * (chunk + 1) / nk;
  auto next = [&](long long un) {
    while (un < un1 && ((int)(un % S) + dz < 0 || (int)(un % S) + dz >= S)) ++un;
    return un;
  };
  // a warp copies whole channels (the place of a value in its row by counting,
  // not by dividing)
  auto fetch = [&](long long un, float* xs) {
    if (un < un1) {
      const int b = (int)(un / S), z = (int)(un % S);
      float* gs = xs + lpg * CP;
      for (int c = wi; c < lpg; c += 8) {
        const float* src = x + ((long long)b * ci + i0 + min(c, nci - 1)) * S3 + S * S * (z + dz);
        int px = wl, py = 0;
        while (px >= P) { px -= P; ++py; }
        for (int e = wl; e < (S + 2) * P; e += 32) {
          const bool in = c < nci && px >= 1 && px <= S && py >= 1 && py <= S;
          copy4(xs + c * CP + e, src + (in ? px - 1 + S * (py - 1) : 0), in);
          px += 32;
          while (px >= P) { px -= P; ++py; }
        }
      }
      for (int c = wi; c < wpg * 8; c += 8) {
        const float* src = gy + ((long long)b * co + o0 + min(c, nco - 1)) * S3 + S * S * z;
        int px = wl, py = 0;
        while (px >= Q) { px -= Q; ++py; }
        for (int e = wl; e < S * Q; e += 32) {
          const bool in = c < nco && px < S;
          copy4(gs + (c / 2 * S * Q + e) * 2 + c % 2, src + (in ? px + S * py : 0), in);
          px += 32;
          while (px >= Q) { px -= Q; ++py; }
        }
      }
    }
    copies_commit();
  };
  long long un = next(un0);
  fetch(un, sm);
  for (int buf = 0; un < un1; buf ^= 1) {
    const float* xs = sm + buf * stage;
    const float* gs = xs + lpg * CP;
    const long long nu = next(un + 1);
    fetch(nu, sm + (buf ^ 1) * stage);
    un = nu;
    copies_wait<1>();
    __syncthreads();
    const float* gw_ = gs + warp * 8 * S * Q;
    const float* xl = xs + lane * CP;
    if (with_bias) {
      const int c = threadIdx.x >> 3;
      if (c < wpg * 8)
        for (int e = threadIdx.x & 7; e < S * Q; e += 8) accb += gs[(c / 2 * S * Q + e) * 2 + c % 2];
    }
    for (int yv = sub; yv < S; yv += nsub)
      for (int sx = 0; sx < NS; ++sx) {
        f32x2 xv[3][6];
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
          const float* xr = xl + (yv + dy) * P + sx * kStrip;
          const float4 a = *reinterpret_cast<const float4*>(xr);
          const float2 a2 = *reinterpret_cast<const float2*>(xr + 4);
          xv[dy][0] = pack2(a.x, a.x); xv[dy][1] = pack2(a.y, a.y); xv[dy][2] = pack2(a.z, a.z);
          xv[dy][3] = pack2(a.w, a.w); xv[dy][4] = pack2(a2.x, a2.x); xv[dy][5] = pack2(a2.y, a2.y);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float* gr = gw_ + ((k * S + yv) * Q + sx * kStrip) * 2;
          const ulonglong2 g0 = *reinterpret_cast<const ulonglong2*>(gr);
          const ulonglong2 g1 = *reinterpret_cast<const ulonglong2*>(gr + 4);
          const f32x2 gv[kStrip] = {g0.x, g0.y, g1.x, g1.y};
#pragma unroll
          for (int dy = 0; dy < 3; ++dy)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
              for (int u = 0; u < kStrip; ++u)
                acc[k][dy * 3 + dx] = fma2(gv[u], xv[dy][u + dx], acc[k][dy * 3 + dx]);
        }
      }
    __syncthreads();                            // the buffer is free for the copies after next
  }
  copies_wait<0>();
  float sum[8][9];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const float2 v = unpack2(acc[k][q]);
      sum[2 * k][q] = v.x;
      sum[2 * k + 1][q] = v.y;
    }
  // the groups that shared the channels' rows, into the first one in order
  const int mine = (warp * lpg + lane) * 73;
  for (int g = 1; g < nsub; ++g) {
    __syncthreads();
    if (sub == g)
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int q = 0; q < 9; ++q) sm[mine + k * 9 + q] = sum[k][q];
    __syncthreads();
    if (sub == 0)
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int q = 0; q < 9; ++q) sum[k][q] += sm[mine + k * 9 + q];
  }
  if (with_bias) {
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) accb += __shfl_down_sync(0xffffffffu, accb, off, 8);
    const int c = threadIdx.x >> 3;
    if ((threadIdx.x & 7) == 0 && c < nco) part_b[(long long)chunk * co + o0 + c] = accb;
  }
  if (sub > 0) return;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int o = o0 + warp * 8 + k;
    if (o >= co || lane >= nci) continue;
    float* p = part + (((long long)chunk * co + o) * ci + i0 + lane) * 27 + (dz + 1) * 9;
#pragma unroll
    for (int q = 0; q < 9; ++q) p[q] = sum[k][q];
  }
}

// Sums the chunks in order, the 27 taps of kSumPairs channel pairs a CTA, then
// the biases'.  Sums that are not finite are formed again from the pairs of voxels
// inside the patch with g != 0 alone (the tile kernel also multiplies non-finite
// inputs by zero padding and zero gradients): by the whole CTA, a pair's taps
// together, as in k_conv_bwd_w.  (32 x 32 channels, 64 patches of
// 11^3: 1070 us with one infinite input, 380 with all NaN; 13800 and 16000 with a
// thread a sum, 1750 with the general kernels.)
constexpr int kSumPairs = 4, kSumThreads = 128;
__global__ void __launch_bounds__(kSumThreads) k_conv_bwd_w_sum(int B, int S, int ci, int co, int nk,
                                                                const float* __restrict__ part,
                                                                const float* __restrict__ part_b,
                                                                const float* __restrict__ x,
                                                                const float* __restrict__ gy,
                                                                float* __restrict__ gw,
                                                                float* __restrict__ gbias) {
  __shared__ unsigned bad[kSumPairs];                     // a pair's taps to be formed again
  __shared__ float red[27][kSumThreads / 32];
  __shared__ unsigned over;
  const int pairs = co * ci, n = pairs * 27, S3 = S * S * S, tid = threadIdx.x;
  const int wblocks = (pairs + kSumPairs - 1) / kSumPairs;
  const bool is_b = (int)blockIdx.x >= wblocks;
  const int e = is_b ? ((int)blockIdx.x - wblocks) * kSumThreads + tid : (int)blockIdx.x * kSumPairs * 27 + tid;
  const bool on = is_b ? e < co : tid < kSumPairs * 27 && e < n;
  if (tid < kSumPairs) bad[tid] = 0u;
  __syncthreads();
  if (on) {
    const float* p = (is_b ? part_b : part) + e;
    const long long st = is_b ? co : n;
    float a[8] = {};                                       // eight sums in flight, a fixed order
    int k = 0;
    for (; k + 8 <= nk; k += 8)
#pragma unroll
      for (int q = 0; q < 8; ++q) a[q] += p[(long long)(k + q) * st];
    for (; k < nk; ++k) a[0] += p[(long long)k * st];
    const float s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    if (is_b) gbias[e] = s;
    else if (isfinite(s)) gw[e] = s;
    else atomicOr(bad + tid / 27, 1u << tid % 27);
  }
  __syncthreads();
  if (is_b) return;
  for (int q = 0; q < kSumPairs; ++q) {
    const unsigned taps = bad[q];                          // (the same in every thread)
    if (taps == 0u) continue;
    if (tid == 0) over = 0u;
    __syncthreads();
    const int pair = (int)blockIdx.x * kSumPairs + q, o = pair / ci, i = pair - o * ci;
    float acc[27];
#pragma unroll
    for (int t = 0; t < 27; ++t) acc[t] = 0.0f;
    for (int b = 0; b < B; ++b) {
      const float* xc = x + ((long long)b * ci + i) * S3;
      const float* gc = gy + ((long long)b * co + o) * S3;
      for (int v = tid; v < S3; v += kSumThreads) {
        const float g = gc[v];
        if (g == 0.0f) continue;
        const int vx = v % S, vy = (v / S) % S, vz = v / (S * S);
#pragma unroll
        for (int t = 0; t < 27; ++t) {
          const int ux = vx + t % 3 - 1, uy = vy + (t / 3) % 3 - 1, uz = vz + t / 9 - 1;
          if (ux < 0 || ux >= S || uy < 0 || uy >= S || uz < 0 || uz >= S) continue;
          acc[t] += g * xc[ux + S * (uy + S * uz)];
        }
      }
      if ((b & (b + 1)) == 0) {                            // sums that are NaN already are over
        unsigned nan = 0u;
#pragma unroll
        for (int t = 0; t < 27; ++t) nan |= isnan(acc[t]) ? 1u << t : 0u;
        nan = __reduce_or_sync(0xffffffffu, nan);
        if (tid % 32 == 0) atomicOr(&over, nan);
        __syncthreads();
        const unsigned o_all = over;
        __syncthreads();                                   // (read by all before the next addition)
        if ((o_all & taps) == taps) break;
      }
    }
#pragma unroll
    for (int t = 0; t < 27; ++t) {
      float s = acc[t];
      for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
      if (tid % 32 == 0) red[t][tid / 32] = s;
    }
    __syncthreads();
    if (tid < 27 && (taps >> tid & 1u)) {
      float s = 0.0f;
      for (int k = 0; k < kSumThreads / 32; ++k) s += red[tid][k];
      gw[(long long)pair * 27 + tid] = s;
    }
    __syncthreads();
  }
}

// Masked mean-squared error: loss = sum_mask (p - t)^2 / count,
// grad = 2 (p - t) mask / count.  Per-block partial sums, then one block.
__global__ void k_mse_partial(long long n, const float* __restrict__ p, const float* __restrict__ t,
                              const float* __restrict__ mask, float inv_count, float* grad,
                              double* part) {
  __shared__ double red[32];
  double s = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const float mk = mask[e];
    const float d = (p[e] - t[e]) * mk;
    grad[e] = 2.0f * d * inv_count;
    s += (double)d * (double)d;
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tsum = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) tsum += red[k];
    part[blockIdx.x] = tsum;
  }
}

// One warp: lane l sums partials l, l + 32, ... in order, then the lanes in a
// tree (a single thread's 512 dependent FP64 additions took 30 us; 4 us now).
__global__ void k_mse_final(int nb, const double* __restrict__ part, double inv_count, double* out) {
  double s = 0.0;
  for (int k = threadIdx.x; k < nb; k += 32) s += part[k];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (threadIdx.x == 0) out[0] = s * inv_count;
}

// Energy norm of the interior error (the norm the coarse space pays in):
// e = mask (p - t), relative face couplings w = exp(x[b][d][u]) for the face
// between u and its lower neighbour along d (x: the network input, whose
// channels 0-2 are the log couplings), E = sum_faces w (e_u - e_v)^2 / count,
// grad = mask dE/dp.  One thread per (patch, channel, cell), grid-stride.
__device__ __forceinline__ float e_at(const float* p, const float* t, const float* mk, long long o) {
  return (p[o] - t[o]) * mk[o];
}

__global__ void k_energy_partial(int B, int S, int C, int cx, const float* __restrict__ p,
                                 const float* __restrict__ t, const float* __restrict__ mk,
                                 const float* __restrict__ x, float inv_count, float* grad,
                                 double* part) {
  __shared__ double red[32];
  const int S3 = S * S * S;
  const long long n = (long long)B * C * S3;
  double acc = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(e % S3);
    const long long bc = e / S3;
    const int b = (int)(bc / C);
    const int l[3] = {v % S, (v / S) % S, v / (S * S)};
    const int st[3] = {1, S, S * S};
    const float ev = e_at(p, t, mk, e);
    float gsum = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float* xd = x + ((long long)b * cx + d) * S3;
      if (l[d] > 0) {                          // face to the lower neighbour
        const float w = expf(xd[v]);
        const float diff = ev - e_at(p, t, mk, e - st[d]);
        acc += (double)(w * diff * diff);
        gsum += w * diff;
      }
      if (l[d] < S - 1) {                      // face to the upper neighbour
        const float w = expf(xd[v + st[d]]);
        gsum += w * (ev - e_at(p, t, mk, e + st[d]));
      }
    }
    grad[e] = 2.0f * gsum * mk[e] * inv_count;
  }
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tsum = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) tsum += red[k];
    part[blockIdx.x] = tsum;
  }
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// p -= lr * (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).
__global__ void k_adam(long long n, float* p, const float* __restrict__ g, float* m, float* v,
                       float lr, float b1, float b2, float eps, float c1, float c2) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const float ge = g[e];
  const float me = b1 * m[e] + (1.0f - b1) * ge;
  const float ve = b2 * v[e] + (1.0f - b2) * ge * ge;
  m[e] = me;
  v[e] = ve;
  p[e] -= lr * (me / c1) / (sqrtf(ve / c2) + eps);
}

constexpr int kMseBlocks = 512;

}  // namespace

// Workspace of the weight gradient's partial sums: stream-ordered allocations
// of at most kNetWork bytes from a pool of the library's own, one for a device's
// context, which keeps that much between calls (the device's default pool gives
// everything back at every synchronisation: 250 us a call in place of 95 when
// each is waited for).  Stream order makes it safe for any streams and threads.
// What is unused goes back with every handle that is destroyed, the pool itself
// with its context: a pool is never used in another one.
namespace {
constexpr unsigned long long kNetWork = 64ull << 20;

std::mutex net_pools_mutex;
std::map<unsigned long long, cudaMemPool_t> net_pools;   // by context_id()

cudaError_t net_pool(cudaMemPool_t* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long ctx = context_id();
  if (ctx == 0) return cudaErrorNotSupported;
  std::lock_guard<std::mutex> lock(net_pools_mutex);
  auto it = net_pools.find(ctx);
  if (it == net_pools.end()) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    e = cudaMemPoolCreate(&p, &props);
    if (e != cudaSuccess) return e;
    unsigned long long keep = kNetWork;
    e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return e;
    }
    it = net_pools.emplace(ctx, p).first;
  }
  *out = it->second;
  return cudaSuccess;
}
}  // namespace

void release_net_workspace() {
  const unsigned long long ctx = context_id();
  std::lock_guard<std::mutex> lock(net_pools_mutex);
  const auto it = net_pools.find(ctx);
  if (it != net_pools.end()) cudaMemPoolTrimTo(it->second, 0);
}

namespace {
constexpr int kSms = 152;               // SMs of the GPU
constexpr int kTileSmem = 100 * 1024;   // more leaves one CTA per SM: the general kernels then
constexpr int kFewCi = 260;             // summed channels whose weights fit a general kernel's CTA
}  // namespace

// Warps that the general kernels would run for `c` result channels.  Where they
// are few, one CTA's latency is the time whatever the batch, and the general
// kernels' is the shorter (8 channels a CTA instead of 32).
static long long general_warps(int B, int S, int c) {
  return (long long)B * ((c + kCoB - 1) / kCoB) * (((long long)S * S * S + 31) / 32);
}

// The tiled kernel where a CTA's planes fit its staging (with the strips per CTA
// that the batch's size gives it: most patches up to 12^3, few above), else the
// general one.  64 patches of 11^3: 32 -> 32 channels 390 -> 176 us, 32 -> 8
// channels 132 -> 79.  With 8 results a thread the general kernel is the faster
// one up to 1024 warps of its own (32 -> 32, 64 patches of 4^3: 72 against 78 us; 64 of
// 6^3, beyond the line: 91 against 74); so it is for patches of one voxel.
cudaError_t launch_conv_fwd(int B, int S, int ci, int co, const float* x, const float* w,
                            const float* bias, int relu, float* y, cudaStream_t s) {
  const int S3 = S * S * S;
  const ConvTile t = conv_tile(B, S, co, kSms);
  const int smem = kCoB * ci * 27 * (int)sizeof(float);
  const bool few = S == 1 || (t.ko == 8 && general_warps(B, S, co) <= 1024);
  if (t.smem <= kTileSmem && !(few && ci <= kFewCi)) {
    cudaError_t e = t.ko == 8 ? raise_smem_limit(k_conv_tile<false, 8>, t.smem)
                                : raise_smem_limit(k_conv_tile<false, 4>, t.smem);
    if (e != cudaSuccess) return e;
    dim3 grid((S * t.NYP * t.NS + t.ST - 1) / t.ST, (co + 31) / 32, B);
    if (t.ko == 8) k_conv_tile<false, 8><<<grid, t.ST * t.ncg, t.smem, s>>>(S, ci, co, t, x, w, bias, relu, nullptr, y);
    else k_conv_tile<false, 4><<<grid, t.ST * t.ncg, t.smem, s>>>(S, ci, co, t, x, w, bias, relu, nullptr, y);
    count_launches(1);
    return cudaGetLastError();
  }
  cudaError_t e = raise_smem_limit(k_conv_fwd, smem);
  if (e != cudaSuccess) return e;
  dim3 grid((S3 + kNetThreads * kVox - 1) / (kNetThreads * kVox), (co + kCoB - 1) / kCoB, B);
  k_conv_fwd<<<grid, kNetThreads, smem, s>>>(S, ci, co, x, w, bias, relu, y);
  count_launches(1);
  return cudaGetLastError();
}

// Data gradient as the forward convolution; weight gradient in chunks of
// planes (two CTAs an SM for the three dz), then one pass over the chunks.
// The general weight kernel stays for patches whose planes do not fit and for
// a stream that is being captured (a graph would have to own the workspace).
// 64 patches of 11^3, 32 x 32 channels: data 440 -> 174 us, weights 1400 -> 180.
// Small calls stay with the general kernels here too: the data gradient up to 2048
// of their warps where 16 channels or fewer are summed (8 channels, 64 patches of
// 4^3: 31 against 37 us; of 8^3, beyond the line: 53 against 37), and the weights where a CTA
// per pair of channels has few passes of 256 voxels to make (4 patches of 11^3,
// 32 x 8 channels: 33 against 21 us; 1 patch: 13 against 19).
cudaError_t launch_conv_bwd(int B, int S, int ci, int co, const float* x, const float* w,
                            const float* gy, const float* xact, float* gx, float* gw,
                            float* gbias, cudaStream_t s) {
  const int S3 = S * S * S;
  cudaError_t e;
  if (gx) {
    const ConvTile t = conv_tile(B, S, ci, kSms);
    const bool few = S == 1 || (t.ko == 8 && co <= 16 && general_warps(B, S, ci) <= 2048);
    if (t.smem <= kTileSmem && !(few && co <= kFewCi)) {
      e = t.ko == 8 ? raise_smem_limit(k_conv_tile<true, 8>, t.smem)
                                : raise_smem_limit(k_conv_tile<true, 4>, t.smem);
      if (e != cudaSuccess) return e;
      dim3 grid((S * t.NYP * t.NS + t.ST - 1) / t.ST, (ci + 31) / 32, B);
      if (t.ko == 8) k_conv_tile<true, 8><<<grid, t.ST * t.ncg, t.smem, s>>>(S, co, ci, t, gy, w, nullptr, 0, xact, gx);
      else k_conv_tile<true, 4><<<grid, t.ST * t.ncg, t.smem, s>>>(S, co, ci, t, gy, w, nullptr, 0, xact, gx);
    } else {
      const int smem = kCoB * co * 27 * (int)sizeof(float);
      e = raise_smem_limit(k_conv_bwd_data, smem);
      if (e != cudaSuccess) return e;
      dim3 grid((S3 + kNetThreads - 1) / kNetThreads, (ci + kCoB - 1) / kCoB, B);
      k_conv_bwd_data<<<grid, kNetThreads, smem, s>>>(S, ci, co, gy, w, xact, gx);
    }
    count_launches(1);
  }
  const int NS = (S + kStrip - 1) / kStrip, P = kStrip * NS + 4;
  const int CP = ((S + 2) * P + 27) / 32 * 32 + 4;       // 4 modulo the 32 banks
  const int nsl = ci <= 16 ? 2 : 1, nsw = co <= 8 ? 8 : co <= 16 ? 4 : 2;
  long long smem = 2 * ((32LL / nsl) * CP + (64LL / nsw) * S * kStrip * NS) * 4;
  const long long add_up = (8LL / nsw) * (32 / nsl) * 73 * 4;
  if (smem < add_up) smem = add_up;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
    cudaGetLastError();
    cap = cudaStreamCaptureStatusActive;
  }
  const long long passes = (long long)B * (((long long)S * S * S + 255) / 256);
  const bool few = passes * (1024 + (long long)ci * co) < 20 * 1024;
  if (smem <= kTileSmem && cap == cudaStreamCaptureStatusNone && !few) {
    // chunks: of one plane at least, and as many as the workspace holds (with many
    // channels the tiles fill the chip, whatever the chunks)
    const long long units = (long long)B * S, per = (long long)co * ci * 27 + co;
    const long long room = (long long)(kNetWork / sizeof(float)) / per;
    const int nk = (int)std::min({units, room, 101LL});
    const size_t n = (size_t)nk * (size_t)per;
    cudaMemPool_t pool = nullptr;
    float* part = nullptr;
    e = nk > 0 ? net_pool(&pool) : cudaErrorMemoryAllocation;
    if (e == cudaSuccess)
      e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&part), n * sizeof(float), pool, s);
    if (e == cudaSuccess) {
      float* part_b = part + (size_t)nk * co * ci * 27;
      e = raise_smem_limit(k_conv_bwd_w_tile, (int)smem);
      if (e == cudaSuccess) {
        dim3 grid(3, nk, ((ci + 31) / 32) * ((co + 31) / 32));
        k_conv_bwd_w_tile<<<grid, kNetThreads, (int)smem, s>>>(B, S, ci, co, NS, P, CP, nk, nsl, nsw, x, gy,
                                                               part, part_b);
        k_conv_bwd_w_sum<<<(co * ci + kSumPairs - 1) / kSumPairs + (co + kSumThreads - 1) / kSumThreads,
                           kSumThreads, 0, s>>>(B, S, ci, co, nk, part, part_b, x, gy, gw, gbias);
        count_launches(2);
        e = cudaGetLastError();
      }
      const cudaError_t f = cudaFreeAsync(part, s);
      return e != cudaSuccess ? e : f;
    }
    cudaGetLastError();                                  // no workspace: the general kernel
  }
  k_conv_bwd_w<<<dim3(ci, co), kNetThreads, 0, s>>>(B, S, ci, co, x, gy, gw, gbias);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_mse(long long n, const float* p, const float* t, const float* mask,
                       double count, float* grad, double* part, double* loss, cudaStream_t s) {
  k_mse_partial<<<kMseBlocks, 256, 0, s>>>(n, p, t, mask, (float)(1.0 / count), grad, part);
  k_mse_final<<<1, 32, 0, s>>>(kMseBlocks, part, 1.0 / count, loss);
  count_launches(2);
  return cudaGetLastError();
}

cudaError_t launch_energy(int B, int S, int C, int cx, const float* p, const float* t,
                          const float* mask, const float* x, double count, float* grad, double* part,
                          double* loss, cudaStream_t s) {
  k_energy_partial<<<kMseBlocks, 256, 0, s>>>(B, S, C, cx, p, t, mask, x, (float)(1.0 / count), grad,
                                              part);
  k_mse_final<<<1, 32, 0, s>>>(kMseBlocks, part, 1.0 / count, loss);
  count_launches(2);
  return cudaGetLastError();
}

cudaError_t launch_adam(long long n, float* p, const float* g, float* m, float* v, float lr,
                        float b1, float b2, float eps, int step, cudaStream_t s) {
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  k_adam<<<(int)((n + 255) / 256), 256, 0, s>>>(n, p, g, m, v, lr, b1, b2, eps, c1, c2);
  count_launches(1);
  return cudaGetLastError();
}

int mse_partial_blocks() { return kMseBlocks; }

// ---------------------------------------------------------------------
// The surrogate's patches.  A full interior dual block is the box of
// (b+1)^3 cells from one vertex plane to the next in every direction
// (S = b+1); its 8 basis functions are those of its corner nodes, corner
// bits (cx, cy, cz).  At local coordinate l (0..b) along d the value of the
// function with corner bit c_d sits in the cell's P slot with bit d = c_d
// between the planes; on the plane l = 0 only c_d = 0 has support (slot bit
// 0), on l = b only c_d = 1 (slot bit 0).  The baseline is the multilinear
// interpolant of the corner values, the exact discrete basis function of a
// homogeneous medium; the network predicts the deviation from it.
namespace {

template <class TP>
__device__ __forceinline__ float patch_value(const Geo& g, const TP* P, long long i, const int* l, int b,
                                             int corner) {
  int slot = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int cd = (corner >> d) & 1;
    if (l[d] == 0) { if (cd) return 0.0f; }
    else if (l[d] == b) { if (!cd) return 0.0f; }
    else if (cd) slot |= 1 << d;
  }
  return (float)P[(long long)slot * g.N + i];
}

__device__ __forceinline__ float baseline(const int* l, int b, int corner) {
  float v = 1.0f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float t = (float)l[d] / (float)b;
    v *= ((corner >> d) & 1) ? t : 1.0f - t;
  }
  return v;
}

// One CTA per patch: x [12][S^3] (log couplings minus their patch mean, the
// relative accumulation term, the boundary deviations of the 8 functions),
// optionally target/mask [8][S^3] (deviation everywhere, mask 1 inside).
template <class TP>
__global__ void __launch_bounds__(256) k_patch_inputs(Geo g, int b, const int* __restrict__ org,
                                                      const TP* __restrict__ P,
                                                      const double* __restrict__ Abd,
                                                      const double* __restrict__ Abx,
                                                      const double* __restrict__ Aby,
                                                      const double* __restrict__ Abz, float* x,
                                                      float* target, float* mask) {
  __shared__ float red[32];
  __shared__ float s_mean;
  const int S = b + 1, S3 = S * S * S;
  const int pidx = blockIdx.x;
  const int ox = org[3 * pidx], oy = org[3 * pidx + 1], oz = org[3 * pidx + 2];
  float* xp = x + (long long)pidx * kNetIn * S3;
  // mean of the log couplings over the patch
  float s = 0.0f;
  for (int v = threadIdx.x; v < S3; v += blockDim.x) {
    const int l[3] = {v % S, (v / S) % S, v / (S * S)};
    const long long i = (ox + l[0]) + g.sy * (oy + l[1]) + g.sz * (oz + l[2]);
    s += logf(fmaxf((float)-Abx[i], 1e-30f)) + logf(fmaxf((float)-Aby[i], 1e-30f)) +
         logf(fmaxf((float)-Abz[i], 1e-30f));
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    s_mean = t / (3.0f * (float)S3);
  }
  __syncthreads();
  const float mean = s_mean;
  for (int v = threadIdx.x; v < S3; v += blockDim.x) {
    const int l[3] = {v % S, (v / S) % S, v / (S * S)};
    const long long i = (ox + l[0]) + g.sy * (oy + l[1]) + g.sz * (oz + l[2]);
    const float wx = (float)-Abx[i], wy = (float)-Aby[i], wz = (float)-Abz[i];
    xp[0 * S3 + v] = logf(fmaxf(wx, 1e-30f)) - mean;
    xp[1 * S3 + v] = logf(fmaxf(wy, 1e-30f)) - mean;
    xp[2 * S3 + v] = logf(fmaxf(wz, 1e-30f)) - mean;
    const double wsum = -(Abx[i] + Aby[i] + Abz[i] + Abx[i + 1] + Aby[i + g.sy] + Abz[i + g.sz]);
    xp[3 * S3 + v] = wsum > 0.0 ? (float)((Abd[i] - wsum) / wsum) : 0.0f;
    const bool inside = l[0] > 0 && l[0] < b && l[1] > 0 && l[1] < b && l[2] > 0 && l[2] < b;
    for (int c = 0; c < 8; ++c) {
      const float dev = patch_value(g, P, i, l, b, c) - baseline(l, b, c);
      xp[(4 + c) * S3 + v] = inside ? 0.0f : dev;
      if (target) {
        target[((long long)pidx * 8 + c) * S3 + v] = dev;
        mask[((long long)pidx * 8 + c) * S3 + v] = inside ? 1.0f : 0.0f;
      }
    }
  }
}

// P at the patches' interior cells = baseline + the network's deviation.
template <class TP>
__global__ void __launch_bounds__(256) k_patch_apply(Geo g, int b, const int* __restrict__ org,
                                                     const float* __restrict__ y, TP* P) {
  const int S = b + 1, S3 = S * S * S;
  const int pidx = blockIdx.x;
  const int ox = org[3 * pidx], oy = org[3 * pidx + 1], oz = org[3 * pidx + 2];
  for (int v = threadIdx.x; v < S3; v += blockDim.x) {
    const int l[3] = {v % S, (v / S) % S, v / (S * S)};
    if (!(l[0] > 0 && l[0] < b && l[1] > 0 && l[1] < b && l[2] > 0 && l[2] < b)) continue;
    const long long i = (ox + l[0]) + g.sy * (oy + l[1]) + g.sz * (oz + l[2]);
    for (int c = 0; c < 8; ++c)
      P[(long long)c * g.N + i] = (TP)(baseline(l, b, c) + y[((long long)pidx * 8 + c) * S3 + v]);
  }
}

// Residual gate: for each function, ||D^{-1} A_b P|| over the interior
// cells against ||D^{-1} (the part of A_b P from the boundary values)||,
// D = diag(A_b) (the Jacobi scaling keeps high-permeability cells from
// dominating both norms); the patch's flag (1 = solve exactly) is set when
// the largest ratio over its 8 functions exceeds tol.
template <class TP>
__global__ void __launch_bounds__(256) k_patch_gate(Geo g, int b, const int* __restrict__ org,
                                                    const int* __restrict__ ent, const TP* __restrict__ P,
                                                    const double* __restrict__ Abd,
                                                    const double* __restrict__ Abx,
                                                    const double* __restrict__ Aby,
                                                    const double* __restrict__ Abz, double tol,
                                                    unsigned char* flag, float* ratio_out) {
  __shared__ float red[2][8][8];
  const int S = b + 1, S3 = S * S * S;
  const int pidx = blockIdx.x;
  const int ox = org[3 * pidx], oy = org[3 * pidx + 1], oz = org[3 * pidx + 2];
  float rr[8], bb[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) { rr[c] = 0.0f; bb[c] = 0.0f; }
  for (int v = threadIdx.x; v < S3; v += blockDim.x) {
    const int l[3] = {v % S, (v / S) % S, v / (S * S)};
    if (!(l[0] > 0 && l[0] < b && l[1] > 0 && l[1] < b && l[2] > 0 && l[2] < b)) continue;
    const long long i = (ox + l[0]) + g.sy * (oy + l[1]) + g.sz * (oz + l[2]);
    const double cpl[6] = {Abx[i], Abx[i + 1], Aby[i], Aby[i + g.sy], Abz[i], Abz[i + g.sz]};
    const long long nbi[6] = {i - 1, i + 1, i - g.sy, i + g.sy, i - g.sz, i + g.sz};
    const double dinv = 1.0 / Abd[i];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      double r = Abd[i] * (double)patch_value(g, P, i, l, b, c), f = 0.0;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        int ln[3] = {l[0], l[1], l[2]};
        ln[k >> 1] += (k & 1) ? 1 : -1;
        const double t = cpl[k] * (double)patch_value(g, P, nbi[k], ln, b, c);
        r += t;
        const bool nb_inside = ln[0] > 0 && ln[0] < b && ln[1] > 0 && ln[1] < b && ln[2] > 0 && ln[2] < b;
        if (!nb_inside) f += t;
      }
      r *= dinv;
      f *= dinv;
      rr[c] += (float)(r * r);
      bb[c] += (float)(f * f);
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float a = rr[c], q = bb[c];
    for (int off = 16; off > 0; off >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, off);
      q += __shfl_down_sync(0xffffffffu, q, off);
    }
    if (lane == 0) { red[0][c][wid] = a; red[1][c][wid] = q; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float worst = 0.0f;
    for (int c = 0; c < 8; ++c) {
      float a = 0.0f, q = 0.0f;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) { a += red[0][c][k]; q += red[1][c][k]; }
      const float ratio = q > 0.0f ? sqrtf(a / q) : (a > 0.0f ? INFINITY : 0.0f);
      worst = fmaxf(worst, ratio);
    }
    if (ratio_out) ratio_out[pidx] = worst;
    flag[ent[pidx]] = (worst > (float)tol || !isfinite(worst)) ? 1 : 0;
  }
}

}  // namespace

cudaError_t launch_patch_inputs(const Geo& g, int b, int n, const int* org, bool single,
                                const Buffers& bf, float* x, float* target, float* mask,
                                cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (single)
    k_patch_inputs<float><<<n, 256, 0, s>>>(g, b, org, bf.f32.P, bf.Abd, bf.Abx, bf.Aby, bf.Abz, x,
                                            target, mask);
  else
    k_patch_inputs<double><<<n, 256, 0, s>>>(g, b, org, bf.P, bf.Abd, bf.Abx, bf.Aby, bf.Abz, x,
                                             target, mask);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_patch_apply(const Geo& g, int b, int n, const int* org, const float* y,
                               bool single, Buffers& bf, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (single) k_patch_apply<float><<<n, 256, 0, s>>>(g, b, org, y, bf.f32.P);
  else k_patch_apply<double><<<n, 256, 0, s>>>(g, b, org, y, bf.P);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_patch_gate(const Geo& g, int b, int n, const int* org, const int* ent,
                              double tol, bool single, Buffers& bf, unsigned char* flag,
                              float* ratio, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (single)
    k_patch_gate<float><<<n, 256, 0, s>>>(g, b, org, ent, bf.f32.P, bf.Abd, bf.Abx, bf.Aby, bf.Abz,
                                          tol, flag, ratio);
  else
    k_patch_gate<double><<<n, 256, 0, s>>>(g, b, org, ent, bf.P, bf.Abd, bf.Abx, bf.Aby, bf.Abz, tol,
                                           flag, ratio);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace cams
