// The learned surrogate's 3x3x3 convolutions on the tensor cores: tcgen05
// MMAs with BF16 operands and FP32 accumulation in tensor memory.
//
// Implicit GEMM over a zero-padded patch.  A patch of S^3 voxels with C
// channels is stored "chunked and padded": the (S+2)^3 grid with a zero
// border, voxels in flat order r = px + S'(py + S' pz) (S' = S + 2), channels
// in chunks of 8 (16 bytes): element (r, c) at ((c / 8) * RP + r) * 8 + c % 8,
// RP rows per chunk plane (the padded grid plus spare zero rows).  For an
// output row r the 27 input rows of its stencil are r + off(t),
// off = dx + S' dy + S'^2 dz, so the A operand of one tap for 128 consecutive
// output rows is 128 consecutive input rows: a shared-memory descriptor
// starting off(t) rows further, no im2col copy.  Rows of one 8-channel chunk
// are 16 bytes apart, so any run of 8 rows is one 128-byte core matrix of the
// no-swizzle K-major layout (SBO = 128 bytes between row groups, LBO = RP x 16
// bytes between the two chunks of a K = 16 step).  The weights of a tap, N x
// C in the same layout, are the B operand; D = A B^T (128 x N, FP32) sits in
// 128 lanes x N columns of tensor memory.
//
// Output rows are computed in tiles of 128 from the first interior voxel
// (r = h, h = S'^2 + S' + 1) to the last; border rows inside those tiles and
// the rows outside them are written as zeros, so a layer's output is the next
// layer's zero-padded input.  A CTA keeps all weights in shared memory and runs
// one patch after the other, each in tiles, with a warp for each kind of work:
// one thread copies a patch's input (one bulk copy) once the last patch's MMAs
// are done, one thread issues the 27 x C/16 MMAs of a tile into one of two
// accumulators and commits them to an mbarrier, and four warps (a thread per
// tensor-memory lane) read the other accumulator back (bias, ReLU, BF16 or
// FP32 out).  What bounds a tile is the MMAs' reads of A from shared memory: 54
// of 128 x 16 BF16 values (C = 32), 4 KB each, 81 cycles an MMA at N = 32 and 74
// at N = 16 (the taps cannot be gathered into a wider N without changing the
// order of the sums).  Measured, 1024 patches of 11^3 through the four layers: 2.47 ms
// with one group of threads that copied, issued and read back in turn, 1.81 with
// the roles apart, 0.87 with the descriptors advanced instead of formed.
#include <cuda_bf16.h>

#include "cams_internal.h"
#include "tc_ptx.h"

namespace cams {

namespace {

constexpr int kTcThreads = 192;            // four epilogue warps, the MMA warp, the copy warp
constexpr int kTile = 128;
constexpr long long kTcWait = 1LL << 24;   // polls of the MMA barrier before giving up

struct TcGeom {
  int S, Sp, h, nt, RP;
};

inline TcGeom tc_geom(int S) {
  TcGeom G;
  G.S = S;
  G.Sp = S + 2;
  G.h = G.Sp * G.Sp + G.Sp + 1;
  const int span = G.Sp * G.Sp * G.Sp - 2 * G.h;
  G.nt = (span + kTile - 1) / kTile;
  G.RP = (2 * G.h + G.nt * kTile + 7) / 8 * 8;
  return G;
}

__device__ __forceinline__ bool interior(const TcGeom& G, int r, int& vox) {
  const int n3 = G.Sp * G.Sp * G.Sp;
  if (r >= n3) return false;
  const int px = r % G.Sp, py = (r / G.Sp) % G.Sp, pz = r / (G.Sp * G.Sp);
  if (px < 1 || px > G.S || py < 1 || py > G.S || pz < 1 || pz > G.S) return false;
  vox = (px - 1) + G.S * ((py - 1) + G.S * (pz - 1));
  return true;
}

// FP32 activations [B][C][S^3] -> BF16 chunked-padded [B][KC][RP][8] (KC
// chunks of 8 channels, channels >= C zero; border and spare rows zero).
__global__ void k_tc_pack(int B, TcGeom G, int C, int KC, const float* __restrict__ x,
                          __nv_bfloat16* __restrict__ out) {
  const long long rows = G.RP;
  const long long n = (long long)B * KC * rows;
  const int S3 = G.S * G.S * G.S;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(e % rows);
    const long long bk = e / rows;
    const int kc = (int)(bk % KC);
    const long long b = bk / KC;
    int vox;
    const bool in = interior(G, r, vox);
    __align__(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int c = kc * 8 + k;
      v[k] = __float2bfloat16_rn(in && c < C ? x[(b * C + c) * S3 + vox] : 0.0f);
    }
    *reinterpret_cast<uint4*>(out + ((b * KC + kc) * G.RP + r) * 8) = *reinterpret_cast<uint4*>(v);
  }
}

// One layer: y = conv(x; w) + bias (ReLU when relu).  x: BF16 chunked-padded
// with KCin chunks (2 or 4).  w: FP32 [co][ci][27] (ci <= 8 KCin real
// input channels), bias [co].  N: the MMA's N (co rounded up to 16).
// kOutBf16: y is BF16 chunked-padded with co / 8 chunks (the next layer's
// input); else y is FP32 [B][co][S^3].
template <int N, int KCin, bool kOutBf16>
__global__ void __launch_bounds__(kTcThreads) k_conv_tc(int B, TcGeom G, int ci, int co,
                                                         const __nv_bfloat16* __restrict__ x,
                                                         const float* __restrict__ w,
                                                         const float* __restrict__ bias, int relu,
                                                         void* __restrict__ yv,
                                                         int* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  // [input: KCin x RP x 16 B][weights: 27 x KCin x N x 16 B][mbarriers][tmem slot]
  unsigned char* xs = smem;
  const int xbytes = KCin * G.RP * 16;
  unsigned char* ws = smem + xbytes;
  const int wbytes = 27 * KCin * N * 16;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + xbytes + wbytes);
  uint64_t* full = bar;          // a patch's input has landed
  uint64_t* empty = bar + 1;     // its MMAs are done
  uint64_t* done = bar + 2;      // [2] an accumulator is ready
  uint64_t* taken = bar + 4;     // [2] ... has been read
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar + 6);
  __shared__ float sb[N];
  const int t = threadIdx.x, warp = t >> 5;
  const int S3 = G.S * G.S * G.S;
  // weights into the B layout: tap, chunk kc, row n at ((tap KCin + kc) N + n) 16 B
  for (int e = t; e < wbytes / 16; e += kTcThreads) reinterpret_cast<uint4*>(ws)[e] = uint4{0, 0, 0, 0};
  if (t < N) sb[t] = t < co ? bias[t] : 0.0f;
  if (t == 0) {
    tc::mbar_init(full, 1);
    tc::mbar_init(empty, 1);
    for (int k = 0; k < 2; ++k) {
      tc::mbar_init(done + k, 1);
      tc::mbar_init(taken + k, 128);
    }
  }
  if (warp == 4) tc::tmem_alloc(slot, 64);
  __syncthreads();
#pragma unroll 8
  for (int e = t; e < co * ci * 27; e += kTcThreads) {       // (in memory order)
    const int q = e / 27, tap = e - q * 27, n = q / ci, c = q - n * ci;
    reinterpret_cast<__nv_bfloat16*>(ws)[((tap * KCin + c / 8) * N + n) * 8 + c % 8] = __float2bfloat16_rn(w[e]);
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *slot;
  constexpr uint32_t kIdesc = tc::idesc_bf16_f32(kTile, N);
  bool ok = true;
  if (warp == 5) {
    if ((t & 31) == 0) {
      uint32_t phase = 0, last = 0;
      bool issued = false;
      for (int b = blockIdx.x; b < B && ok; b += gridDim.x, phase ^= 1u) {
        // (a new barrier's preceding phase counts as complete)
        ok = tc::mbar_wait(empty, phase ^ 1u, kTcWait);
        if (ok) {
          tc::mbar_arrive_expect_tx(full, (uint32_t)xbytes);
          tc::bulk_g2s(xs, x + (long long)b * KCin * G.RP * 8, (uint32_t)xbytes, full);
          issued = true;
          last = phase;
        }
      }
      // the CTA does not end with a copy in flight, whoever gave up on it
      if (issued && !tc::mbar_wait(full, last, kTcWait)) ok = false;
    }
  } else if (warp == 4) {
    if ((t & 31) == 0) {
      // An MMA takes fewer cycles than forming two descriptors from scratch would:
      // they are formed once and advanced (their address field counts 16-byte
      // units), the 27 row offsets stay in registers.
      const uint64_t a0 = tc::smem_desc(tc::smem_u32(xs), G.RP * 16, 128);
      const uint64_t b0 = tc::smem_desc(tc::smem_u32(ws), N * 16, 128);
      int off[27];
#pragma unroll
      for (int tap = 0; tap < 27; ++tap)
        off[tap] = G.h + (tap % 3 - 1) + G.Sp * ((tap / 3) % 3 - 1) + G.Sp * G.Sp * (tap / 9 - 1);
      uint32_t phase = 0;
      int it = 0;
      for (int b = blockIdx.x; b < B && ok; b += gridDim.x, phase ^= 1u) {
        ok = tc::mbar_wait(full, phase, kTcWait);
        for (int m = 0; m < G.nt && ok; ++m, ++it) {
          const int q = it & 1;
          ok = tc::mbar_wait(taken + q, (uint32_t)(it >> 1 & 1) ^ 1u, kTcWait);
          if (!ok) break;
          tc::fence_after_sync();
          const uint64_t am = a0 + (uint64_t)(m * kTile);
#pragma unroll
          for (int tap = 0; tap < 27; ++tap)
#pragma unroll
            for (int ks = 0; ks < KCin / 2; ++ks)
              tc::mma_bf16(tmem + q * 32, am + (uint64_t)(off[tap] + 2 * ks * G.RP),
                           b0 + (uint64_t)((tap * KCin + 2 * ks) * N), kIdesc, tap + ks > 0);
          tc::mma_commit(done + q);
          if (m == G.nt - 1) tc::mma_commit(empty);
        }
      }
      // ... nor with MMAs in flight (the read-back may have given up on them)
      if (!ok && it > 0) tc::mbar_wait(done + ((it - 1) & 1), (uint32_t)((it - 1) >> 1 & 1), kTcWait);
    }
  } else {
    int it = 0;
    for (int b = blockIdx.x; b < B && ok; b += gridDim.x) {
      const int KCo = (co + 7) / 8;
      if constexpr (kOutBf16) {
        // the rows outside the tiles
        __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(yv) + (long long)b * KCo * G.RP * 8;
        const int above = G.h + G.nt * kTile, spare = G.RP - G.nt * kTile;
        for (int e = t; e < KCo * spare; e += 128) {
          const int kc = e / spare, k = e - kc * spare, r = k < G.h ? k : above + k - G.h;
          *reinterpret_cast<uint4*>(y + ((long long)kc * G.RP + r) * 8) = uint4{0, 0, 0, 0};
        }
      }
      for (int m = 0; m < G.nt; ++m, ++it) {
        const int q = it & 1;
        if (!tc::mbar_wait(done + q, (uint32_t)(it >> 1 & 1), kTcWait)) {
          ok = false;
          tc::mbar_wait(done + q, (uint32_t)(it >> 1 & 1), kTcWait);   // once more before TMEM is freed
          break;
        }
        tc::fence_after_sync();
        // thread t holds output row row0 + t (tensor-memory lane t)
        const uint32_t tl = tmem + q * 32 + ((uint32_t)(warp * 32) << 16);
        float v[N];
#pragma unroll
        for (int n0 = 0; n0 < N; n0 += 16) tc::tmem_ld16(tl + n0, *reinterpret_cast<float(*)[16]>(v + n0));
        tc::fence_before_sync();
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(taken + q)) : "memory");
        const int r = G.h + m * kTile + t;
        int vox = 0;
        const bool in = interior(G, r, vox);
#pragma unroll
        for (int n = 0; n < N; ++n) {
          float y = n < co ? v[n] + sb[n] : 0.0f;
          if (relu) y = fmaxf(y, 0.0f);
          v[n] = in ? y : 0.0f;
        }
        if constexpr (kOutBf16) {
          __nv_bfloat16* y = reinterpret_cast<__nv_bfloat16*>(yv) + (long long)b * KCo * G.RP * 8;
#pragma unroll
          for (int kc = 0; kc < N / 8; ++kc) {
            if (kc >= KCo) continue;
            __align__(16) __nv_bfloat16 o[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) o[k] = __float2bfloat16_rn(v[kc * 8 + k]);
            *reinterpret_cast<uint4*>(y + ((long long)kc * G.RP + r) * 8) = *reinterpret_cast<uint4*>(o);
          }
        } else {
          float* y = reinterpret_cast<float*>(yv);
          if (in)
#pragma unroll
            for (int n = 0; n < N; ++n)
              if (n < co) y[((long long)b * co + n) * S3 + vox] = v[n];
        }
      }
    }
  }
  if (!ok) atomicOr(status, kStatTimeout);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 4) tc::tmem_dealloc(tmem, 64);
}

int tc_smem_bytes(const TcGeom& G, int KCin, int N) { return KCin * G.RP * 16 + 27 * KCin * N * 16 + 64; }

template <int N, int KCin, bool kOutBf16>
cudaError_t launch_conv_tc_n(int B, const TcGeom& G, int ci, int co, const __nv_bfloat16* x,
                             const float* w, const float* bias, int relu, void* y, int* status,
                             int sms, cudaStream_t s) {
  const int smem = tc_smem_bytes(G, KCin, N);
  cudaError_t e = raise_smem_limit(k_conv_tc<N, KCin, kOutBf16>, smem);
  if (e != cudaSuccess) return e;
  // two CTAs an SM where shared memory allows (the first layer's 12 channels)
  const int ctas = sms * (2 * (smem + 2048) <= 227 * 1024 ? 2 : 1), grid = B < ctas ? B : ctas;
  k_conv_tc<N, KCin, kOutBf16><<<grid, kTcThreads, smem, s>>>(B, G, ci, co, x, w, bias, relu, y, status);
  count_launches(1);
  return cudaGetLastError();
}

template <int N, bool kOutBf16>
cudaError_t launch_conv_tc_k(int B, const TcGeom& G, int KCin, int ci, int co,
                             const __nv_bfloat16* x, const float* w, const float* bias, int relu,
                             void* y, int* status, int sms, cudaStream_t s) {
  return KCin == 2 ? launch_conv_tc_n<N, 2, kOutBf16>(B, G, ci, co, x, w, bias, relu, y, status, sms, s)
                   : launch_conv_tc_n<N, 4, kOutBf16>(B, G, ci, co, x, w, bias, relu, y, status, sms, s);
}

}  // namespace

long long net_tc_act_elems(int B, int S, int C) {
  const TcGeom G = tc_geom(S);
  const int KC = (C + 15) / 16 * 2;
  return (long long)B * KC * G.RP * 8;
}

bool net_tc_fits(int S, int max_smem) {
  const TcGeom G = tc_geom(S);
  return tc_smem_bytes(G, 4, 32) <= max_smem;
}

cudaError_t launch_tc_pack(int B, int S, int C, const float* x, void* out, cudaStream_t s) {
  const TcGeom G = tc_geom(S);
  const int KC = (C + 15) / 16 * 2;
  const long long n = (long long)B * KC * G.RP;
  const int blocks = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  k_tc_pack<<<blocks, 256, 0, s>>>(B, G, C, KC, x, static_cast<__nv_bfloat16*>(out));
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_conv_tc(int B, int S, int ci, int co, const void* xv, const float* w,
                           const float* bias, int relu, bool out_bf16, void* y, int* status,
                           int sms, cudaStream_t s) {
  const TcGeom G = tc_geom(S);
  const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(xv);
  const int KCin = (ci + 15) / 16 * 2;
  if (KCin > 4) return cudaErrorInvalidValue;
  if (co <= 16) {
    return out_bf16 ? launch_conv_tc_k<16, true>(B, G, KCin, ci, co, x, w, bias, relu, y, status, sms, s)
                    : launch_conv_tc_k<16, false>(B, G, KCin, ci, co, x, w, bias, relu, y, status, sms, s);
  }
  if (co <= 32) {
    return out_bf16 ? launch_conv_tc_k<32, true>(B, G, KCin, ci, co, x, w, bias, relu, y, status, sms, s)
                    : launch_conv_tc_k<32, false>(B, G, KCin, ci, co, x, w, bias, relu, y, status, sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace cams
