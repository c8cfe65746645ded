// sparkattn_quant_fp8: per-(batch, head, token block) absmax scale + E4M3
// encode in one pass over memory (paper Sec. 4.3: FP8 E4M3, scaling and
// casting fused in a single kernel).
//
// One CTA owns one token block: it loads the block's bf16 elements into
// registers once (16-byte loads, rows contiguous), reduces |x| to the block
// maximum, then scales, encodes (cvt.rn.satfinite.e4m3x2.f32) and stores from
// the same registers, so HBM sees one read of x and one write of the codes:
// 3 bytes per element.
#include <cuda_fp8.h>

#include "common.cuh"
#include "launch.h"
#include "tmap.h"

namespace sparkattn {

constexpr int kQuantThreads = 256;

__device__ __forceinline__ float absmax8(uint4 v) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
  float amax = 0.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 f = __bfloat1622float2(p[j]);
    amax = fmaxf(amax, fmaxf(fabsf(f.x), fabsf(f.y)));
  }
  return amax;
}

// eight elements times `inv` as E4M3
__device__ __forceinline__ uint2 encode8(uint4 v, float inv) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
  uint32_t w[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float2 f0 = __bfloat1622float2(p[2 * j]);
    const float2 f1 = __bfloat1622float2(p[2 * j + 1]);
    const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(__fmul_rn(f0.x, inv), __fmul_rn(f0.y, inv)),
                                                  __NV_SATFINITE, __NV_E4M3);
    const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(__fmul_rn(f1.x, inv), __fmul_rn(f1.y, inv)),
                                                  __NV_SATFINITE, __NV_E4M3);
    w[j] = lo | (hi << 16);
  }
  return make_uint2(w[0], w[1]);
}

// the CTA's largest |x| (at least 1e-12) from every thread's; s_red: a float per warp
__device__ __forceinline__ float block_absmax(float amax, float* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = amax;
  __syncthreads();
  amax = s_red[0];
#pragma unroll
  for (int w = 1; w < kQuantThreads / 32; ++w) amax = fmaxf(amax, s_red[w]);
  return fmaxf(amax, 1e-12f);
}

template <int D, int BLK>
__global__ void __launch_bounds__(kQuantThreads, 3)
quant_fp8_kernel(const __nv_bfloat16* x, uint8_t* __restrict__ codes, float* __restrict__ scales,
                 int H, int N, int nb, int64_t stride_b, int64_t stride_h, int64_t stride_n) {
  constexpr int kChunksPerRow = D / 8;                      // 16-byte chunks per token row
  constexpr int kChunks = BLK * kChunksPerRow;              // chunks per token block
  constexpr int kPerThread = kChunks / kQuantThreads;       // 8 for (128,128), 2 for (64,64)
  static_assert(kChunks % kQuantThreads == 0, "block must split evenly over the CTA");

  const int blk = blockIdx.x % nb;
  const int bh = blockIdx.x / nb;
  const int h = bh % H, b = bh / H;
  const int row0 = blk * BLK;
  const int nvalid = min(BLK, N - row0);
  const int64_t base = b * stride_b + h * stride_h;

  pdl_wait();
  uint4 v[kPerThread];
  float amax = 0.0f;
#pragma unroll
  for (int i = 0; i < kPerThread; ++i) {
    const int ci = threadIdx.x + i * kQuantThreads;
    const int r = ci / kChunksPerRow, cc = ci % kChunksPerRow;
    if (r < nvalid) {
      v[i] = *reinterpret_cast<const uint4*>(x + base + (int64_t)(row0 + r) * stride_n + cc * 8);
    } else {
      v[i] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
#pragma unroll
  for (int i = 0; i < kPerThread; ++i) amax = fmaxf(amax, absmax8(v[i]));
  __shared__ float s_red[kQuantThreads / 32];
  amax = block_absmax(amax, s_red);
  const float inv = __fdiv_rn(448.0f, amax);
  if (threadIdx.x == 0) scales[(int64_t)bh * nb + blk] = __fdiv_rn(amax, 448.0f);

#pragma unroll
  for (int i = 0; i < kPerThread; ++i) {
    const int ci = threadIdx.x + i * kQuantThreads;
    const int r = ci / kChunksPerRow, cc = ci % kChunksPerRow;
    if (r < nvalid) *reinterpret_cast<uint2*>(codes + base + (int64_t)(row0 + r) * stride_n + cc * 8) = encode8(v[i], inv);
  }
}

// The same pass with the block's pooled mean for the selection in it (Sec. 4.3 fuses scaling and casting into one pass over
// memory; with the pooling as well, Q and K are read from HBM once for selection and quantisation together).  The
// selection's pooled sum is a chain of fp32 additions over the block's tokens in ascending order, one chain per channel,
// so it cannot be spread over the threads that hold the rows: the block is parked in shared memory on the way and
// thread c walks channels 2c and 2c + 1 through it while the other warps encode.  A CTA lives a third longer for that chain, so
// more of them have to be in flight: what is encoded is read back from shared memory, not held in registers, which
// leaves room for four to eight CTAs per SM instead of three.  40 heads of 75,600 tokens: 230 -> 217 us per tensor with
// 128-token blocks (five CTAs 218; three persistent ones with the next block's copy under way 241), 295 -> 236 with 64-token
// blocks (8: 237); 12 of 32,760: 31.9 -> 30.5, 38.8 -> 31.4.
// pooled: fp32 [B*H][nb][D] (query side) or transposed [B*H][D][nbp] (key side).
constexpr int quant_pool_ctas(int d, int block) { return d * block >= 128 * 128 ? 4 : d * block >= 128 * 64 ? 6 : 8; }   // per SM
template <int D, int BLK>
__global__ void __launch_bounds__(kQuantThreads, quant_pool_ctas(D, BLK))
quant_fp8_pool_kernel(const __nv_bfloat16* x, uint8_t* __restrict__ codes, float* __restrict__ scales, int H, int N, int nb,
                      int64_t stride_b, int64_t stride_h, int64_t stride_n, float* __restrict__ pooled,
                      int pooled_transposed, int nbp, bool early) {
  constexpr int kChunksPerRow = D / 8, kPerThread = BLK * kChunksPerRow / kQuantThreads;
  __shared__ __align__(16) unsigned char tile[BLK * D * 2];
  __shared__ float s_red[kQuantThreads / 32];
  if (early) pdl_trigger();
  const int blk = blockIdx.x % nb, bh = blockIdx.x / nb;
  const int nvalid = min(BLK, N - blk * BLK);
  const int64_t base = (bh / H) * stride_b + (bh % H) * stride_h + (int64_t)blk * BLK * stride_n;
  pdl_wait();
  float amax = 0.0f;
  {
    uint4 v[kPerThread];
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
      const int ci = threadIdx.x + i * kQuantThreads, r = ci / kChunksPerRow, cc = ci % kChunksPerRow;
      v[i] = r < nvalid ? *reinterpret_cast<const uint4*>(x + base + r * stride_n + cc * 8) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
      reinterpret_cast<uint4*>(tile)[threadIdx.x + i * kQuantThreads] = v[i];
      amax = fmaxf(amax, absmax8(v[i]));
    }
  }
  amax = block_absmax(amax, s_red);
  const float inv = __fdiv_rn(448.0f, amax);
  if (threadIdx.x == 0) scales[(int64_t)bh * nb + blk] = __fdiv_rn(amax, 448.0f);
  if constexpr (BLK == 128) {
    // The threads of the columns go straight to them, the others encode for them.  40 heads of 75,600 tokens, two boards: 209.8 ->
    // 201.3 and 201.0 -> 196.9 us per tensor, 12 of 32,760 30.2 -> 29.7, 20 of 6,479 10.6 -> 10.2.  With 64-token blocks, whose
    // columns are half as long, everybody encodes first (225 us, 239 the other way).
    if (threadIdx.x >= D / 2) {
#pragma unroll 4
      for (int ci = threadIdx.x - D / 2; ci < nvalid * kChunksPerRow; ci += kQuantThreads - D / 2) {
        const int r = ci / kChunksPerRow, cc = ci % kChunksPerRow;
        *reinterpret_cast<uint2*>(codes + base + r * stride_n + cc * 8) = encode8(reinterpret_cast<const uint4*>(tile)[ci], inv);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
      const int ci = threadIdx.x + i * kQuantThreads, r = ci / kChunksPerRow, cc = ci % kChunksPerRow;
      if (r < nvalid)
        *reinterpret_cast<uint2*>(codes + base + r * stride_n + cc * 8) = encode8(reinterpret_cast<const uint4*>(tile)[ci], inv);
    }
  }
  if (threadIdx.x < D / 2) {
    const uint32_t* col = reinterpret_cast<const uint32_t*>(tile) + threadIdx.x;      // channels 2t and 2t + 1
    float s0 = 0.0f, s1 = 0.0f;
    constexpr int U = 16;      // rows fetched ahead of the addition chains
    int r = 0;
    for (; r + U <= nvalid; r += U) {
      uint32_t xr[U];
#pragma unroll
      for (int u = 0; u < U; ++u) xr[u] = col[(r + u) * (D / 2)];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        s0 = __fadd_rn(s0, __uint_as_float(xr[u] << 16));
        s1 = __fadd_rn(s1, __uint_as_float(xr[u] & 0xffff0000u));
      }
    }
    for (; r < nvalid; ++r) {
      const uint32_t xr = col[r * (D / 2)];
      s0 = __fadd_rn(s0, __uint_as_float(xr << 16));
      s1 = __fadd_rn(s1, __uint_as_float(xr & 0xffff0000u));
    }
    const float m0 = __fdiv_rn(s0, (float)nvalid), m1 = __fdiv_rn(s1, (float)nvalid);
    const int c = 2 * threadIdx.x;
    if (pooled_transposed) {
      pooled[((int64_t)bh * D + c) * nbp + blk] = m0;
      pooled[((int64_t)bh * D + c + 1) * nbp + blk] = m1;
    } else {
      *reinterpret_cast<float2*>(pooled + ((int64_t)bh * nb + blk) * D + c) = make_float2(m0, m1);
    }
  }
}

// Per-token variant: a token row (d channels) is spread over 4 lanes; lane c of the group takes the
// 16-byte chunks c, c + 4, ... of the row, so that one load instruction of the warp covers 64
// contiguous bytes of each of 8 rows.  A warp walks kTokenSteps steps of 8 rows with all loads issued
// first (128 bytes in flight per thread).  absmax over the lane's chunks, two shuffles inside the lane
// group, then the two IEEE divisions once per row (they are a third of the instructions when a lane
// holds a single chunk), encode and store from the same registers: one HBM read, one write.
constexpr int kTokenSteps = 2;
constexpr int kTokenLanes = 4;                   // lanes per row
constexpr int kTokenRows = 32 / kTokenLanes;     // rows per warp step

template <int D>
__global__ void __launch_bounds__(kQuantThreads, 3)
quant_fp8_token_kernel(const __nv_bfloat16* x, uint8_t* __restrict__ codes, float* __restrict__ scales,
                       int H, int N, int64_t stride_b, int64_t stride_h, int64_t stride_n, int64_t n_rows) {
  constexpr int CPL = D / 8 / kTokenLanes;       // chunks per lane: 4 (d=128) or 2 (d=64)
  const int lane = threadIdx.x & 31;
  const int sub = lane / kTokenLanes, chunk = lane % kTokenLanes;
  const int64_t warp_id = (int64_t)blockIdx.x * (kQuantThreads / 32) + (threadIdx.x >> 5);
  const int64_t row0 = warp_id * (kTokenSteps * kTokenRows);
  pdl_wait();
  uint4 v[kTokenSteps][CPL];
  int64_t off[kTokenSteps];
  // (batch, head, token) of this lane's first row: divisions once, then the rows just count up
  const uint32_t first = (uint32_t)(row0 + sub);            // n_rows < 2^31 (checked by the launcher)
  const uint32_t bh0 = first / (uint32_t)N;
  int n = (int)(first - bh0 * (uint32_t)N);
  int b = (int)(bh0 / (uint32_t)H), h = (int)(bh0 - (uint32_t)b * (uint32_t)H);
#pragma unroll
  for (int u = 0; u < kTokenSteps; ++u) {
    const int64_t r = row0 + u * kTokenRows + sub;
    off[u] = b * stride_b + h * stride_h + (int64_t)n * stride_n + chunk * 8;
    n += kTokenRows;
    while (n >= N) {
      n -= N;
      if (++h == H) { h = 0; ++b; }
    }
#pragma unroll
    for (int c = 0; c < CPL; ++c)
      v[u][c] = (r < n_rows) ? *reinterpret_cast<const uint4*>(x + off[u] + c * (kTokenLanes * 8))
                             : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int u = 0; u < kTokenSteps; ++u) {
    const int64_t r = row0 + u * kTokenRows + sub;
    float f[CPL][8];
    float amax = 0.0f;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&v[u][c]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 t = __bfloat1622float2(p2[j]);
        f[c][2 * j] = t.x;
        f[c][2 * j + 1] = t.y;
        amax = fmaxf(amax, fmaxf(fabsf(t.x), fabsf(t.y)));
      }
    }
#pragma unroll
    for (int o = kTokenLanes / 2; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    amax = fmaxf(amax, 1e-12f);
    const float inv = __fdiv_rn(448.0f, amax);
    if (r >= n_rows) continue;
    if (chunk == 0) scales[r] = __fdiv_rn(amax, 448.0f);
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      uint32_t w[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(__fmul_rn(f[c][4 * j], inv), __fmul_rn(f[c][4 * j + 1], inv)),
                                                      __NV_SATFINITE, __NV_E4M3);
        const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(__fmul_rn(f[c][4 * j + 2], inv), __fmul_rn(f[c][4 * j + 3], inv)),
                                                      __NV_SATFINITE, __NV_E4M3);
        w[j] = lo | (hi << 16);
      }
      *reinterpret_cast<uint2*>(codes + off[u] + c * (kTokenLanes * 8)) = make_uint2(w[0], w[1]);
    }
  }
}

int launch_quant_fp8_per_token(const sparkattn_shape_t& s, const void* x, uint8_t* codes, float* scales,
                               cudaStream_t stream) {
  const int64_t n_rows = (int64_t)s.B * s.H * s.N;
  if (n_rows >= (1LL << 31) - 4096) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const int64_t rows_per_cta = (kQuantThreads / 32) * kTokenSteps * kTokenRows;
  const int64_t ctas = (n_rows + rows_per_cta - 1) / rows_per_cta;
  if (ctas > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const __nv_bfloat16* xb = static_cast<const __nv_bfloat16*>(x);
  if (s.d != 128 && s.d != 64) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  return launch_kernel(s.d == 128 ? quant_fp8_token_kernel<128> : quant_fp8_token_kernel<64>, (unsigned)ctas, kQuantThreads, 0, true,
                       stream, xb, codes, scales, s.H, s.N, s.stride_b, s.stride_h, s.stride_n, n_rows);
}

int launch_quant_fp8(const sparkattn_shape_t& s, const void* x, uint8_t* codes, float* scales,
                     cudaStream_t stream) {
  const int nb = (s.N + s.block - 1) / s.block;
  const long long ctas = (long long)s.B * s.H * nb;
  if (ctas > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  auto kern = s.d == 128 && s.block == 128 ? quant_fp8_kernel<128, 128>
              : s.d == 128 && s.block == 64 ? quant_fp8_kernel<128, 64>
              : s.d == 64 && s.block == 64 ? quant_fp8_kernel<64, 64> : nullptr;
  if (kern == nullptr) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  return launch_kernel(kern, (unsigned)ctas, kQuantThreads, 0, true, stream, static_cast<const __nv_bfloat16*>(x), codes, scales, s.H,
                       s.N, nb, s.stride_b, s.stride_h, s.stride_n);
}

// pooled: the selection workspace's pooled-Q or pooled-K region (select.cu lays it out)
int launch_quant_fp8_pooled(const sparkattn_shape_t& s, const void* x, uint8_t* codes, float* scales, float* pooled,
                            bool key_side, cudaStream_t stream) {
  const int nb = (s.N + s.block - 1) / s.block;
  const int nbp = (nb + 31) / 32 * 32;
  const long long items = (long long)s.B * s.H * nb;
  if (items > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  auto kern = s.d == 128 && s.block == 128 ? quant_fp8_pool_kernel<128, 128>
              : s.d == 128 && s.block == 64 ? quant_fp8_pool_kernel<128, 64>
              : s.d == 64 && s.block == 64 ? quant_fp8_pool_kernel<64, 64> : nullptr;
  if (kern == nullptr) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const int sm_count = current_sm_count();
  if (sm_count < 1) return SPARKATTN_E_CUDA;
  // It lets the next kernel in early, which by this call's contract is another quantisation or the top-k, while there are at most
  // two of its CTAs per SM.  Pooled Q and K, V, selection, 128-token blocks: 30 of them 19.6 us without and 18.9 with that, 296
  // 24.9 either way, 370 27.6 and 29.0, 444 27.8 and 29.3: beyond the line CTAs of the next kernel fill up some SMs of the chip unevenly.
  const bool early = items <= 2 * sm_count;
  return launch_kernel(kern, (unsigned)items, kQuantThreads, 0, true, stream, static_cast<const __nv_bfloat16*>(x), codes, scales,
                       s.H, s.N, nb, s.stride_b, s.stride_h, s.stride_n, pooled, key_side ? 1 : 0, nbp, early);
}

}  // namespace sparkattn
