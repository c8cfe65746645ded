// sparkattn_fwd, d = 64 (64-token blocks, bf16): block-sparse flash-attention forward for sm_100a, and the entry
// launcher of the forward.
//
// Computes the paper's sparse branch O_s = A_M(Q, K, V) (Sec. 4.1): exact
// softmax attention (Sec. 2, softmax(Q K^T / sqrt(d)) V) restricted, for every
// query block, to the key blocks of its kept list.
//
// One CTA owns one (batch, head, query block) work item.  A tile's chain (S product, softmax, P V product) is a
// string of latencies, 2800 clocks when a 64-key tile was taken in two halves by one chain, so the kept tiles are
// dealt out to C independent chains, each with its own S / P and O columns in TMEM, K / V slots, running maximum and
// row sum: chain c takes list positions c, c + C, ...  The chains are merged at the end: every warp can read the O
// of every chain for its own rows.  C = 4 (the whole TMEM, one CTA per SM) when the items do not fill the device,
// where the length of the chain is the whole time; else C = 2 with two CTAs per SM, which overlap one item's start and
// end with the other's tiles.
// 2 heads of 2,048 tokens, 16 tiles per item: 12.5 us (C = 2: 14.5; one chain in halves: 25); 12 heads of 8,000 tokens, 125
// tiles: 513 us (C = 4: 531; before: 1036), 770 clocks per tile and SM.  What bounds it there is the softmax: 64 rows live
// in two of the SM's four quarters, whose special-function units need 512 clocks for a tile's 4096 exponentials.
//   warps 4c, 4c+1   softmax of chain c: thread r owns query row r (the other two warps of each four would own MMA
//                    rows 64-127, which do not exist).  The row of S comes into registers in one pass, fp32 online
//                    softmax with packed fp32x2 FMA / ADD and 3-input max (row max / row sum need no shuffles), P is
//                    written back to TMEM over S as bf16, conditional rescale of O.
//   warp 4c+2        TMA producer of chain c: its K / V tiles, two slots each (128-byte swizzle); the first one Q as well.
//   warp 4c+3        MMA issuer of chain c: S = Q K_j^T (operands in shared memory) and O += P V_j (P from TMEM, V MN-major
//                    from shared memory) as tcgen05.mma with fp32 accumulators in TMEM.  S of the next tile is issued
//                    right behind the PV that reads P out of the same columns.  (One issuer for all chains takes
//                    14.1 us for the 16 tiles with four chains as with two.)
//
// Every wait on an mbarrier is bounded (common.cuh); a kept index outside
// [0, nb) is reported in the status word and its tile skipped by all roles.
#include <cuda.h>

#include "common.cuh"
#include "launch.h"
#include "tmap.h"

namespace sparkattn {

// In log2 units: O and l are only rescaled when the running row maximum grows
// by more than this; until then P may exceed 1 by at most 2^threshold, which
// bf16 holds without loss.  Exact: the final division by l uses the same
// reference maximum.
constexpr float kLazyRescaleLog2 = 8.0f;
constexpr int kD = 64, kBlk = 64;
constexpr int kFwdTile = kBlk * kD * 2;                 // bytes of a K or V tile: 64 rows of 128 bytes

template <int C>
struct Fwd64Smem {
  static constexpr int kQ = 0;                          // 128 MMA rows of 128 bytes, the first 64 loaded
  static constexpr int kKV = 2 * kFwdTile;              // [C][2 slots][K, V]
  static constexpr int kBars = kKV + C * 4 * kFwdTile;  // 12 barriers per chain, Q, flags
  static constexpr int kSums = kBars + 512;             // [C][64] (reference maximum, row sum)
  static constexpr int kList = kSums + C * 64 * 8;      // [kFwdMaxKept]
  static constexpr int kBytes = 1024 /*align slack*/ + kList + kFwdMaxKept * 4;
};

struct FwdParams {
  const int32_t* kept_idx;
  const int32_t* kept_cnt;
  __nv_bfloat16* out;
  float* lse;
  int32_t* status;
  int H, N, nb, kmax;
  int frame_tokens, window;  // causal frame window (0 = none): key frame in (query frame - window, query frame]
  int64_t stride_b, stride_h, stride_n;
  float scale_log2;  // softmax_scale * log2(e)
};

template <int C, bool WINDOW>
__global__ void __launch_bounds__(128 * C, C == 2 ? 2 : 1)
fwd_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
           const __grid_constant__ CUtensorMap tmap_v, const FwdParams p) {
  using Smem = Fwd64Smem<C>;
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Smem::kBars);
  // per chain: [2] K landed, [2] K free, [2] V landed, [2] V free, S complete, P written (64 arrivals), PV complete
  auto bar_k_full = [&](int c, int slot) { return bars + c * 12 + slot; };
  auto bar_k_free = [&](int c, int slot) { return bars + c * 12 + 2 + slot; };
  auto bar_v_full = [&](int c, int slot) { return bars + c * 12 + 4 + slot; };
  auto bar_v_free = [&](int c, int slot) { return bars + c * 12 + 6 + slot; };
  auto bar_s_full = [&](int c) { return bars + c * 12 + 8; };
  auto bar_p_full = [&](int c) { return bars + c * 12 + 9; };
  auto bar_pv_done = [&](int c) { return bars + c * 12 + 10; };
  uint64_t* bar_q_full = bars + 48;
  uint64_t* bar_sums = bars + 49;     // 64 C arrivals: every chain's last PV is complete and its sums are published
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(bars + 50);
  volatile int* s_abort = reinterpret_cast<volatile int*>(bars + 51);
  int* s_ntiles = reinterpret_cast<int*>(bars + 52);
  float2* s_sums = reinterpret_cast<float2*>(smem + Smem::kSums);
  int32_t* s_list = reinterpret_cast<int32_t*>(smem + Smem::kList);   // validated kept block indices
  auto tile_k = [&](int c, int slot) { return smem + Smem::kKV + (c * 4 + slot * 2) * kFwdTile; };
  auto tile_v = [&](int c, int slot) { return smem + Smem::kKV + (c * 4 + slot * 2 + 1) * kFwdTile; };

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int qb = blockIdx.x % p.nb;
  const int bh = blockIdx.x / p.nb;
  const int h = bh % p.H, b = bh / p.H;

  if (threadIdx.x == 0) {
    mbar_init(bar_q_full, 1);
    mbar_init(bar_sums, 64 * C);
#pragma unroll
    for (int c = 0; c < C; ++c) {
#pragma unroll
      for (int i = 0; i < 9; ++i) mbar_init(bars + c * 12 + i, 1);
      mbar_init(bar_p_full(c), 64);
      mbar_init(bar_pv_done(c), 1);
    }
    mbar_fence_init();
  }
  if (warp == 2) {
    if (lane == 0) {
      tma_prefetch_desc(&tmap_q);
      tma_prefetch_desc(&tmap_k);
      tma_prefetch_desc(&tmap_v);
    }
    __syncwarp();
    tmem_alloc(s_tmem_base, 128 * C);
    tmem_relinquish();
  }
  pdl_wait();
  // a timeout recorded by an earlier CTA of this launch makes the rest of the grid drain at once
  if (threadIdx.x == 0) *s_abort = (*reinterpret_cast<volatile int32_t*>(p.status) == SPARKATTN_E_DEVICE_TIMEOUT) ? 1 : 0;
  if (warp == 6) {
    // Stage the kept list in shared memory, in order, dropping (and reporting) indices outside [0, nb).
    const int cnt = p.kept_cnt ? min(max(p.kept_cnt[(int64_t)bh * p.nb + qb], 0), p.kmax) : p.kmax;
    const int32_t* list = p.kept_idx + ((int64_t)bh * p.nb + qb) * p.kmax;
    int out = 0;
    for (int base = 0; base < cnt; base += 32) {
      const int t = base + lane;
      const int kb = (t < cnt) ? list[t] : 0;
      const bool valid = (t < cnt) && kb >= 0 && kb < p.nb;
      if (t < cnt && !valid) report_status(p.status, SPARKATTN_E_BAD_INDEX, kb);
      const uint32_t ballot = __ballot_sync(0xffffffffu, valid);
      if (valid) s_list[out + __popc(ballot & ((1u << lane) - 1u))] = kb;
      out += __popc(ballot);
    }
    if (lane == 0) *s_ntiles = out;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem_base;      // chain c: S (P overlays its start) at columns [128 c, +64), O at [128 c + 64, +64)
  const bool dead = *s_abort != 0;
  const int ntiles = *s_ntiles;
  auto tiles_of = [&](int c) { return (ntiles - c + C - 1) / C; };

  if (dead) {
    // nothing to do: fall through to the teardown
  } else if ((warp & 3) == 2) {
    // ------------------------------------------------------------ TMA producer of chain warp / 4 (the first one: Q as well)
    const int c = warp >> 2, mine = tiles_of(c);
    if (lane == 0 && mine > 0) {
      if (c == 0) {
        mbar_expect_tx(bar_q_full, kFwdTile);
        tma_load_4d(smem + Smem::kQ, &tmap_q, bar_q_full, 0, qb * kBlk, h, b);
      }
      for (int n = 0; n < mine; ++n) {
        const int slot = n & 1;
        const int kb = s_list[n * C + c];
        if (n >= 2 && !mbar_wait(bar_k_free(c, slot), ((n >> 1) - 1) & 1, s_abort, p.status, 1)) break;
        mbar_expect_tx(bar_k_full(c, slot), kFwdTile);
        tma_load_4d(tile_k(c, slot), &tmap_k, bar_k_full(c, slot), 0, kb * kBlk, h, b);
        if (n >= 2 && !mbar_wait(bar_v_free(c, slot), ((n >> 1) - 1) & 1, s_abort, p.status, 2)) break;
        mbar_expect_tx(bar_v_full(c, slot), kFwdTile);
        tma_load_4d(tile_v(c, slot), &tmap_v, bar_v_full(c, slot), 0, kb * kBlk, h, b);
      }
    }
  } else if ((warp & 3) == 3) {
    // -------------------------------------------------------------- MMA issuer of chain warp / 4 (one thread; its MMAs execute in order)
    const int c = warp >> 2, mine = tiles_of(c);
    if (lane == 0 && mine > 0) {
      constexpr uint32_t idesc_qk = make_idesc(1u, 128, kBlk, false);
      constexpr uint32_t idesc_pv = make_idesc(1u, 128, kD, true);
      const uint32_t tS = tmem + c * 128;
      const uint64_t dQ = make_smem_desc_sw128(smem_u32(smem + Smem::kQ), 16);
      const uint32_t q_lo = (uint32_t)dQ, q_hi = (uint32_t)(dQ >> 32);
      auto issue_s = [&](int n) {
        const uint64_t dK = make_smem_desc_sw128(smem_u32(tile_k(c, n & 1)), 16);
        const uint32_t k_lo = (uint32_t)dK, k_hi = (uint32_t)(dK >> 32);
#pragma unroll
        for (int kk = 0; kk < kD / 16; ++kk)
          mma_ss<false>(tS, make_desc(q_lo + ((kk * 32) >> 4), q_hi), make_desc(k_lo + ((kk * 32) >> 4), k_hi), idesc_qk,
                        kk != 0 ? 1u : 0u);
        tc_commit(bar_s_full(c));
        tc_commit(bar_k_free(c, n & 1));
      };
      bool ok = mbar_wait(bar_q_full, 0, s_abort, p.status, 3) && mbar_wait(bar_k_full(c, 0), 0, s_abort, p.status, 5);
      if (ok) {
        tc_fence_after();
        issue_s(0);
      }
      for (int n = 0; ok && n < mine; ++n) {
        const int slot = n & 1;
        const bool more = n + 1 < mine;
        // this V and the next K have normally landed long before P is written
        ok = mbar_wait(bar_v_full(c, slot), (n >> 1) & 1, s_abort, p.status, 6);
        if (ok && more) ok = mbar_wait(bar_k_full(c, slot ^ 1), ((n + 1) >> 1) & 1, s_abort, p.status, 5);
        if (ok) ok = mbar_wait(bar_p_full(c), n & 1, s_abort, p.status, 7);
        if (!ok) break;
        tc_fence_after();
        const uint64_t dV = make_smem_desc_sw128(smem_u32(tile_v(c, slot)), kFwdTile);
        const uint32_t v_lo = (uint32_t)dV, v_hi = (uint32_t)(dV >> 32);
#pragma unroll
        for (int kk = 0; kk < kBlk / 16; ++kk)
          mma_ts<false>(tS + 64, tS + kk * 8, make_desc(v_lo + ((kk * 16 * 128) >> 4), v_hi), idesc_pv, (n | kk) != 0 ? 1u : 0u);
        if (more) issue_s(n + 1);
        tc_commit(bar_pv_done(c));
        tc_commit(bar_v_free(c, slot));
      }
    }
  } else if ((warp & 2) == 0) {
    // ----------------------------------------------------------------- softmax of chain warp / 4
    const int chain = warp >> 2;
    const int row = threadIdx.x & 127;                // query row inside the block = TMEM lane (0..63)
    const uint32_t lane_off = (uint32_t)((warp & 1) * 32) << 16;
    const int q_row = qb * kBlk + row;
    const bool row_valid = q_row < p.N;
    // keys this row may attend to: [klo, khi) (everything up to N without a causal window)
    int klo = 0, khi = p.N;
    if constexpr (WINDOW) {
      const int fi = min(q_row, p.N - 1) / p.frame_tokens;
      klo = max(fi - p.window + 1, 0) * p.frame_tokens;
      khi = (int)min((long long)(fi + 1) * p.frame_tokens, (long long)p.N);
    }
    const uint32_t tS = tmem + chain * 128 + lane_off;
    const float c = p.scale_log2;                     // logit -> log2 units
    const int mine = tiles_of(chain);
    float m_used = -INFINITY, l = 0.0f;
    bool ok = true;
    for (int n = 0; ok && n < mine; ++n) {
      const int kb = s_list[n * C + chain];
      const int c_lo = klo - kb * kBlk, c_hi = khi - kb * kBlk;      // this row's valid columns of the tile: [c_lo, c_hi)
      ok = __all_sync(0xffffffffu, mbar_wait(bar_s_full(chain), n & 1, s_abort, p.status, 8));
      if (!ok) break;
      tc_fence_after();
      uint32_t sr[kBlk];
#pragma unroll
      for (int ch = 0; ch < kBlk / 32; ++ch) tmem_ld32(tS + ch * 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[ch * 32]));
      tc_wait_ld();
      if ((WINDOW && c_lo > 0) || c_hi < kBlk) {  // ragged last key block / keys outside the causal window get weight 0
#pragma unroll
        for (int i = 0; i < kBlk; ++i)
          if ((WINDOW && i < c_lo) || i >= c_hi) sr[i] = 0xff800000u;
      }
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < kBlk; i += 2) mx[(i >> 1) & 3] = fmax3(mx[(i >> 1) & 3], __uint_as_float(sr[i]), __uint_as_float(sr[i + 1]));
      const float m_new = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * c;
      float alpha = 1.0f;
      bool need = false;
      if (n == 0 || m_used == -INFINITY) {
        m_used = m_new;               // first tile, or nothing accumulated for this row yet (all keys so far masked)
      } else if (m_new > m_used + kLazyRescaleLog2) {
        alpha = fast_exp2(m_used - m_new);
        m_used = m_new;
        need = true;
      }
      if (__any_sync(0xffffffffu, need)) {
        // O must be quiescent: the chain's last PV is the previous tile's
        ok = __all_sync(0xffffffffu, mbar_wait(bar_pv_done(chain), (n - 1) & 1, s_abort, p.status, 10));
        if (!ok) break;
        tc_fence_after();
        l *= alpha;
        const uint64_t a2 = pack_f32x2(alpha, alpha);
#pragma unroll 1
        for (int ch = 0; ch < kD / 16; ++ch) {
          uint32_t r[16];
          tmem_ld16(tS + 64 + ch * 16, r);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float2 o2 = unpack_f32x2(fmul2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), a2));
            r[i] = __float_as_uint(o2.x);
            r[i + 1] = __float_as_uint(o2.y);
          }
          tmem_st16(tS + 64 + ch * 16, r);
        }
      }

      // P = exp2(S*c - m) as bf16, written over the start of S
      const float neg_m = m_used == -INFINITY ? 0.0f : -m_used;   // a fully masked row: exp2(-inf) = 0, not NaN
      const uint64_t c2 = pack_f32x2(c, c), nm2 = pack_f32x2(neg_m, neg_m);
      uint64_t lsum0 = pack_f32x2(0.0f, 0.0f), lsum1 = lsum0;
      uint32_t w[kBlk / 2];
#pragma unroll
      for (int i = 0; i < kBlk; i += 2) {
        const float2 x = unpack_f32x2(ffma2(pack_f32x2(__uint_as_float(sr[i]), __uint_as_float(sr[i + 1])), c2, nm2));
        const float e0 = fast_exp2(x.x), e1 = fast_exp2(x.y);
        if ((i >> 1) & 1) lsum1 = fadd2(lsum1, pack_f32x2(e0, e1));
        else lsum0 = fadd2(lsum0, pack_f32x2(e0, e1));
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(e0, e1);
        w[i / 2] = *reinterpret_cast<const uint32_t*>(&h2);
      }
      tmem_st32(tS, *reinterpret_cast<const uint32_t(*)[32]>(&w[0]));
      const float2 ls = unpack_f32x2(fadd2(lsum0, lsum1));
      l += ls.x + ls.y;
      tc_wait_st();
      tc_fence_before();
      mbar_arrive(bar_p_full(chain));
    }

    // ---------------------------------------------------------------- merge of the chains and epilogue
    if (ok && mine > 0) ok = __all_sync(0xffffffffu, mbar_wait(bar_pv_done(chain), (mine - 1) & 1, s_abort, p.status, 9));
    if (ok) {
      tc_fence_after();
      tc_fence_before();
      s_sums[chain * 64 + row] = make_float2(m_used, l);
      mbar_arrive(bar_sums);
      ok = __all_sync(0xffffffffu, mbar_wait(bar_sums, 0, s_abort, p.status, 11));
    }
    if (ok) {
      tc_fence_after();
      float2 sums[C];
      float m = -INFINITY;
#pragma unroll
      for (int i = 0; i < C; ++i) {
        sums[i] = s_sums[i * 64 + row];
        if (sums[i].y != 0.0f) m = fmaxf(m, sums[i].x);
      }
      float w[C], total = 0.0f;
#pragma unroll
      for (int i = 0; i < C; ++i) {
        w[i] = sums[i].y != 0.0f ? fast_exp2(sums[i].x - m) : 0.0f;
        total += w[i] * sums[i].y;
      }
      const float inv = total > 0.0f ? 1.0f / total : 0.0f;     // no admissible key at all: zero row, lse = -inf
      // this chain's warps write columns [64 / C * chain, +64 / C) of the row
      constexpr int kCols = kD / C;
      float o[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) o[j] = 0.0f;
#pragma unroll
      for (int i = 0; i < C; ++i) {
        if (i < ntiles) {                                        // chains without a tile have no O
#pragma unroll
          for (int ch = 0; ch < kCols / 16; ++ch) {
            uint32_t r[16];
            tmem_ld16(tmem + i * 128 + 64 + lane_off + chain * kCols + ch * 16, r);
            tc_wait_ld();
            if (w[i] != 0.0f) {
#pragma unroll
              for (int j = 0; j < 16; ++j) o[ch * 16 + j] = fmaf(__uint_as_float(r[j]), w[i], o[ch * 16 + j]);
            }
          }
        }
      }
      if (row_valid) {
        __nv_bfloat16* orow = p.out + b * p.stride_b + h * p.stride_h + (int64_t)q_row * p.stride_n + chain * kCols;
#pragma unroll
        for (int i = 0; i < kCols / 8; ++i) {
          uint32_t ww[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(o[8 * i + 2 * j] * inv, o[8 * i + 2 * j + 1] * inv);
            ww[j] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          reinterpret_cast<uint4*>(orow)[i] = make_uint4(ww[0], ww[1], ww[2], ww[3]);
        }
        if (p.lse && chain == 0) p.lse[(int64_t)bh * p.N + q_row] = fmaf(m, 0.6931471805599453f, log2f(total) * 0.6931471805599453f);   // one rounding
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    if (*s_abort) __nanosleep(200000);  // let copies / MMAs in flight land before the CTA's resources go
    tc_fence_after();
    tmem_dealloc(tmem, 128 * C);
  }
}

// ------------------------------------------------------------------ host side

size_t fwd_workspace_bytes(const sparkattn_shape_t& s, int kmax) {
  // the pipelined kernel keeps range-checked, compacted copies of the kept lists behind the header
  if (fwd_pipe_supported(s)) return fwd_pipe_workspace_bytes(s, kmax);
  return kWorkspaceHeaderBytes;
}

// clears the workspace header ahead of a kernel that reports into it
__global__ void clear_header_kernel(int32_t* header) {
  pdl_trigger();
  pdl_wait();
  header[threadIdx.x] = 0;
}

template <int C>
static int launch_fwd_t(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const FwdParams& prm, long long ctas,
                        cudaStream_t stream) {
  auto kern = prm.frame_tokens > 0 ? fwd_kernel<C, true> : fwd_kernel<C, false>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Fwd64Smem<C>::kBytes) != cudaSuccess)
    return SPARKATTN_E_CUDA;
  return launch_kernel(kern, (unsigned)ctas, 128 * C, Fwd64Smem<C>::kBytes, true, stream, mq, mk, mv, prm);
}

int launch_fwd(const sparkattn_shape_t& s, int dtype, const void* q, const void* k, const void* v,
               const float* q_scale, const float* k_scale, const float* v_scale, const int32_t* kept_idx,
               const int32_t* kept_cnt, int kmax, int frame_tokens, int window, const int32_t* block_valid, void* out,
               float* lse, void* workspace, cudaStream_t stream) {
  const bool fp8 = dtype == SPARKATTN_FP8_E4M3;
  if (fwd_pipe_supported(s))
    return launch_fwd_pipe(s, fp8, q, k, v, q_scale, k_scale, v_scale, kept_idx, kept_cnt, kmax, frame_tokens, window,
                           block_valid, out, lse, workspace, stream);
  // d = 128 always runs the persistent kernel; a sequence too long for its list pre-pass is not served
  if (s.d != 64 || s.block != 64 || fp8 || block_valid != nullptr) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const int elt = 2;
  CUtensorMap mq, mk, mv;
  int rc;
  if ((rc = make_token_map(&mq, q, elt, s, s.block)) != SPARKATTN_OK) return rc;
  if ((rc = make_token_map(&mk, k, elt, s, s.block)) != SPARKATTN_OK) return rc;
  if ((rc = make_token_map(&mv, v, elt, s, s.block)) != SPARKATTN_OK) return rc;
  FwdParams prm;
  prm.kept_idx = kept_idx;
  prm.kept_cnt = kept_cnt;
  prm.out = static_cast<__nv_bfloat16*>(out);
  prm.lse = lse;
  prm.status = static_cast<int32_t*>(workspace);
  prm.H = s.H;
  prm.N = s.N;
  prm.nb = (s.N + s.block - 1) / s.block;
  prm.kmax = kmax;
  prm.frame_tokens = frame_tokens;
  prm.window = window;
  prm.stride_b = s.stride_b;
  prm.stride_h = s.stride_h;
  prm.stride_n = s.stride_n;
  const float sc = s.softmax_scale > 0.0f ? s.softmax_scale : 1.0f / sqrtf((float)s.d);
  prm.scale_log2 = sc * 1.4426950408889634f;
  const long long ctas = (long long)s.B * s.H * prm.nb;
  if (ctas > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const int sm_count = current_sm_count();
  if (sm_count < 1) return SPARKATTN_E_CUDA;
  if ((rc = launch_kernel(clear_header_kernel, 1, kWorkspaceHeaderBytes / 4, 0, true, stream, prm.status)) != SPARKATTN_OK) return rc;
  // four chains while no SM gets a second item: 64 to 144 items of 16 tiles 12.5-13 us against 14.5-15 with two; 256 items
  // of 3 tiles 11.3 against 7.9, 512 of 32 tiles 68 against 59
  return ctas <= sm_count ? launch_fwd_t<4>(mq, mk, mv, prm, ctas, stream) : launch_fwd_t<2>(mq, mk, mv, prm, ctas, stream);
}

}  // namespace sparkattn
