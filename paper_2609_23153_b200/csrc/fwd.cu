// sparkattn_fwd, d = 64 (64-token blocks, bf16): block-sparse flash-attention forward for sm_100a, and the entry
// launcher of the forward.
//
// Computes the paper's sparse branch O_s = A_M(Q, K, V) (Sec. 4.1): exact
// softmax attention (Sec. 2, softmax(Q K^T / sqrt(d)) V) restricted, for every
// query block, to the key blocks of its kept list.
//
// One CTA owns one (batch, head, query block) work item.  A query block has 64 rows and the tensor core 128, each half of
// them in two of the SM's four quarters, so the rows are there twice and the halves take different key blocks: [Q; Q] times
// [K1; K2] has Q K1^T and Q K2^T on its diagonal, [P1; P2] times [V1 | V2] has P1 V1 and P2 V2.  What lies off the diagonal is
// computed and never read: the products cost as much as two of half the size, and the softmax warps of all four
// quarters have work (with 64 rows in two quarters the special-function units of the other two stood idle).
// A chain takes pairs of kept blocks one after the other (S product, softmax, P V product), each half with its own running
// maximum and row sum; S of the next pair runs under the softmax of this one.  C chains share the list (chain c takes pairs c,
// c + C, ...), and the 2 C partial results of a row are merged through shared memory at the end.  C = 2 (the whole
// TMEM, one CTA per SM) when the items do not fill the device; else C = 1 with two CTAs per SM, which overlap one
// item's start and end with the other's tiles.
//   warps 4c .. 4c+3     softmax of chain c: thread r owns query row r mod 64, warps 4c and 4c+1 the pair's first block, the other
//                        two its second.  The row of S comes into registers in one pass, fp32 online softmax with packed
//                        fp32x2 FMA / ADD and 3-input max (row max / row sum need no shuffles), P goes to shared memory as
//                        bf16 (S may be overwritten as soon as it sits in registers), conditional rescale of O.
//   warp 4C + c          TMA producer of chain c: its K / V pairs, two slots each (128-byte swizzle); the first one Q as well.
//   warp 5C + c          MMA issuer of chain c: tcgen05.mma with fp32 accumulators in TMEM, all operands from shared memory.
// An odd list's last pair has a block past the end for a second one: zeros from the copy, all of its columns masked.
// Bound by the softmax warps: a pair's 8192 exponentials are 512 clocks of the SM's special-function units, 1,170 clocks per
// pair and SM at 125 tiles per item, where one chain runs its short steps under the other's exponentials.  Against one query block
// per CTA with its 64 rows in two quarters (four or two chains of single tiles), us: 2 heads of 2,048 tokens, 16 of 32 tiles 12.6 ->
// 10.2 (9.5 since it clears the status itself); 16 heads, 32 of 32 59 -> 42; 6 heads of 6,479, 10 of 102 30.5 -> 26.0, in a window of three frames 48 -> 38.5; 12 heads of
// 8,000, 125 of 125 520 -> 410; 40 heads of 32,760, 15 of 512 1020 -> 900.
//
// Every wait on an mbarrier is bounded (common.cuh); a kept index outside
// [0, nb) is skipped by all roles and reported in the status word when the CTA winds down.
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

constexpr int kFwdPair = 2 * kFwdTile;                  // of the two tiles of a pair

template <int C>
struct Fwd64Smem {
  static constexpr int kQ = 0;                          // the 64 query rows twice
  static constexpr int kP = kFwdPair;                   // [C] P of both halves
  static constexpr int kKV = kP + C * kFwdPair;         // [C][2 slots][K, V]
  static constexpr int kBars = kKV + C * 4 * kFwdPair;  // 12 barriers per chain, Q, flags
  static constexpr int kSums = kBars + 512;             // [2 C][64] (reference maximum, row sum)
  static constexpr int kList = kSums + 2 * C * 64 * 8;  // [kFwdMaxKept]
  static constexpr int kBytes = 1024 /*align slack*/ + kList + kFwdMaxKept * 4;
  // after the last product the K / V slots hold the weighted O of the 2 C half chains, fp32, rows padded to 68
  static constexpr int kORow = kD + 4;
  static_assert(2 * C * 64 * kORow * 4 <= C * 4 * kFwdPair, "partial results fit the K / V slots");
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
__global__ void __launch_bounds__(192 * C, C == 1 ? 2 : 1)
fwd_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
           const __grid_constant__ CUtensorMap tmap_v, const FwdParams p) {
  using Smem = Fwd64Smem<C>;
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Smem::kBars);
  // per chain: [2] K landed, [2] K free, [2] V landed, [2] V free, S complete, S in registers (128 arrivals), P written (128
  // arrivals), PV complete
  auto bar_k_full = [&](int c, int slot) { return bars + c * 12 + slot; };
  auto bar_k_free = [&](int c, int slot) { return bars + c * 12 + 2 + slot; };
  auto bar_v_full = [&](int c, int slot) { return bars + c * 12 + 4 + slot; };
  auto bar_v_free = [&](int c, int slot) { return bars + c * 12 + 6 + slot; };
  auto bar_s_full = [&](int c) { return bars + c * 12 + 8; };
  auto bar_s_free = [&](int c) { return bars + c * 12 + 9; };
  auto bar_p_full = [&](int c) { return bars + c * 12 + 10; };
  auto bar_pv_done = [&](int c) { return bars + c * 12 + 11; };
  uint64_t* bar_q_full = bars + 48;
  uint64_t* bar_sums = bars + 49;     // 128 C arrivals: every chain's last PV is complete and its sums are published
  uint64_t* bar_parts = bars + 50;    // 128 C arrivals: every half chain's weighted O is in shared memory
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(bars + 51);
  volatile int* s_abort = reinterpret_cast<volatile int*>(bars + 52);
  int* s_ntiles = reinterpret_cast<int*>(bars + 53);
  int* s_bad = s_ntiles + 1;          // place of an invalid index in the list, or -1
  int* s_code = s_ntiles + 2;         // first CTA, C = 2: there was a code in the header it has taken
  float2* s_sums = reinterpret_cast<float2*>(smem + Smem::kSums);
  int32_t* s_list = reinterpret_cast<int32_t*>(smem + Smem::kList);   // validated kept block indices
  auto tile_k = [&](int c, int slot) { return smem + Smem::kKV + (c * 4 + slot * 2) * kFwdPair; };
  auto tile_v = [&](int c, int slot) { return smem + Smem::kKV + (c * 4 + slot * 2 + 1) * kFwdPair; };

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int qb = blockIdx.x % p.nb;
  const int bh = blockIdx.x / p.nb;
  const int h = bh % p.H, b = bh / p.H;
  constexpr int kTmaWarp = 4 * C, kMmaWarp = 5 * C;

  if (threadIdx.x == 0) {
    mbar_init(bar_q_full, 1);
    mbar_init(bar_sums, 128 * C);
    mbar_init(bar_parts, 128 * C);
#pragma unroll
    for (int c = 0; c < C; ++c) {
#pragma unroll
      for (int i = 0; i < 9; ++i) mbar_init(bars + c * 12 + i, 1);
      mbar_init(bar_s_free(c), 128);
      mbar_init(bar_p_full(c), 128);
      mbar_init(bar_pv_done(c), 1);
    }
    mbar_fence_init();
  }
  if (warp == kTmaWarp) {
    if (lane == 0) {
      tma_prefetch_desc(&tmap_q);
      tma_prefetch_desc(&tmap_k);
      tma_prefetch_desc(&tmap_v);
    }
    __syncwarp();
    tmem_alloc(s_tmem_base, 256 * C);
    tmem_relinquish();
  }
  pdl_wait();
  // C = 2 is one wave of CTAs at most and clears the status itself (64 items of 16 tiles 9.5 us, 10.2 with a kernel in front for it;
  // one launch less: of 3 tiles 6.1 and 8.4); C = 1 has it cleared, and a timeout recorded by an earlier
  // CTA of the launch makes the rest of the grid drain at once
  if (threadIdx.x == 0) {
    if constexpr (C == 2) {
      if (blockIdx.x == 0) *s_code = take_header(p.status);
      *s_abort = 0;
    } else {
      *s_abort = (*reinterpret_cast<volatile int32_t*>(p.status) == SPARKATTN_E_DEVICE_TIMEOUT) ? 1 : 0;
    }
  }
  if (warp == kMmaWarp) {
    // Stage the kept list in shared memory, in order, dropping (and noting, for the report at the end) indices outside [0, nb).
    const int cnt = p.kept_cnt ? min(max(p.kept_cnt[(int64_t)bh * p.nb + qb], 0), p.kmax) : p.kmax;
    const int32_t* list = p.kept_idx + ((int64_t)bh * p.nb + qb) * p.kmax;
    int out = 0, bad = -1;                          // bad: place in the list of one of them
    for (int base = 0; base < cnt; base += 32) {
      const int t = base + lane;
      const int kb = (t < cnt) ? list[t] : 0;
      const bool valid = (t < cnt) && kb >= 0 && kb < p.nb;
      if (t < cnt && !valid) bad = t;
      const uint32_t ballot = __ballot_sync(0xffffffffu, valid);
      if (valid) s_list[out + __popc(ballot & ((1u << lane) - 1u))] = kb;
      out += __popc(ballot);
    }
    bad = __reduce_max_sync(0xffffffffu, bad);
    if (lane == 0) {
      *s_ntiles = out;
      *s_bad = bad;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem_base;      // chain c: S at columns [256 c, +128), O at [256 c + 128, +128)
  const bool dead = *s_abort != 0;
  const int ntiles = *s_ntiles;
  auto pairs_of = [&](int c) { return ((ntiles + 1) / 2 - c + C - 1) / C; };
  // key block of half `half` of pair n of chain c; past the end of an odd list: the block behind the last one, which is empty
  auto block_of = [&](int c, int n, int half) {
    const int at = 2 * (n * C + c) + half;
    return at < ntiles ? s_list[at] : p.nb;
  };

  if (dead) {
    // nothing to do: fall through to the teardown
  } else if (warp >= kMmaWarp) {
    // -------------------------------------------------------------- MMA issuer of chain warp - 5 C (one thread; its MMAs execute in order)
    const int c = warp - kMmaWarp, mine = pairs_of(c);
    if (lane == 0 && mine > 0) {
      constexpr uint32_t idesc_qk = make_idesc(1u, 128, 2 * kBlk, false);
      constexpr uint32_t idesc_pv = make_idesc(1u, 128, 2 * kD, true);
      const uint32_t tS = tmem + c * 256;
      const uint64_t dQ = make_smem_desc_sw128(smem_u32(smem + Smem::kQ), 16);
      const uint64_t dP = make_smem_desc_sw128(smem_u32(smem + Smem::kP + c * kFwdPair), 16);
      const uint32_t q_lo = (uint32_t)dQ, p_lo = (uint32_t)dP, q_hi = (uint32_t)(dQ >> 32);
      auto issue_s = [&](int n) {
        const uint32_t k_lo = (uint32_t)make_smem_desc_sw128(smem_u32(tile_k(c, n & 1)), 16);
#pragma unroll
        for (int kk = 0; kk < kD / 16; ++kk)
          mma_ss<false>(tS, make_desc(q_lo + ((kk * 32) >> 4), q_hi), make_desc(k_lo + ((kk * 32) >> 4), q_hi), idesc_qk,
                        kk != 0 ? 1u : 0u);
        tc_commit(bar_s_full(c));
        tc_commit(bar_k_free(c, n & 1));
      };
      bool ok = pipe_wait(bar_q_full, 0, s_abort, 3) && pipe_wait(bar_k_full(c, 0), 0, s_abort, 5);
      if (ok) {
        tc_fence_after();
        issue_s(0);
      }
      for (int n = 0; ok && n < mine; ++n) {
        const int slot = n & 1;
        if (n + 1 < mine) {
          ok = pipe_wait(bar_k_full(c, slot ^ 1), ((n + 1) >> 1) & 1, s_abort, 5);
          if (ok) ok = pipe_wait(bar_s_free(c), n & 1, s_abort, 4);
          if (!ok) break;
          tc_fence_after();
          issue_s(n + 1);
        }
        ok = pipe_wait(bar_v_full(c, slot), (n >> 1) & 1, s_abort, 6);
        if (ok) ok = pipe_wait(bar_p_full(c), n & 1, s_abort, 7);
        if (!ok) break;
        tc_fence_after();
        const uint64_t dV = make_smem_desc_sw128(smem_u32(tile_v(c, slot)), kFwdTile);      // the pair's tiles are two slabs of columns
        const uint32_t v_lo = (uint32_t)dV, v_hi = (uint32_t)(dV >> 32);
#pragma unroll
        for (int kk = 0; kk < kBlk / 16; ++kk)
          mma_ss<false>(tS + 128, make_desc(p_lo + ((kk * 32) >> 4), q_hi), make_desc(v_lo + ((kk * 16 * 128) >> 4), v_hi), idesc_pv,
                        (n | kk) != 0 ? 1u : 0u);
        tc_commit(bar_pv_done(c));
        tc_commit(bar_v_free(c, slot));
      }
    }
  } else if (warp >= kTmaWarp) {
    // ------------------------------------------------------------ TMA producer of chain warp - 4 C (the first one: Q as well)
    const int c = warp - kTmaWarp, mine = pairs_of(c);
    if (lane == 0 && mine > 0) {
      if (c == 0) {
        mbar_expect_tx(bar_q_full, kFwdPair);
        tma_load_4d(smem + Smem::kQ, &tmap_q, bar_q_full, 0, qb * kBlk, h, b);
        tma_load_4d(smem + Smem::kQ + kFwdTile, &tmap_q, bar_q_full, 0, qb * kBlk, h, b);
      }
      for (int n = 0; n < mine; ++n) {
        const int slot = n & 1;
        const int k0 = block_of(c, n, 0) * kBlk, k1 = block_of(c, n, 1) * kBlk;
        if (n >= 2 && !pipe_wait(bar_k_free(c, slot), ((n >> 1) - 1) & 1, s_abort, 1)) break;
        mbar_expect_tx(bar_k_full(c, slot), kFwdPair);
        tma_load_4d(tile_k(c, slot), &tmap_k, bar_k_full(c, slot), 0, k0, h, b);
        tma_load_4d(tile_k(c, slot) + kFwdTile, &tmap_k, bar_k_full(c, slot), 0, k1, h, b);
        if (n >= 2 && !pipe_wait(bar_v_free(c, slot), ((n >> 1) - 1) & 1, s_abort, 2)) break;
        mbar_expect_tx(bar_v_full(c, slot), kFwdPair);
        tma_load_4d(tile_v(c, slot), &tmap_v, bar_v_full(c, slot), 0, k0, h, b);
        tma_load_4d(tile_v(c, slot) + kFwdTile, &tmap_v, bar_v_full(c, slot), 0, k1, h, b);
      }
    }
  } else {
    // ----------------------------------------------------------------- softmax of chain warp / 4
    const int chain = warp >> 2, half = (warp >> 1) & 1;
    const int row = threadIdx.x & 63;                 // query row inside the block
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const int q_row = qb * kBlk + row;
    const bool row_valid = q_row < p.N;
    // keys this row may attend to: [klo, khi) (everything up to N without a causal window)
    int klo = 0, khi = p.N;
    if constexpr (WINDOW) {
      const int fi = min(q_row, p.N - 1) / p.frame_tokens;
      klo = max(fi - p.window + 1, 0) * p.frame_tokens;
      khi = (int)min((long long)(fi + 1) * p.frame_tokens, (long long)p.N);
    }
    const uint32_t tS = tmem + chain * 256 + lane_off + half * kBlk;           // this half's columns of S and of O
    const uint32_t tO = tmem + chain * 256 + 128 + lane_off + half * kD;
    unsigned char* p_row = smem + Smem::kP + chain * kFwdPair + (half * kBlk + row) * 128;
    const float c = p.scale_log2;                     // logit -> log2 units
    const int mine = pairs_of(chain);
    float m_used = -INFINITY, l = 0.0f;
    bool ok = true;
    for (int n = 0; ok && n < mine; ++n) {
      const int kb = block_of(chain, n, half);
      const int c_lo = klo - kb * kBlk, c_hi = khi - kb * kBlk;      // this row's valid columns of the tile: [c_lo, c_hi)
      ok = __all_sync(0xffffffffu, pipe_wait(bar_s_full(chain), n & 1, s_abort, 8));
      if (!ok) break;
      tc_fence_after();
      uint32_t sr[kBlk];
#pragma unroll
      for (int ch = 0; ch < kBlk / 32; ++ch) tmem_ld32(tS + ch * 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[ch * 32]));
      tc_wait_ld();
      tc_fence_before();
      mbar_arrive(bar_s_free(chain));             // the next pair's S may overwrite this one
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
      // The chain's last PV is the previous pair's: once it is complete P has been read and O is quiescent.  It is waited for behind
      // the first kWaitAt pieces of eight columns.  Two of them where the length of the chain is all there is (C = 2: 64 items
      // of 16 tiles 0.2 us less than with none); none where the stores of P should run under the exponentials (C = 1: 12 heads of
      // 8,000 tokens 410 us, two 432, all eight 450).
      constexpr int kWaitAt = C == 2 ? 2 : 0;
      auto wait_pv = [&]() { return n == 0 || __all_sync(0xffffffffu, pipe_wait(bar_pv_done(chain), (n - 1) & 1, s_abort, 10)); };
      const bool rescale = __any_sync(0xffffffffu, need);
      if (rescale) {
        ok = wait_pv();
        if (!ok) break;
        tc_fence_after();
        l *= alpha;
        const uint64_t a2 = pack_f32x2(alpha, alpha);
#pragma unroll 1
        for (int ch = 0; ch < kD / 16; ++ch) {
          uint32_t r[16];
          tmem_ld16(tO + ch * 16, r);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float2 o2 = unpack_f32x2(fmul2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), a2));
            r[i] = __float_as_uint(o2.x);
            r[i + 1] = __float_as_uint(o2.y);
          }
          tmem_st16(tO + ch * 16, r);
        }
        tc_wait_st();
      }

      // P = exp2(S*c - m) as bf16
      const float neg_m = m_used == -INFINITY ? 0.0f : -m_used;   // a fully masked row: exp2(-inf) = 0, not NaN
      const uint64_t c2 = pack_f32x2(c, c), nm2 = pack_f32x2(neg_m, neg_m);
      uint64_t lsum0 = pack_f32x2(0.0f, 0.0f), lsum1 = lsum0;
      uint32_t w[kBlk / 2];
      auto store = [&](int j) {                   // 128-byte swizzle
        *reinterpret_cast<uint4*>(p_row + ((j ^ (row & 7)) << 4)) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      };
#pragma unroll
      for (int j = 0; j < kBlk / 8; ++j) {
        if (j == kWaitAt) {
          if (!rescale) ok = wait_pv();
          if (!ok) break;
#pragma unroll
          for (int i = 0; i < j; ++i) store(i);
        }
#pragma unroll
        for (int i = 8 * j; i < 8 * j + 8; i += 2) {
          const float2 x = unpack_f32x2(ffma2(pack_f32x2(__uint_as_float(sr[i]), __uint_as_float(sr[i + 1])), c2, nm2));
          const float e0 = fast_exp2(x.x), e1 = fast_exp2(x.y);
          if ((i >> 1) & 1) lsum1 = fadd2(lsum1, pack_f32x2(e0, e1));
          else lsum0 = fadd2(lsum0, pack_f32x2(e0, e1));
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(e0, e1);
          w[i / 2] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        if (j >= kWaitAt) store(j);
      }
      if (!ok) break;
      const float2 ls = unpack_f32x2(fadd2(lsum0, lsum1));
      l += ls.x + ls.y;
      tc_fence_before();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(bar_p_full(chain));
    }

    // ---------------------------------------------------------------- merge of the half chains and epilogue
    if (ok && mine > 0) ok = __all_sync(0xffffffffu, pipe_wait(bar_pv_done(chain), (mine - 1) & 1, s_abort, 9));
    const int part = chain * 2 + half;
    if (ok) {
      tc_fence_after();
      s_sums[part * 64 + row] = make_float2(m_used, l);
      mbar_arrive(bar_sums);
      ok = __all_sync(0xffffffffu, pipe_wait(bar_sums, 0, s_abort, 11));
    }
    if (ok) {
      // every product of the CTA is complete: the K / V slots are free for the weighted O of the half chains
      float m = -INFINITY;
#pragma unroll
      for (int i = 0; i < 2 * C; ++i) {
        const float2 s = s_sums[i * 64 + row];
        if (s.y != 0.0f) m = fmaxf(m, s.x);
      }
      float total = 0.0f;
#pragma unroll
      for (int i = 0; i < 2 * C; ++i) {
        const float2 s = s_sums[i * 64 + row];
        if (s.y != 0.0f) total += fast_exp2(s.x - m) * s.y;
      }
      const float inv = total > 0.0f ? 1.0f / total : 0.0f;     // no admissible key at all: zero row, lse = -inf
      const float w = l != 0.0f ? fast_exp2(m_used - m) : 0.0f;
      constexpr int kORow = Smem::kORow;
      float* parts = reinterpret_cast<float*>(smem + Smem::kKV);
      float* mine_o = parts + (part * 64 + row) * kORow;
#pragma unroll
      for (int ch = 0; ch < kD / 16; ++ch) {
        uint32_t r[16] = {};
        if (mine > 0) {                                          // (a chain without a pair has no O)
          tmem_ld16(tO + ch * 16, r);
          tc_wait_ld();
        }
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
          float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (w != 0.0f)
            v = make_float4(__uint_as_float(r[j]) * w, __uint_as_float(r[j + 1]) * w, __uint_as_float(r[j + 2]) * w, __uint_as_float(r[j + 3]) * w);
          *reinterpret_cast<float4*>(mine_o + ch * 16 + j) = v;
        }
      }
      mbar_arrive(bar_parts);
      ok = __all_sync(0xffffffffu, pipe_wait(bar_parts, 0, s_abort, 12));
      if (ok && row_valid) {
        // this half chain's threads write columns [64 / 2C * part, +64 / 2C) of the row
        constexpr int kCols = kD / (2 * C);
        __nv_bfloat16* orow = p.out + b * p.stride_b + h * p.stride_h + (int64_t)q_row * p.stride_n + part * kCols;
        const float* src = parts + row * kORow + part * kCols;
#pragma unroll
        for (int i = 0; i < kCols / 8; ++i) {
          float o[8] = {};
#pragma unroll
          for (int k = 0; k < 2 * C; ++k) {
            const float4 x = *reinterpret_cast<const float4*>(src + k * 64 * kORow + 8 * i);
            const float4 y = *reinterpret_cast<const float4*>(src + k * 64 * kORow + 8 * i + 4);
            o[0] += x.x; o[1] += x.y; o[2] += x.z; o[3] += x.w;
            o[4] += y.x; o[5] += y.y; o[6] += y.z; o[7] += y.w;
          }
          uint32_t ww[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(o[2 * j] * inv, o[2 * j + 1] * inv);
            ww[j] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          reinterpret_cast<uint4*>(orow)[i] = make_uint4(ww[0], ww[1], ww[2], ww[3]);
        }
        if (p.lse && part == 0) p.lse[(int64_t)bh * p.N + q_row] = fmaf(m, 0.6931471805599453f, log2f(total) * 0.6931471805599453f);   // one rounding
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kTmaWarp) {
    if (*s_abort) __nanosleep(200000);  // let copies / MMAs in flight land before the CTA's resources go
    tc_fence_after();
    tmem_dealloc(tmem, 256 * C);
  }
  if (threadIdx.x == 0 && (*s_abort >= kAbortTimeout || *s_bad >= 0)) {
    if (*s_bad >= 0) report_early(p.status, SPARKATTN_E_BAD_INDEX, p.kept_idx[((int64_t)bh * p.nb + qb) * p.kmax + *s_bad]);
    report_abort(p.status, *s_abort);
  }
  if constexpr (C == 2) {
    if (blockIdx.x == 0 && *s_code) recheck_lists(p.kept_idx, p.kept_cnt, (int)gridDim.x, p.nb, p.kmax, p.status, threadIdx.x, 192 * C);
  }
}

// ------------------------------------------------------------------ host side

size_t fwd_workspace_bytes(const sparkattn_shape_t& s, int kmax) {
  // the pipelined kernel keeps range-checked, compacted copies of the kept lists behind the header
  if (fwd_pipe_supported(s)) return fwd_pipe_workspace_bytes(s, kmax);
  return kWorkspaceHeaderBytes;
}

// clears the workspace header ahead of a kernel that reports into it (C = 1, whose CTAs come in waves)
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
  return launch_kernel(kern, (unsigned)ctas, 192 * C, Fwd64Smem<C>::kBytes, true, stream, mq, mk, mv, prm);
}

int launch_fwd(const sparkattn_shape_t& s, int dtype, const void* q, const void* k, const void* v,
               const float* q_scale, const float* k_scale, const float* v_scale, const int32_t* kept_idx,
               const int32_t* kept_cnt, int kmax, int frame_tokens, int window, const int32_t* block_valid, void* out,
               float* lse, void* workspace, cudaStream_t stream) {
  const bool fp8 = dtype == SPARKATTN_FP8_E4M3;
  if (fwd_pipe_supported(s))
    return launch_fwd_pipe(s, fp8, q, k, v, q_scale, k_scale, v_scale, kept_idx, kept_cnt, kmax, frame_tokens, window,
                           block_valid, out, lse, workspace, stream);
  // d = 128 always runs the persistent kernel; a sequence too long for its merged lists is not served
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
  // two chains while no SM gets a second item, us against one chain and two CTAs per SM (the status cleared in front of both): 64 items of 16 tiles 10.3 / 11.5, 128 10.7 /
  // 11.9; but 160 19.0 / 14.2, 256 items of 3 tiles 12.3 / 8.1, 512 of 32 56.5 / 42.4
  if (ctas <= sm_count) return launch_fwd_t<2>(mq, mk, mv, prm, ctas, stream);
  if ((rc = launch_kernel(clear_header_kernel, 1, kWorkspaceHeaderBytes / 4, 0, true, stream, prm.status)) != SPARKATTN_OK) return rc;
  return launch_fwd_t<1>(mq, mk, mv, prm, ctas, stream);
}

}  // namespace sparkattn
