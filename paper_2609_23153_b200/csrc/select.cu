// sparkattn_select: pooled block scores + top-k kept-block lists.
//
// The paper's selector M_phi (Sec. 2, Sec. 4.1) is left open (it lists kinds of
// selectors, top-k over per-block scores among them); the rule implemented here is
//   pooled mean of every token block (fp32, tokens added in ascending order,
//   one IEEE divide), score(i,j) = fmaf chain over channels, keep the topk
//   key blocks first under (score descending, index ascending), emit ascending.
// Every floating-point step has a fixed order so that the result is defined
// bit for bit; this is why scoring runs on the FMA pipe and not on tensor cores.
//
// Two kernels:
//   pool_kernel       two resident CTAs per SM walk the (tensor, batch, head, block) items: a block's rows go to shared
//                     memory in one go (asynchronous copies into one of two buffers) while thread c adds up two
//                     channels of the block before.  The only HBM-heavy step (2 bytes per element); writes pooled Q
//                     [BH][nb][d] and pooled K transposed [BH][d][nbp].
//   topk_small_kernel nb <= 64: one CTA per 8 query blocks, a warp each, all of the head's pooled K in shared memory.
//   topk_kernel       nb <= 256: one CTA per 8, 16 or 32 query blocks of one (batch, head): scores against all key
//                     blocks as an RT x 4 register tile per thread (pooled K through a ring of asynchronous copies in
//                     shared memory, packed fp32x2 FMAs over row pairs), then a warp per query block (or two) selects
//                     the topk largest keys exactly (keys in registers for nb <= 1280) and compacts them in order.
//   topk_wide_kernel  nb > 256: 16 or 8 query blocks per CTA of ten warps, pooled K straight from L2.
//   list_all_kernel   in place of all of them when every block is kept.
// The second is launched before the first has drained (programmatic dependent launch) and waits inside.
#include <atomic>

#include "common.cuh"
#include "launch.h"
#include "tmap.h"

namespace sparkattn {

constexpr int kTopkThreads = 256;
constexpr int kSmallBlocks = 64;      // key blocks up to which topk_small_kernel scores and selects

static inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

size_t select_workspace_bytes(const sparkattn_shape_t& s) {
  const int nb = (s.N + s.block - 1) / s.block;
  const int nbp = round_up(nb, 32);
  const size_t bh = (size_t)s.B * s.H;
  return kWorkspaceHeaderBytes + bh * nb * s.d * sizeof(float) + bh * s.d * nbp * sizeof(float);
}

// Bound by HBM.  A sum is a chain of additions over the block's tokens, so a warp that reads its rows as it adds
// them waits for memory block / 16 times over; here a whole block (32 KB at most) is on its way at once, into one of
// two buffers, while the block before it is added up.
// 40 heads of 75,600 tokens: 225 us (6.9 TB/s) against 255 us for one warp per block with 16 rows in flight; 3 heads of
// 1,200 tokens: a few us against 12, all of them latency.  Two CTAs of two buffers per SM; three take 238 us.
constexpr int kPoolCtasPerSm = 2;
template <int D>
__global__ void __launch_bounds__(D / 2)
pool_kernel(const __nv_bfloat16* q, const __nv_bfloat16* k, float* __restrict__ pq,
            float* __restrict__ pkT, int H, int N, int blk_size, int nb, int nbp, int64_t stride_b,
            int64_t stride_h, int64_t stride_n, int64_t n_items /* B*H*nb */,
            const int32_t* block_valid /* [nb] real tokens per block, or NULL */,
            int32_t* __restrict__ header) {
  extern __shared__ __align__(16) unsigned char smem_raw[];      // [2][blk_size][D] bf16
  constexpr int kThreads = D / 2;
  constexpr int kRowChunks = D / 8;                    // 16-byte chunks of a row
  constexpr int kRowStep = kThreads / kRowChunks;      // rows the CTA covers with one copy per thread
  const int buf_bytes = blk_size * D * 2;
  const int chunk = threadIdx.x % kRowChunks, r0 = threadIdx.x / kRowChunks;
  struct Item {
    bool is_k;
    int blk, nvalid;
    int64_t bh;
  };
  auto item_at = [&](int64_t w) {
    Item it;
    it.is_k = w >= n_items;
    const int64_t item = it.is_k ? w - n_items : w;
    it.blk = (int)(item % nb);
    it.bh = item / nb;
    it.nvalid = min(blk_size, N - it.blk * blk_size);
    if (block_valid != nullptr) it.nvalid = max(1, min(it.nvalid, block_valid[it.blk]));   // bricks padded to whole blocks
    return it;
  };
  auto fetch = [&](const Item& it, int buf) {
    const int h = (int)(it.bh % H), b = (int)(it.bh / H);
    const __nv_bfloat16* src =
        (it.is_k ? k : q) + b * stride_b + h * stride_h + (int64_t)(it.blk * blk_size + r0) * stride_n + chunk * 8;
    uint32_t dst = smem_u32(smem_raw) + buf * buf_bytes + r0 * (D * 2) + chunk * 16;
#pragma unroll 8
    for (int r = r0; r < it.nvalid; r += kRowStep, src += kRowStep * stride_n, dst += kRowStep * D * 2) cp_async16(dst, src);
  };

  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0)
    for (int e = threadIdx.x; e < kWorkspaceHeaderBytes / 4; e += kThreads) header[e] = 0;
  Item next = item_at(blockIdx.x);
  fetch(next, 0);
  cp_async_commit();
  int buf = 0;
  for (int64_t w = blockIdx.x; w < 2 * n_items; w += gridDim.x, buf ^= 1) {
    const Item it = next;
    if (w + gridDim.x < 2 * n_items) {
      next = item_at(w + gridDim.x);
      fetch(next, buf ^ 1);
    }
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const uint32_t* col = reinterpret_cast<const uint32_t*>(smem_raw + buf * buf_bytes) + threadIdx.x;   // channels 2t and 2t + 1
    float s0 = 0.0f, s1 = 0.0f;
    constexpr int U = 16;
    int r = 0;
    for (; r + U <= it.nvalid; r += U) {
      uint32_t x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = col[(r + u) * (D / 2)];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        s0 = __fadd_rn(s0, __uint_as_float(x[u] << 16));
        s1 = __fadd_rn(s1, __uint_as_float(x[u] & 0xffff0000u));
      }
    }
    for (; r < it.nvalid; ++r) {
      const uint32_t x = col[r * (D / 2)];
      s0 = __fadd_rn(s0, __uint_as_float(x << 16));
      s1 = __fadd_rn(s1, __uint_as_float(x & 0xffff0000u));
    }
    const float nv = (float)it.nvalid;
    const float m0 = __fdiv_rn(s0, nv), m1 = __fdiv_rn(s1, nv);
    const int ch = 2 * threadIdx.x;
    if (it.is_k) {
      pkT[(it.bh * D + ch) * nbp + it.blk] = m0;
      pkT[(it.bh * D + ch + 1) * nbp + it.blk] = m1;
    } else {
      *reinterpret_cast<float2*>(pq + (it.bh * nb + it.blk) * D + ch) = make_float2(m0, m1);
    }
    __syncthreads();                     // the buffer may be filled again
  }
}

// Order-preserving map fp32 -> uint32 (larger float = larger key); -0 is folded onto +0.
__device__ __forceinline__ uint32_t score_key(float s) {
  const uint32_t u = __float_as_uint(s + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Exact selection of the topk largest keys of one row by one warp (ties: lowest index first),
// written in ascending index order.  KeyAt(j) returns key j; the keys are visited several times.
// Only the key blocks jlo..jhi are candidates (the whole row without a causal window); the caller
// passes topk <= jhi - jlo + 1 and key_at returns 0 (below every real key) outside that range.
template <typename KeyAt>
__device__ __forceinline__ void select_row(KeyAt key_at, int nb, int jlo, int jhi, int topk, int lane,
                                           int32_t* __restrict__ dst) {
  // value of the topk-th largest key, one bit per pass from the top; bits above the highest bit in
  // which the row's keys differ are common to all keys and need no pass
  uint32_t kmin = 0xffffffffu, kmaxv = 0u;
  for (int j = jlo + lane; j <= jhi; j += 32) {
    const uint32_t kj = key_at(j);
    kmin = min(kmin, kj);
    kmaxv = max(kmaxv, kj);
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmaxv = __reduce_max_sync(0xffffffffu, kmaxv);
  const int top_bit = 31 - __clz(kmin ^ kmaxv);              // -1 when all keys are equal
  uint32_t thr = (top_bit >= 31) ? 0u : (kmaxv & ~((2u << max(top_bit, 0)) - 1u));
  if (top_bit < 0) thr = kmaxv;
  for (int bit = top_bit; bit >= 0; --bit) {
    const uint32_t cand = thr | (1u << bit);
    int cnt = 0;
    for (int j = lane; j < nb; j += 32) cnt += (key_at(j) >= cand);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (cnt >= topk) thr = cand;
    if (cnt == topk) break;          // exactly the keys wanted: the lower bits of the threshold do not matter
  }
  int ngreater = 0;
  for (int j = lane; j < nb; j += 32) ngreater += (key_at(j) > thr);
  ngreater = __reduce_add_sync(0xffffffffu, ngreater);
  const int ties_allowed = topk - ngreater;  // >= 1: lowest indices among the keys equal to thr

  int out = 0, ties_seen = 0;
  const uint32_t lt_mask = (1u << lane) - 1u;
  for (int base = 0; base < nb; base += 32) {
    const int j = base + lane;
    const bool valid = j >= jlo && j <= jhi;
    const uint32_t kj = valid ? key_at(j) : 0u;
    const bool tie = valid && (kj == thr);
    const uint32_t tie_ballot = __ballot_sync(0xffffffffu, tie);
    const int tie_rank = ties_seen + __popc(tie_ballot & lt_mask);
    const bool keep = valid && ((kj > thr) || (tie && tie_rank < ties_allowed));
    const uint32_t keep_ballot = __ballot_sync(0xffffffffu, keep);
    if (keep) dst[out + __popc(keep_ballot & lt_mask)] = j;
    out += __popc(keep_ballot);
    ties_seen += __popc(tie_ballot);
  }
}

// The same with a row's keys held in KR registers per lane (nb <= 32 * KR), for NR rows of a warp at once: the search
// is a chain of warp reductions, and two rows' chains fill each other's gaps.  Keys outside the candidate range
// are held as 0, below every candidate (candidates are >= 1).
//
// The threshold is first sought among the four largest keys of every lane, 128 values, two bits per pass (the
// counts of the three candidates share one reduction), and the search ends as soon as a candidate has exactly topk
// keys at or above it.  When no lane holds more than four keys >= the threshold found, every key >= it is among the
// 128 and it separates the row's topk largest keys.  Otherwise (a lane with five such keys, or topk > 128) the
// search runs over all KR keys.  Either way the selection is exact; only the cost differs.
template <int KR, bool WINDOW, int NR>
__device__ __forceinline__ void select_rows_regs(const uint32_t* const (&key)[NR], int nb, const int (&jlo)[NR],
                                                 const int (&jhi)[NR], const int (&topk)[NR], int lane,
                                                 int32_t* const (&dst)[NR]) {
  constexpr uint32_t kFull = 0xffffffffu;
  uint32_t kr[NR][KR];
  uint32_t m1[NR], m2[NR], m3[NR], m4[NR];                     // sorted four largest keys of the lane
  uint32_t kmaxv[NR], thr[NR];
  int sh[NR];
  bool active[NR];
  bool any = false;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    m1[r] = m2[r] = m3[r] = m4[r] = 0u;
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      const int j = lane + 32 * u;
      kr[r][u] = (WINDOW ? (j >= jlo[r] && j <= jhi[r]) : (j < nb)) ? key[r][j] : 0u;
    }
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      uint32_t x = kr[r][u], t;
      t = min(m1[r], x); m1[r] = max(m1[r], x); x = t;
      t = min(m2[r], x); m2[r] = max(m2[r], x); x = t;
      t = min(m3[r], x); m3[r] = max(m3[r], x); x = t;
      m4[r] = max(m4[r], x);
    }
    kmaxv[r] = __reduce_max_sync(kFull, m1[r]);
    // the topk-th largest lies between the smallest of the lanes' p-th largest keys, p = ceil(topk / 32) (32 p values
    // are at least that), and the row maximum; the bits above the highest bit in which the two differ are common to
    // both and need no pass
    const int p = (topk[r] + 31) / 32;
    const uint32_t lo = __reduce_min_sync(kFull, p == 1 ? m1[r] : p == 2 ? m2[r] : p == 3 ? m3[r] : p == 4 ? m4[r] : 0u);
    const int top_bit = 31 - __clz(lo ^ kmaxv[r]);             // -1 when the two are equal
    sh[r] = max(top_bit, 0) & ~1;
    thr[r] = sh[r] >= 30 ? 0u : (kmaxv[r] & ~((4u << sh[r]) - 1u));
    active[r] = topk[r] <= 128 && top_bit >= 0;
    if (top_bit < 0) thr[r] = kmaxv[r];
    any = any || active[r];
  }
  while (any) {
    any = false;
    int cnt[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const uint32_t c1 = thr[r] | (1u << sh[r]), c2 = thr[r] | (2u << sh[r]), c3 = thr[r] | (3u << sh[r]);
      cnt[r] = (m1[r] >= c1) + (m2[r] >= c1) + (m3[r] >= c1) + (m4[r] >= c1) +
               (((m1[r] >= c2) + (m2[r] >= c2) + (m3[r] >= c2) + (m4[r] >= c2)) << 10) +
               (((m1[r] >= c3) + (m2[r] >= c3) + (m3[r] >= c3) + (m4[r] >= c3)) << 20);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) cnt[r] = __reduce_add_sync(kFull, cnt[r]);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (active[r]) {
        const int n1 = cnt[r] & 1023, n2 = (cnt[r] >> 10) & 1023, n3 = cnt[r] >> 20;
        int n = -1;
        if (n3 >= topk[r]) { thr[r] |= 3u << sh[r]; n = n3; }
        else if (n2 >= topk[r]) { thr[r] |= 2u << sh[r]; n = n2; }
        else if (n1 >= topk[r]) { thr[r] |= 1u << sh[r]; n = n1; }
        active[r] = n != topk[r] && sh[r] > 0;
        sh[r] = max(sh[r] - 2, 0);
        any = any || active[r];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int k = topk[r];
    uint32_t t = thr[r];
    int nge = 0;
#pragma unroll
    for (int u = 0; u < KR; ++u) nge += (kr[r][u] >= t);
    if (k > 128 || t == 0u || __any_sync(kFull, nge > 4)) {
      // bitwise search over all keys, from the highest bit in which the row's candidates differ
      uint32_t kmin = 0xffffffffu;
#pragma unroll
      for (int u = 0; u < KR; ++u) {
        const int j = lane + 32 * u;
        if (WINDOW ? (j >= jlo[r] && j <= jhi[r]) : (j < nb)) kmin = min(kmin, kr[r][u]);
      }
      kmin = __reduce_min_sync(kFull, kmin);
      const int top_bit = 31 - __clz(kmin ^ kmaxv[r]);
      t = (top_bit >= 31) ? 0u : (kmaxv[r] & ~((2u << max(top_bit, 0)) - 1u));
      if (top_bit < 0) t = kmaxv[r];
      for (int bit = top_bit; bit >= 0; --bit) {
        const uint32_t cand = t | (1u << bit);
        int cnt = 0;
#pragma unroll
        for (int u = 0; u < KR; ++u) cnt += (kr[r][u] >= cand);
        cnt = __reduce_add_sync(kFull, cnt);
        if (cnt >= k) t = cand;
        if (cnt == k) break;
      }
      nge = 0;
#pragma unroll
      for (int u = 0; u < KR; ++u) nge += (kr[r][u] >= t);
    }
    // ordered compaction: keys above the threshold, then the lowest-indexed keys equal to it.  With t >= 1 the
    // zero keys that stand for blocks outside the candidate range never pass a comparison (t = 0 only when a
    // candidate's own key is 0, the key of one NaN pattern: the general path below handles it).
    nge = __reduce_add_sync(kFull, nge);
    const uint32_t lt_mask = (1u << lane) - 1u;
    int out = 0;
    if (nge == k && t != 0u) {   // no surplus of keys equal to the threshold: keep every key >= t
      // lane u takes the ballot of keys 32u .. 32u + 31 (and of the 32 ballots after the 32nd), an exclusive sum over
      // the lanes gives its place in the list, and it writes its few indices itself
#pragma unroll
      for (int base = 0; base < KR; base += 32) {
        uint32_t mine = 0u;
#pragma unroll
        for (int u = base; u < KR && u < base + 32; ++u) {
          const uint32_t keep_ballot = __ballot_sync(kFull, kr[r][u] >= t);
          if (lane == u - base) mine = keep_ballot;
        }
        int at = __popc(mine);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int before = __shfl_up_sync(kFull, at, o);
          if (lane >= o) at += before;
        }
        const int total = __shfl_sync(kFull, at, 31);
        int32_t* d = dst[r] + out + at - __popc(mine);
        for (; mine != 0u; mine &= mine - 1u) *d++ = (base + lane) * 32 + __ffs(mine) - 1;
        out += total;
      }
      continue;
    }
    int ngreater = 0;
#pragma unroll
    for (int u = 0; u < KR; ++u) ngreater += (kr[r][u] > t);
    ngreater = __reduce_add_sync(kFull, ngreater);
    const int ties_allowed = k - ngreater;  // >= 1: lowest indices among the keys equal to t
    int ties_seen = 0;
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      if (32 * u < nb) {
        const int j = lane + 32 * u;
        const bool valid = WINDOW ? (j >= jlo[r] && j <= jhi[r]) : (j < nb);
        const bool tie = valid && (kr[r][u] == t);
        const uint32_t tie_ballot = __ballot_sync(kFull, tie);
        const int tie_rank = ties_seen + __popc(tie_ballot & lt_mask);
        const bool keep = valid && ((kr[r][u] > t) || (tie && tie_rank < ties_allowed));
        const uint32_t keep_ballot = __ballot_sync(kFull, keep);
        if (keep) dst[r][out + __popc(keep_ballot & lt_mask)] = j;
        out += __popc(keep_ballot);
        ties_seen += __popc(tie_ballot);
      }
    }
  }
}

// Causal frame window (Sec. 1, auto-regressive extension): only the key blocks that hold a key some row of query block i may
// attend to are candidates, a contiguous run jlo..jhi.
__device__ __forceinline__ void window_range(int i, int N, int blk_size, int frame_tokens, int window, int& jlo, int& jhi) {
  const int r0 = i * blk_size, r1 = min((i + 1) * blk_size, N) - 1;
  const int f0 = max(r0 / frame_tokens - window + 1, 0);
  const int kend = (int)min((long long)(r1 / frame_tokens + 1) * frame_tokens, (long long)N);
  jlo = (int)((long long)f0 * frame_tokens / blk_size);
  jhi = (kend - 1) / blk_size;
}

// Selection of a CTA's rows from their keys in shared memory: a warp takes rows WARPS apart, NR of them at a time.
// KR: keys per lane, nb <= 32 KR; 0: more than 256 blocks, by their number.
template <bool WINDOW, int WARPS, int NR, int KR>
__device__ __forceinline__ void select_tile(const uint32_t* s_key, int nb, int nbp, int topk, int64_t bh, int i0, int nrows, int N,
                                            int blk_size, int frame_tokens, int window, int32_t* __restrict__ kept_idx,
                                            int32_t* __restrict__ kept_cnt) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int first = warp; first < nrows; first += WARPS * NR) {
    const uint32_t* key[NR];
    int32_t* dst[NR];
    int jlo[NR], jhi[NR], k_row[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int row = first + WARPS * r < nrows ? first + WARPS * r : first;        // (beyond the last row: the first one again)
      key[r] = s_key + (int64_t)row * nbp;
      dst[r] = kept_idx + (bh * nb + i0 + row) * (int64_t)topk;
      jlo[r] = 0;
      jhi[r] = nb - 1;
      if constexpr (WINDOW) {
        window_range(i0 + row, N, blk_size, frame_tokens, window, jlo[r], jhi[r]);
      }
      k_row[r] = min(topk, jhi[r] - jlo[r] + 1);
      if constexpr (WINDOW)
        for (int t = k_row[r] + lane; t < topk; t += 32) dst[r][t] = -1;    // unused tail of a list cut short by the window
      if (lane == 0 && kept_cnt != nullptr) kept_cnt[bh * nb + i0 + row] = k_row[r];
    }
    if constexpr (KR > 0) {
      select_rows_regs<KR, WINDOW, NR>(key, nb, jlo, jhi, k_row, lane, dst);
    } else if (nb <= 32 * 20) {
      select_rows_regs<20, WINDOW, NR>(key, nb, jlo, jhi, k_row, lane, dst);
    } else if (nb <= 32 * 40) {
      select_rows_regs<40, WINDOW, NR>(key, nb, jlo, jhi, k_row, lane, dst);
    } else {
#pragma unroll
      for (int r = 0; r < NR; ++r)
        select_row([&](int j) { return (WINDOW ? (j >= jlo[r] && j <= jhi[r]) : (j < nb)) ? key[r][j] : 0u; }, nb, jlo[r],
                   jhi[r], k_row[r], lane, dst[r]);
    }
  }
}

// the keys of a thread's 2 * PAIRS x 4 scores into the rows of the key tile
template <int PAIRS>
__device__ __forceinline__ void store_keys(const uint64_t (&acc)[4][PAIRS], uint32_t* out, int nbp) {
#pragma unroll
  for (int r = 0; r < PAIRS; ++r) {
    uint4 lo, hi;
    float2 a;
    a = unpack_f32x2(acc[0][r]); lo.x = score_key(a.x); hi.x = score_key(a.y);
    a = unpack_f32x2(acc[1][r]); lo.y = score_key(a.x); hi.y = score_key(a.y);
    a = unpack_f32x2(acc[2][r]); lo.z = score_key(a.x); hi.z = score_key(a.y);
    a = unpack_f32x2(acc[3][r]); lo.w = score_key(a.x); hi.w = score_key(a.y);
    *reinterpret_cast<uint4*>(out + (2 * r) * nbp) = lo;
    *reinterpret_cast<uint4*>(out + (2 * r + 1) * nbp) = hi;
  }
}

// Where the means were pooled by another call, the top-k is the kernel that clears the workspace's header (a memset in front of it kept
// it from being launched early: FP8 chain of 3 heads of 1,200 tokens 37.6 us with it, 35.5 without, 6 of 6,479 56.0 and 52.1, 12 of
// 32,760 590.8 and 587.9).  Nothing in these kernels reports into it.
__device__ __forceinline__ void clear_header(int32_t* header) {
  if (header != nullptr && blockIdx.x == 0 && threadIdx.x < kWorkspaceHeaderBytes / 4) header[threadIdx.x] = 0;
}

// RT x 4 scores per thread; the CTA's 8 warps are RG groups of RT rows times 8 / RG groups of 128 key blocks.  NS ring
// stages of KC channels.
template <int RT, int RG, int KC, int NS>
struct TopkShape {
  static constexpr int kRows = RT * RG, kCols = 128 * (8 / RG);
  static constexpr int kStageFloats = KC * kCols;
  static constexpr size_t smem_bytes(int d, int nbp) {
    return (size_t)(NS * kStageFloats + kRows * d) * sizeof(float) + (size_t)kRows * nbp * sizeof(uint32_t);
  }
};

template <int D, int RT, int RG, int KC, int NS, bool WINDOW>
__global__ void __launch_bounds__(kTopkThreads, 2)
topk_kernel(const float* pq, const float* pkT, int32_t* __restrict__ kept_idx,
            int32_t* __restrict__ kept_cnt, int nb, int nbp, int topk, int groups_per_bh, int N, int blk_size,
            int frame_tokens, int window, int32_t* __restrict__ header) {
  using Shape = TopkShape<RT, RG, KC, NS>;
  constexpr int R = Shape::kRows, JT = Shape::kCols;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* s_ring = reinterpret_cast<float*>(smem_raw);                 // [NS][KC][JT] pooled K, channel-major
  // pooled Q of the CTA's R query blocks, channel-major: s_pq[c][r], so that one 16-byte load yields four rows of one
  // channel as two packed fp32x2 operands
  float* s_pq = s_ring + NS * Shape::kStageFloats;                    // [D][R]
  uint32_t* s_key = reinterpret_cast<uint32_t*>(s_pq + R * D);        // [R][nbp]

  const int64_t bh = blockIdx.x / groups_per_bh;
  const int i0 = (blockIdx.x % groups_per_bh) * R;
  const int nrows = min(R, nb - i0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* kcol = pkT + bh * D * (int64_t)nbp;

  constexpr int kSteps = D / KC;                                      // stages per sweep over JT key blocks
  const int steps = (nbp + JT - 1) / JT * kSteps;
  auto issue = [&](int step) {
    if (step < steps) {
      const int j0 = step / kSteps * JT, c0 = step % kSteps * KC;
      const int w4 = min(JT, nbp - j0) / 4;
      const uint32_t dst = smem_u32(s_ring + step % NS * Shape::kStageFloats);
      const float* src = kcol + (int64_t)c0 * nbp + j0;
#pragma unroll
      for (int e = threadIdx.x; e < KC * JT / 4; e += kTopkThreads) {
        const int c = e / (JT / 4), x = e % (JT / 4);
        if (x < w4) cp_async16(dst + (c * JT + 4 * x) * 4, src + (int64_t)c * nbp + 4 * x);
      }
    }
    cp_async_commit();
  };

  pdl_wait();
  clear_header(header);
#pragma unroll
  for (int p = 0; p < NS - 1; ++p) issue(p);
  for (int e = threadIdx.x; e < R * (D / 4); e += kTopkThreads) {
    const int r = e % R, c = e / R * 4;
    const float4 x = r < nrows ? *reinterpret_cast<const float4*>(pq + (bh * nb + i0 + r) * D + c)
                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    s_pq[c * R + r] = x.x; s_pq[(c + 1) * R + r] = x.y; s_pq[(c + 2) * R + r] = x.z; s_pq[(c + 3) * R + r] = x.w;
  }

  // scores: a thread owns 4 adjacent key blocks and RT query blocks and walks the channels in ascending order.
  // fma.rn.f32x2 is a pair of IEEE fmaf over two rows, so every accumulator sees exactly the chain
  // a = fmaf(pq[i,c], pk[j,c], a), c ascending.  Columns nb..nbp-1 of pooled K are padding whose scores are stored
  // but never read.
  constexpr int kPairs = RT / 2;
  const int rg = warp % RG, jc = warp / RG * 128 + lane * 4;        // first row of the thread: rg * RT; its column in the sweep
  for (int j0 = 0, step = 0; j0 < nbp; j0 += JT) {
    uint64_t acc[4][kPairs];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int r = 0; r < kPairs; ++r) acc[u][r] = pack_f32x2(0.0f, 0.0f);
    const bool mine = j0 + warp / RG * 128 < nbp;                   // the warp has a key block in this sweep
#pragma unroll 1
    for (int s = 0; s < kSteps; ++s, ++step) {
      cp_async_wait<NS - 2>();
      __syncthreads();                 // this stage has landed for everybody, and the slot of the last one is free
      issue(step + NS - 1);
      if (mine) {
        const float* kst = s_ring + step % NS * Shape::kStageFloats + jc;
        const float* qst = s_pq + s * KC * R + rg * RT;
#pragma unroll
        for (int cc = 0; cc < KC; ++cc) {
          uint64_t q2[kPairs];
          if constexpr (RT >= 4) {
#pragma unroll
            for (int g = 0; g < RT / 4; ++g) {
              const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(qst + cc * R + 4 * g);   // rows (4g, 4g+1), (4g+2, 4g+3)
              q2[2 * g] = t.x;
              q2[2 * g + 1] = t.y;
            }
          } else {
            q2[0] = *reinterpret_cast<const uint64_t*>(qst + cc * R);
          }
          const float4 kv = *reinterpret_cast<const float4*>(kst + cc * JT);
          const uint64_t k2[4] = {pack_f32x2(kv.x, kv.x), pack_f32x2(kv.y, kv.y), pack_f32x2(kv.z, kv.z),
                                  pack_f32x2(kv.w, kv.w)};
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int r = 0; r < kPairs; ++r) acc[u][r] = ffma2(q2[r], k2[u], acc[u][r]);
        }
      }
    }
    if (j0 + jc < nbp) {
      store_keys<kPairs>(acc, s_key + (int64_t)(rg * RT) * nbp + j0 + jc, nbp);
    }
  }
  __syncthreads();

  select_tile<WINDOW, 8, (R >= 16 ? 2 : 1), 8>(s_key, nb, nbp, topk, bh, i0, nrows, N, blk_size, frame_tokens, window, kept_idx, kept_cnt);
}

// The same for long rows of key blocks: a CTA of WARPS warps takes R query blocks, a thread owns an RT x 4 register tile
// and reads its own pooled K columns straight from L2 (two batches of 4 channels in flight), so that a warp never
// waits for another one until the scores are complete.  Bound by the FMA pipe and, in the selection, by latency: what
// helps both is warps, so the tile is 8 x 4 (96 registers, two CTAs of ten warps per SM) although 16 x 4 needs fewer
// shared loads per FMA.  40 heads of 591 blocks: 126 us (16 x 4 with five warps, three CTAs: 121; with one row searched
// bit by bit at a time, as it was: 147); of 1182: 439 us (484; 596).  The FMAs alone are 50 and 200 us.
template <int D, int R, int RT, int WARPS, int CTAS, bool WINDOW>
__global__ void __launch_bounds__(WARPS * 32, CTAS)
topk_wide_kernel(const float* pq, const float* pkT, int32_t* __restrict__ kept_idx,
                 int32_t* __restrict__ kept_cnt, int nb, int nbp, int topk, int groups_per_bh, int N, int blk_size,
                 int frame_tokens, int window, int32_t* __restrict__ header) {
  constexpr int kThreads = WARPS * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* s_pq = reinterpret_cast<float*>(smem_raw);                   // [D][R], see topk_kernel
  uint32_t* s_key = reinterpret_cast<uint32_t*>(s_pq + R * D);        // [R][nbp]
  const int64_t bh = blockIdx.x / groups_per_bh;
  const int i0 = (blockIdx.x % groups_per_bh) * R;
  const int nrows = min(R, nb - i0);

  pdl_wait();
  clear_header(header);
  for (int e = threadIdx.x; e < R * (D / 4); e += kThreads) {
    const int r = e % R, c = e / R * 4;
    const float4 x = r < nrows ? *reinterpret_cast<const float4*>(pq + (bh * nb + i0 + r) * D + c)
                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    s_pq[c * R + r] = x.x; s_pq[(c + 1) * R + r] = x.y; s_pq[(c + 2) * R + r] = x.z; s_pq[(c + 3) * R + r] = x.w;
  }
  __syncthreads();
  const float* kcol = pkT + bh * D * (int64_t)nbp;
  const ulonglong2* s_pq2 = reinterpret_cast<const ulonglong2*>(s_pq);       // [D][R / 4]
  constexpr int RG = R / RT, kPairs = RT / 2;
  constexpr int kCB = 4;   // channels per batch of loads
  const int rg = (threadIdx.x >> 5) % RG;
  for (int j0 = (threadIdx.x / (32 * RG) * 32 + (threadIdx.x & 31)) * 4; j0 < nb; j0 += kThreads / RG * 4) {
    uint64_t acc[4][kPairs];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int r = 0; r < kPairs; ++r) acc[u][r] = pack_f32x2(0.0f, 0.0f);
    const float* kp = kcol + j0;
    auto load_batch = [&](float4 (&kv)[kCB], int c0) {
#pragma unroll
      for (int cc = 0; cc < kCB; ++cc) kv[cc] = *reinterpret_cast<const float4*>(kp + (int64_t)(c0 + cc) * nbp);
    };
    auto fma_batch = [&](const float4 (&kv)[kCB], int c0) {
#pragma unroll
      for (int cc = 0; cc < kCB; ++cc) {
        uint64_t q2[kPairs];
#pragma unroll
        for (int g = 0; g < RT / 4; ++g) {
          const ulonglong2 t = s_pq2[(c0 + cc) * (R / 4) + rg * (RT / 4) + g];   // rows (4g, 4g+1), (4g+2, 4g+3)
          q2[2 * g] = t.x;
          q2[2 * g + 1] = t.y;
        }
        const uint64_t k2[4] = {pack_f32x2(kv[cc].x, kv[cc].x), pack_f32x2(kv[cc].y, kv[cc].y),
                                pack_f32x2(kv[cc].z, kv[cc].z), pack_f32x2(kv[cc].w, kv[cc].w)};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int r = 0; r < kPairs; ++r) acc[u][r] = ffma2(q2[r], k2[u], acc[u][r]);
      }
    };
    float4 kva[kCB], kvb[kCB];
    load_batch(kva, 0);
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 2 * kCB) {
      load_batch(kvb, c0 + kCB);
      fma_batch(kva, c0);
      if (c0 + 2 * kCB < D) load_batch(kva, c0 + 2 * kCB);
      fma_batch(kvb, c0 + kCB);
    }
    store_keys<kPairs>(acc, s_key + (int64_t)(rg * RT) * nbp + j0, nbp);
  }
  __syncthreads();
  select_tile<WINDOW, WARPS, 1, 0>(s_key, nb, nbp, topk, bh, i0, nrows, N, blk_size, frame_tokens, window, kept_idx, kept_cnt);
}

// Up to 64 key blocks: latency is all there is.  The pooled K of the (batch, head) comes into shared memory in one go, not
// through a ring, a warp takes a query block, a lane one or two key blocks (lane, lane + 32) with their chains in registers,
// and the selection holds one or two keys per lane instead of eight.  38 KB of shared memory at most, so that its CTAs are
// on the SMs while the pooling kernel drains.  Whole selection against topk_kernel, us, d = 128: 3 heads of 10 blocks 8.3 -> 5.6, 8 of 25 9.9 ->
// 7.1, 6 of 51 11.5 -> 9.4, 20 of 51 17.5 -> 15.4, 40 of 51 34.4 -> 28.4, 80 of 64 71.5 -> 62.6; d = 64: 3 of 10 6.4 -> 5.1, 6 of 51 6.9 -> 5.8, 40 of 33
// 10.8 -> 9.1, 40 of 51 15.0 -> 10.8, 80 of 64 26.7 -> 21.4.  The same for up to 128 blocks (72 KB): 6 of 94 15.8 -> 19.1.  Two query blocks per
// warp: 6 of 51 21.4.
template <int D, int KPL, bool WINDOW>
__global__ void __launch_bounds__(kTopkThreads)
topk_small_kernel(const float* pq, const float* pkT, int32_t* __restrict__ kept_idx, int32_t* __restrict__ kept_cnt, int nb, int nbp,
                  int topk, int groups_per_bh, int N, int blk_size, int frame_tokens, int window, int32_t* __restrict__ header) {
  constexpr int W = 32 * KPL, R = kTopkThreads / 32;                  // nbp = W
  __shared__ __align__(16) float s_k[D * W];                          // [D][W]
  __shared__ __align__(16) float s_q[R * D];                          // [R][D]
  __shared__ uint32_t s_key[R * W];                                   // [R][W]
  const int64_t bh = blockIdx.x / groups_per_bh;
  const int i0 = (blockIdx.x % groups_per_bh) * R;
  const int nrows = min(R, nb - i0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* kcol = pkT + bh * D * (int64_t)W;
  const float* qrow = pq + (bh * nb + i0) * D;
  pdl_wait();
  clear_header(header);
  for (int e = threadIdx.x; e < D * W / 4; e += kTopkThreads) cp_async16(smem_u32(s_k + 4 * e), kcol + 4 * e);
  for (int e = threadIdx.x; e < nrows * (D / 4); e += kTopkThreads) cp_async16(smem_u32(s_q + 4 * e), qrow + 4 * e);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  if (warp < nrows) {
    float acc[KPL] = {};
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      const float4 q = *reinterpret_cast<const float4*>(s_q + warp * D + c);
#pragma unroll
      for (int u = 0; u < KPL; ++u) {                                 // each its own chain, channels in ascending order
        const float* k = s_k + c * W + 32 * u + lane;
        acc[u] = fmaf(q.x, k[0], acc[u]);
        acc[u] = fmaf(q.y, k[W], acc[u]);
        acc[u] = fmaf(q.z, k[2 * W], acc[u]);
        acc[u] = fmaf(q.w, k[3 * W], acc[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < KPL; ++u) s_key[warp * W + 32 * u + lane] = score_key(acc[u]);
  }
  __syncwarp();                        // (a warp reads the keys of its own row)
  select_tile<WINDOW, R, 1, KPL>(s_key, nb, W, topk, bh, i0, nrows, N, blk_size, frame_tokens, window, kept_idx, kept_cnt);
}

// topk = nb: every candidate is kept whatever its score, so nothing is pooled and nothing compared.  A warp per list.
// (Pooled and scored all the same, and then listed: attention over all blocks, 6 heads of 6,479 tokens, 150.2 us, now 143.0;
// 3 heads in a causal window of three frames 36.2, now 31.1.)
constexpr int kAllWarps = 8;
__global__ void __launch_bounds__(kAllWarps * 32)
list_all_kernel(int32_t* __restrict__ kept_idx, int32_t* __restrict__ kept_cnt, int64_t lists, int nb, int N, int blk_size,
                int frame_tokens, int window, int32_t* __restrict__ header) {
  pdl_wait();
  clear_header(header);
  const int lane = threadIdx.x & 31;
  for (int64_t w = (int64_t)blockIdx.x * kAllWarps + (threadIdx.x >> 5); w < lists; w += (int64_t)gridDim.x * kAllWarps) {
    int jlo = 0, jhi = nb - 1;
    if (frame_tokens > 0) window_range((int)(w % nb), N, blk_size, frame_tokens, window, jlo, jhi);
    int32_t* dst = kept_idx + w * nb;
    for (int t = lane; t < nb; t += 32) dst[t] = jlo + t <= jhi ? jlo + t : -1;
    if (lane == 0 && kept_cnt != nullptr) kept_cnt[w] = jhi - jlo + 1;
  }
}

// The kernels of a selection stand by while the one before them drains, so they have to agree on how an SM's memory is split between
// L1 and shared memory.  Left to itself the runtime picks a split for each kernel, and a CTA that needs another one waits until
// the SM is empty.  Selection with the runtime's splits / with the most shared memory for all, us: 3 heads of 192 blocks 18.8 /
// 15.2, 6 of 94 15.6 / 13.8, 35 of 48 29.0 / 25.0, 40 of 48 31.8 / 27.8, elsewhere the same.  A preference of the kernel, told once per device.
template <auto Kern>
static bool max_shared_memory() {
  static std::atomic<uint64_t> told{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const uint64_t bit = 1ull << (dev & 63);
  if (told.load(std::memory_order_relaxed) & bit) return true;
  if (cudaFuncSetAttribute(Kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess) return false;
  if (dev < 64) told.fetch_or(bit, std::memory_order_relaxed);
  return true;
}

// The limit of a kernel's dynamic shared memory belongs to the kernel, not to a launch: it is always set to the most that any
// launch of the kernel asks for.  Set to what this launch needs, it could be lowered by another thread before the
// launch, which then fails.
constexpr int kSmemOfOne = 227 * 1024, kSmemOfTwo = 113 * 1024;      // of a CTA alone on its SM, and of one of two

template <int D, int RT, int RG, int KC, int NS>
static int launch_topk(const float* pq, const float* pkT, int32_t* kept_idx, int32_t* kept_cnt, int nb, int nbp, int topk,
                       int64_t bh, int N, int block, int frame_tokens, int window, int32_t* header, cudaStream_t stream) {
  using Shape = TopkShape<RT, RG, KC, NS>;
  const int groups = (nb + Shape::kRows - 1) / Shape::kRows;
  const int64_t ctas = bh * groups;
  if (ctas > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const size_t smem = Shape::smem_bytes(D, nbp);
  auto kern = frame_tokens > 0 ? topk_kernel<D, RT, RG, KC, NS, true> : topk_kernel<D, RT, RG, KC, NS, false>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Shape::smem_bytes(D, 256)) != cudaSuccess ||
      !(frame_tokens > 0 ? max_shared_memory<topk_kernel<D, RT, RG, KC, NS, true>>() : max_shared_memory<topk_kernel<D, RT, RG, KC, NS, false>>()))
    return SPARKATTN_E_CUDA;
  return launch_kernel(kern, (unsigned)ctas, kTopkThreads, smem, true, stream, pq, pkT, kept_idx, kept_cnt, nb, nbp, topk,
                       groups, N, block, frame_tokens, window, header);
}

template <int D, int KPL>
static int launch_topk_small(const float* pq, const float* pkT, int32_t* kept_idx, int32_t* kept_cnt, int nb, int nbp, int topk,
                             int64_t bh, int N, int block, int frame_tokens, int window, int32_t* header, cudaStream_t stream) {
  constexpr int R = kTopkThreads / 32;
  const int groups = (nb + R - 1) / R;
  const int64_t ctas = bh * groups;
  if (ctas > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  auto kern = frame_tokens > 0 ? topk_small_kernel<D, KPL, true> : topk_small_kernel<D, KPL, false>;
  if (!(frame_tokens > 0 ? max_shared_memory<topk_small_kernel<D, KPL, true>>() : max_shared_memory<topk_small_kernel<D, KPL, false>>()))
    return SPARKATTN_E_CUDA;
  return launch_kernel(kern, (unsigned)ctas, kTopkThreads, 0, true, stream, pq, pkT, kept_idx, kept_cnt, nb, nbp, topk, groups, N, block,
                       frame_tokens, window, header);
}

static size_t wide_smem(int rows, int d, int nbp) { return (size_t)rows * (d + nbp) * sizeof(float); }

template <int D, int R, int RT, int WARPS, int CTAS>
static int launch_topk_wide(const float* pq, const float* pkT, int32_t* kept_idx, int32_t* kept_cnt, int nb, int nbp, int topk,
                            int64_t bh, int N, int block, int frame_tokens, int window, int32_t* header, cudaStream_t stream) {
  const int groups = (nb + R - 1) / R;
  const int64_t ctas = bh * groups;
  if (ctas > 0x7fffffffLL) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const size_t smem = wide_smem(R, D, nbp);
  auto kern = frame_tokens > 0 ? topk_wide_kernel<D, R, RT, WARPS, CTAS, true> : topk_wide_kernel<D, R, RT, WARPS, CTAS, false>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CTAS == 2 && R == 16 ? kSmemOfTwo : kSmemOfOne) != cudaSuccess ||
      !(frame_tokens > 0 ? max_shared_memory<topk_wide_kernel<D, R, RT, WARPS, CTAS, true>>()
                         : max_shared_memory<topk_wide_kernel<D, R, RT, WARPS, CTAS, false>>()))
    return SPARKATTN_E_CUDA;
  return launch_kernel(kern, (unsigned)ctas, WARPS * 32, smem, true, stream, pq, pkT, kept_idx, kept_cnt, nb, nbp, topk,
                       groups, N, block, frame_tokens, window, header);
}

// Where the pooled means live in a selection workspace: pooled Q [B*H][nb][d] right behind the header, pooled K
// transposed [B*H][d][nbp] behind it.
float* select_pooled_ptr(const sparkattn_shape_t& s, void* workspace, bool key_side) {
  const int nb = (s.N + s.block - 1) / s.block;
  float* pq = reinterpret_cast<float*>(static_cast<char*>(workspace) + kWorkspaceHeaderBytes);
  return key_side ? pq + (int64_t)s.B * s.H * nb * s.d : pq;
}

// scores + top-k on pooled means that are, or by the launch before will be, in the workspace (header: to be cleared, or NULL)
template <int D>
static int launch_topk_d(const sparkattn_shape_t& s, int topk, int frame_tokens, int window, int32_t* kept_idx,
                         int32_t* kept_cnt, void* workspace, int32_t* header, cudaStream_t stream) {
  const int nb = (s.N + s.block - 1) / s.block;
  const int nbp = round_up(nb, 32);
  const int64_t bh = (int64_t)s.B * s.H;
  const float* pq = select_pooled_ptr(s, workspace, false);
  const float* pkT = select_pooled_ptr(s, workspace, true);
  auto go = [&](auto launch) {
    return launch(pq, pkT, kept_idx, kept_cnt, nb, nbp, topk, bh, s.N, s.block, frame_tokens, window, header, stream);
  };
  constexpr int kNumSMs = 148;   // B200; another count only moves the points where the CTAs get smaller
  const int64_t ctas32 = bh * ((nb + 31) / 32), ctas16 = bh * ((nb + 15) / 16);
  // More than 256 key blocks: the wide kernel, with 8 rows while 16 would leave SMs idle or do not fit twice into an SM,
  // else 16.  8 against 16 rows, whole selection (pooling included), d = 128: 1 head of 260 / 591 / 1182 blocks of 128
  // 16.5 / 23.5 / 35 us against 21.1 / 26.7 / 71, 4 of 591 (148 CTAs of 16) 47.6 against 52.6, 3 of 1000 (189) 69 against 82,
  // but 12 of 257 (204) 64.7 against 57.3, 12 of 591 132 against 127, 40 of 591 425 against 389; d = 64: 1 of 260 / 591 10.6 /
  // 13.6 against 14.0 / 17.1, 4 of 591 22.0 against 25.9, 12 of 257 26.7 against 25.9, 40 of 591 197 against 178.  The other
  // kernel on these rows: d = 128 1 head of 260 / 591 15.9 / 33.5, 12 of 257 / 591 59.9 / 154, 40 of 591 463; d = 64 1 of 260 /
  // 591 10.1 / 14.4, 12 of 257 / 591 26.8 / 80, 40 of 591 232.  Up to 256 blocks: the other one (its column split leaves
  // no warp idle there; wide with 16 rows: 1 / 12 / 40 heads of 256 20.6 / 54 / 158 against 12.8 / 51 / 143, d = 64 14.7 / 23.9 /
  // 65 against 9.1 / 20.8 / 59), with as many rows per CTA as still leave 1.5 CTAs (32 rows) or one CTA (16) per SM:
  // 80 heads of 250 blocks 63.9 us with 32 rows, 69.9 with 16, 94.6 with 8; 12 heads of 256 22.0 / 20.8 / 22.2; 3 heads
  // of 100 19.8 / 14.3 / 11.5.  Up to 64 blocks: the small kernel, which has both sides.
  if (nb <= kSmallBlocks) return nbp == 32 ? go(launch_topk_small<D, 1>) : go(launch_topk_small<D, 2>);
  if (nb > 256) {
    if (ctas16 > kNumSMs && wide_smem(16, D, nbp) <= kSmemOfTwo) return go(launch_topk_wide<D, 16, 8, 10, 2>);
    return go(launch_topk_wide<D, 8, 8, 10, 2>);               // at most 132 KB
  }
  static_assert(TopkShape<8, 4, 16, 4>::smem_bytes(D, 256) <= kSmemOfOne, "the tile of 32 rows of 256 keys");
  if (2 * ctas32 >= 3 * kNumSMs) return go(launch_topk<D, 8, 4, 16, 4>);
  if (ctas16 >= kNumSMs) return go(launch_topk<D, 4, 4, 16, 4>);
  return go(launch_topk<D, 2, 4, 16, 4>);
}

static int launch_list_all(const sparkattn_shape_t& s, int frame_tokens, int window, int32_t* kept_idx, int32_t* kept_cnt, int32_t* header,
                           cudaStream_t stream) {
  const int nb = (s.N + s.block - 1) / s.block;
  const int64_t lists = (int64_t)s.B * s.H * nb, ctas = (lists + kAllWarps - 1) / kAllWarps;
  return launch_kernel(list_all_kernel, (unsigned)(ctas < 4096 ? ctas : 4096), kAllWarps * 32, 0, true, stream, kept_idx, kept_cnt, lists, nb,
                       s.N, s.block, frame_tokens, window, header);
}

static int launch_topk_any(const sparkattn_shape_t& s, int topk, int frame_tokens, int window, int32_t* kept_idx,
                           int32_t* kept_cnt, void* workspace, int32_t* header, cudaStream_t stream) {
  if (s.d == 128) return launch_topk_d<128>(s, topk, frame_tokens, window, kept_idx, kept_cnt, workspace, header, stream);
  if (s.d == 64) return launch_topk_d<64>(s, topk, frame_tokens, window, kept_idx, kept_cnt, workspace, header, stream);
  return SPARKATTN_E_UNSUPPORTED_SHAPE;
}

int launch_select_pooled(const sparkattn_shape_t& s, int topk, int32_t* kept_idx, int32_t* kept_cnt, void* workspace,
                         cudaStream_t stream) {
  const int nb = (s.N + s.block - 1) / s.block;
  if (nb > kSelectMaxBlocks) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  if (s.d != 128 && s.d != 64) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  if (topk >= nb) return launch_list_all(s, 0, 0, kept_idx, kept_cnt, static_cast<int32_t*>(workspace), stream);
  const int rc = launch_topk_any(s, topk, 0, 0, kept_idx, kept_cnt, workspace, static_cast<int32_t*>(workspace), stream);
  if (rc != SPARKATTN_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? SPARKATTN_OK : SPARKATTN_E_CUDA;
}

int launch_select(const sparkattn_shape_t& s, const void* q, const void* k, int topk, int frame_tokens, int window,
                  const int32_t* block_valid, int32_t* kept_idx, int32_t* kept_cnt, void* workspace, cudaStream_t stream) {
  const int nb = (s.N + s.block - 1) / s.block;
  const int nbp = round_up(nb, 32);
  if (nb > kSelectMaxBlocks) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  const int64_t n_items = (int64_t)s.B * s.H * nb;
  float* pq = select_pooled_ptr(s, workspace, false);
  float* pkT = select_pooled_ptr(s, workspace, true);
  const __nv_bfloat16* qb = static_cast<const __nv_bfloat16*>(q);
  const __nv_bfloat16* kb = static_cast<const __nv_bfloat16*>(k);
  if (s.d != 128 && s.d != 64) return SPARKATTN_E_UNSUPPORTED_SHAPE;
  if (topk >= nb) return launch_list_all(s, frame_tokens, window, kept_idx, kept_cnt, static_cast<int32_t*>(workspace), stream);
  const int sm_count = current_sm_count();
  if (sm_count < 1) return SPARKATTN_E_CUDA;
  const size_t pool_smem = (size_t)2 * s.block * s.d * 2;
  auto pool = s.d == 128 ? pool_kernel<128> : pool_kernel<64>;
  if (cudaFuncSetAttribute(pool, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 128 * s.d * 2) != cudaSuccess)    // (see kSmemOfOne)
    return SPARKATTN_E_CUDA;
  if (!(s.d == 128 ? max_shared_memory<pool_kernel<128>>() : max_shared_memory<pool_kernel<64>>())) return SPARKATTN_E_CUDA;
  const int64_t resident = (int64_t)sm_count * kPoolCtasPerSm * (65536 / (int)pool_smem);
  const int64_t pool_ctas = 2 * n_items < resident ? 2 * n_items : resident;
  // Launched early while a CTA has fewer than four blocks.  Beyond that the microsecond it saves is lost in the noise (256 blocks of 12
  // heads 50.8 us either way), and behind a kernel that lets it in its CTAs are placed unevenly for their whole run (see pdl_wait):
  // comp_state then select, 12 heads of 32,760 tokens 92.5 us let in, 88.4 not; 40 of 75,600 675 and 620.  Below the line it
  // would be 0.2 us of a selection of 12 to 17 us, and that order of calls stays slower there (2 heads of 12,000 26.5 us, 24.2 if not let in).
  const bool early = 2 * n_items < 4 * resident;
  const int rc0 = launch_kernel(pool, (unsigned)pool_ctas, s.d / 2, pool_smem, early, stream, qb, kb, pq, pkT, s.H, s.N, s.block, nb,
                                nbp, s.stride_b, s.stride_h, s.stride_n, n_items, block_valid, static_cast<int32_t*>(workspace));
  if (rc0 != SPARKATTN_OK) return rc0;
  const int rc = launch_topk_any(s, topk, frame_tokens, window, kept_idx, kept_cnt, workspace, nullptr, stream);
  if (rc != SPARKATTN_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? SPARKATTN_OK : SPARKATTN_E_CUDA;
}

}  // namespace sparkattn
