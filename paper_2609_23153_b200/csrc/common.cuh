// Shared device helpers for the sparkattn kernels (sm_100a only): mbarrier,
// TMA and tcgen05 wrappers in inline PTX, plus the device status word.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sparkattn.h"

namespace sparkattn {

// Layout of the 256-byte header at the start of every workspace.
//   word 0: device status (0 = OK, else a negative sparkattn_status)
//   word 1: detail (offending index, or an id of the wait that expired)
constexpr int kWorkspaceHeaderBytes = 256;

__device__ __forceinline__ void report_status(int32_t* status, int code, int detail) {
  if (atomicCAS(status, 0, code) == 0) status[1] = detail;
}

// Every call starts with a clean status, in memory of any content.  A small kernel in front can see to it (report_status above
// relies on that), or the kernel does it itself: its first CTA takes the two words in one exchange.  CTAs run in no order, so
// a report may come before that, and nobody waits to find out: report_early puts its code over everything but
// another code, and a first CTA that has taken a code, which may be one of this launch or what an earlier call left, looks
// through all of the call's indices itself (recheck_lists; the gather has its own) and reports again what it finds.  A bad index
// is reported whatever the order; it costs what the CTAs that hold it need for an atomic each, and the next call on
// that workspace the first CTA's look.  (A wait that runs out can't be looked up again.  It is reported two seconds after
// its CTA began, and lost only if the first CTA begins later than that.)  Having waited for the first CTA, for a millisecond
// where it could have begun before, cost one bad index among the 75,600 of 40 heads 1,256 us instead of 235.
__device__ __forceinline__ bool is_status_code(unsigned long long header) {
  const int32_t code = (int32_t)(uint32_t)header;
  return code < 0 && code >= SPARKATTN_E_NO_DEVICE;
}
__device__ __forceinline__ bool take_header(int32_t* status) {
  return is_status_code(atomicExch(reinterpret_cast<unsigned long long*>(status), 0ull));
}
__device__ __forceinline__ void report_early(int32_t* status, int code, int detail) {
  unsigned long long* header = reinterpret_cast<unsigned long long*>(status);
  const unsigned long long mine = (unsigned long long)(uint32_t)detail << 32 | (uint32_t)code;
  const unsigned long long found = atomicCAS(header, 0ull, mine);
  if (found != 0 && !is_status_code(found)) atomicExch(header, mine);      // (nothing of this launch, unless the first CTA came in between)
}
// Thread `thread` of the `threads` of the first CTA that look the kept lists up again, up to 2048 entries of a few thousand lists;
// each reports one bad index.  All entries are asked for eight at a time, those behind a list's count as well, and only one that is out of
// range is looked at closely: 2040 lists of 10 add 30 us to the call (list by list 125).  (Behind everything else in the kernel: in front of the tile
// loops, 40 heads of 75,600 tokens took 2974 us instead of 2954, 64-token blocks 3408 and 3344.)
__device__ __forceinline__ void recheck_lists(const int32_t* kept_idx, const int32_t* kept_cnt, int lists, int nb, int kmax, int32_t* status,
                                              int thread, int threads) {
  const uint32_t n = (uint32_t)lists * (uint32_t)kmax;
#pragma unroll 1
  for (uint32_t first = thread; first < n; first += 8 * threads) {
    bool odd = false;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t e = first + u * threads;
      odd = odd || (uint32_t)(e < n ? kept_idx[e] : 0) >= (uint32_t)nb;
    }
    if (!odd) continue;
#pragma unroll 1
    for (uint32_t e = first; e < n && e < first + 8 * threads; e += threads) {
      const int kb = kept_idx[e], list = (int)(e / (uint32_t)kmax), at = (int)(e - (uint32_t)list * (uint32_t)kmax);
      if ((uint32_t)kb < (uint32_t)nb || at >= (kept_cnt ? kept_cnt[list] : kmax)) continue;
      report_early(status, SPARKATTN_E_BAD_INDEX, kb);
      return;
    }
  }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Non-blocking test of a phase (never suspends the thread): for loops that poll several barriers.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: polls the barrier until it flips, another thread of the CTA
// raises `abort_flag`, or `limit_ns` (kWaitLimitNs unless the caller says
// otherwise) of wall time have passed (checked every 64 polls).  On expiry it
// raises the flag, records a timeout and `wait_id` in the status words and
// returns false; callers then leave their role loop.
constexpr uint64_t kWaitLimitNs = 2000000000ull;
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          int32_t* status, int wait_id, uint64_t limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 0u) {
      if (*abort_flag) return false;
      if (global_timer_ns() - t0 > limit_ns) break;
    }
  }
  *abort_flag = 1;
  report_status(status, SPARKATTN_E_DEVICE_TIMEOUT, wait_id);
  return false;
}

// mbar_wait in the shortest form, for a kernel with some twenty waits whose code does not fit the SM's instruction cache
// as it is.  The limit is the same; on expiry only the wait's id goes to the abort flag (the first one stays), and
// report_abort takes it to the status words when the CTA winds down.
constexpr int kAbortTimeout = 256;
__device__ __forceinline__ uint32_t global_timer_lo() {
  uint32_t t;
  asm volatile("mov.u32 %0, %%globaltimer_lo;" : "=r"(t));
  return t;
}
__device__ __forceinline__ void abort_timeout(volatile int* abort_flag, int wait_id) {
  atomicCAS(const_cast<int*>(abort_flag), 0, kAbortTimeout + wait_id);
}
__device__ __forceinline__ bool pipe_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int wait_id,
                                          uint32_t limit_ns = (uint32_t)kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  static_assert(kWaitLimitNs < 0xf0000000ull, "the limit is counted in 32 bits");
  const uint32_t t0 = global_timer_lo();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 0u) {
      if (*abort_flag) return false;
      if (global_timer_lo() - t0 > limit_ns) {
        abort_timeout(abort_flag, wait_id);
        return false;
      }
    }
  }
}
__device__ __forceinline__ void report_abort(int32_t* status, int abort_flag) {
  if (abort_flag >= kAbortTimeout) report_early(status, SPARKATTN_E_DEVICE_TIMEOUT, abort_flag - kAbortTimeout);
}

// Asynchronous 16-byte copies global -> shared (both sides 16-byte aligned) and their groups.
__device__ __forceinline__ void cp_async16(uint32_t smem_dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Programmatic dependent launch.  A kernel that may be launched while the one before it on the stream is still
// running (launch_kernel with overlap) calls pdl_wait before its first access to device memory: it returns when
// everything earlier on the stream is complete and visible.  pdl_trigger lets the next such kernel be launched.  The last
// kernel of a call has none unless the call's purpose says what comes next, because of the selection's pooling kernel: two
// persistent CTAs per SM with their blocks dealt out beforehand, which come to stand three deep on some SMs and alone on
// others when they are let in while SMs become free one by one.  comp_apply then select, 40 heads of 75,600 tokens: 880 us
// with a trigger at the start of the apply pass, 837 without; three quant_fp8 then select, 444 64-token blocks 24.1 and 20.9, 40 heads
// of 75,600 999 and 947.  The two exceptions are the pooling quantisation (quant.cu) and the state pass, whose state comp_apply
// or fwd_gated takes next: selection, state and gated forward of 10 heads of 7,252 tokens 174 us with its trigger, 184 without;
// state and apply of 3 heads of 1,200 18.2 and 19.2.  (launch_select has what that leaves for the pooling kernel to do.)
// A kernel launched early reads device memory with ordinary loads only: a read-only load (__ldg, or through a const __restrict__
// parameter) is for data that nothing writes during the whole life of the kernel, and the compiler may move it ahead of
// the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// --------------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_prefetch_desc(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
// 4-D tiled load global -> shared of this CTA, completion on an mbarrier.
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const void* tmap, uint64_t* bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1),
      "r"(c2), "r"(c3)
      : "memory");
}

// ----------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_result, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_result)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// All tcgen05.mma issued so far by this thread arrive on `bar` when complete.
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor for a 128-byte-swizzled tile whose rows are
// 128 bytes long and whose 8-row groups are 1024 bytes apart (the layout a TMA
// load with CU_TENSOR_MAP_SWIZZLE_128B produces for a box that is 128 bytes
// wide).  `lbo_bytes` is only read for MN-major operands wider than one
// 128-byte atom (distance between two 64-element column slabs).
__device__ __forceinline__ uint64_t make_smem_desc_sw128(uint32_t smem_addr, uint32_t lbo_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);          // start address, bits [0,14)
  d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;     // leading byte offset, bits [16,30)
  d |= static_cast<uint64_t>((1024u >> 4) & 0x3FFFu) << 32;         // stride byte offset, bits [32,46)
  d |= static_cast<uint64_t>(1) << 46;                              // descriptor version (Blackwell)
  d |= static_cast<uint64_t>(2) << 61;                              // layout type: SWIZZLE_128B
  return d;
}

// A descriptor from its two 32-bit words (the low word carries the start address and LBO).
__device__ __forceinline__ uint64_t make_desc(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}

// Instruction descriptor, dense, fp32 accumulate.  fmt: 0 = f16 / e4m3 (by
// kind), 1 = bf16 / e5m2.  b_mn_major: B operand stored with N contiguous.
__host__ __device__ constexpr uint32_t make_idesc(uint32_t fmt, uint32_t M, uint32_t N, bool b_mn_major) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((N >> 3) << 17) |
         ((M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]
template <bool kFp8>
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  if constexpr (kFp8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
// D[tmem] (+)= A[tmem] * B[smem]
template <bool kFp8>
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  if constexpr (kFp8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane
// (taddr.lane + i), registers r[0..31] = columns taddr.col .. +31.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// the same for 16 columns
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}

// Packed fp32x2 arithmetic (one issue slot for two lanes of a row).
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack_f32x2(uint64_t v) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
  return d;
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Register re-balancing between warpgroups (all warps of a warpgroup execute it).
template <int N>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace sparkattn
