// Test-only kernels (built by tests/test_gpu_timeout.py, not part of the library): they call the library's two
// bounded barrier waits on an mbarrier that nothing ever arrives at, with a limit of about a millisecond
// instead of the library's default.  The wait runs out, SPARKATTN_E_DEVICE_TIMEOUT and the wait id end up in
// the status words of the workspace, and the kernel returns normally: no trap, no fault, nothing left
// spinning.
#include "../../paper_2609_23153_b200/csrc/common.cuh"
#include "../../paper_2609_23153_b200/csrc/launch.h"

using namespace sparkattn;

__global__ void timeout_probe_kernel(int32_t* status, unsigned long long limit_ns, int wait_id) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0, &abort_flag, status, wait_id, limit_ns);
  // word 2: threads whose wait gave up; word 3: threads that (wrongly) saw the barrier flip
  atomicAdd(status + (ok ? 3 : 2), 1);
}

// The wait of the pipelined kernels: two warps wait, the second with four times the limit, so it leaves because the first
// one has given up; then a second expiry is recorded, which must not replace the first.
__global__ void pipe_timeout_probe_kernel(int32_t* status, unsigned limit_ns, int wait_id) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  const bool ok = pipe_wait(&bar, 0, &abort_flag, wait_id + warp, limit_ns << (2 * warp));
  atomicAdd(status + (ok ? 3 : 2), 1);
  __syncthreads();
  if (threadIdx.x == 32) abort_timeout(&abort_flag, wait_id + 1);
  __syncthreads();
  if (threadIdx.x == 0) report_abort(status, abort_flag);
}

extern "C" int timeout_probe(void* workspace, unsigned long long limit_ns, int wait_id, int pipelined, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(workspace, 0, kWorkspaceHeaderBytes, s) != cudaSuccess) return -1;
  int32_t* status = static_cast<int32_t*>(workspace);
  if (pipelined) pipe_timeout_probe_kernel<<<1, 64, 0, s>>>(status, (unsigned)limit_ns, wait_id);
  else timeout_probe_kernel<<<1, 32, 0, s>>>(status, limit_ns, wait_id);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// The status header of a kernel that clears it itself: the first of two CTAs takes the header and looks the two lists up again
// when a code was in it, the second reports the bad index of its list, if it has one.  Whichever is not `early` begins some
// milliseconds late (neither waits for the other).
__global__ void header_probe_kernel(int32_t* status, const int32_t* lists, int nb, int kmax, int early) {
  if ((int)blockIdx.x != early)
    for (int i = 0; i < 5000; ++i) __nanosleep(1000);
  if (blockIdx.x == 0) {
    bool code_there = false;
    if (threadIdx.x == 0) code_there = take_header(status);
    if (__syncthreads_or(code_there)) recheck_lists(lists, nullptr, 2, nb, kmax, status, threadIdx.x, 64);
  } else if (threadIdx.x < kmax) {
    const int32_t kb = lists[kmax + threadIdx.x];
    if (kb < 0 || kb >= nb) report_early(status, SPARKATTN_E_BAD_INDEX, kb);
  }
}

extern "C" int header_probe(void* workspace, const void* lists, int nb, int kmax, int early, void* stream) {
  header_probe_kernel<<<2, 64, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<int32_t*>(workspace), static_cast<const int32_t*>(lists), nb,
                                                                      kmax, early);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// A launch without blocks, which the runtime refuses on the host, through the library's launch helper.  Bit 0: the helper
// did not report it; bit 1: the runtime still holds the error.
__global__ void never_run_kernel(int) {}

extern "C" int launch_probe(int overlap) {
  const int rc = launch_kernel(never_run_kernel, 0, 32, 0, overlap != 0, nullptr, 1);
  return (rc != SPARKATTN_E_CUDA ? 1 : 0) | (cudaGetLastError() != cudaSuccess ? 2 : 0);
}
