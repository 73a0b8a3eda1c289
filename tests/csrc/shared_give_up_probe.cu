// Test-only kernel for the wait that the warps of a block give up together (warp_wait
// in dmc_internal.cuh). The test builds it with a shortened DMC_WAIT_LIMIT_NS. Warp w
// waits on barrier w, which has its one arrival already if bit w of `arrived` is set,
// and then on a barrier that nobody arrives at. No tensor-core work or copy runs.
#include "dmc_internal.cuh"

constexpr int kMaxWarps = 12;

__global__ void shared_give_up_kernel(unsigned arrived, unsigned int* err, int* first, int* second,
                                      unsigned long long* ns) {
  __shared__ __align__(8) uint64_t bars[kMaxWarps + 1];
  __shared__ int abort_word;
  const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  if (threadIdx.x == 0) {
    for (int i = 0; i <= warps; ++i) dmc::mbar_init(dmc::smem_u32(&bars[i]), 1);
    dmc::fence_mbar_init();
    abort_word = 0;
  }
  __syncthreads();
  if (threadIdx.x < (unsigned)warps && (arrived >> threadIdx.x & 1u)) dmc::mbar_arrive(dmc::smem_u32(&bars[threadIdx.x]));
  __syncthreads();
  const uint64_t t0 = dmc::globaltimer_ns();
  first[threadIdx.x] = dmc::warp_wait(dmc::smem_u32(&bars[warp]), 0, &abort_word, err) ? 1 : 0;
  second[threadIdx.x] = dmc::warp_wait(dmc::smem_u32(&bars[warps]), 0, &abort_word, err) ? 1 : 0;
  ns[threadIdx.x] = dmc::globaltimer_ns() - t0;
}

extern "C" int dmc_shared_give_up_probe(int warps, unsigned arrived, unsigned int* err_dev, int* first_dev,
                                        int* second_dev, unsigned long long* ns_dev, cudaStream_t stream) {
  if (warps < 1 || warps > kMaxWarps) return (int)cudaErrorInvalidValue;
  shared_give_up_kernel<<<1, warps * 32, 0, stream>>>(arrived, err_dev, first_dev, second_dev, ns_dev);
  return (int)cudaGetLastError();
}
