// The kernels' small bounded wait (mbar_wait_small, warp_wait_small, record_abort in common.cuh) made to run
// out, with a limit of 20 ms on a barrier that nothing completes.  One CTA of four warps:
//   warp 0, lane 0  gives up after the limit and raises the abort flag;
//   warp 1, lane 0  would wait a hundred times longer, and is released by the flag;
//   warp 2          the same as a whole warp, with one outcome in every lane;
//   warp 3          waits on a barrier that completes, and later asks once more with the flag set.
// Then one thread records the status.  Prints what each waiter saw and the status word.
#include <cstdio>

#include "common.cuh"

namespace {

constexpr uint32_t kLimitNs = 20000000u;

__global__ void __launch_bounds__(128) wait_kernel(unsigned* status, int* saw, unsigned long long* ns) {
  __shared__ uint64_t bar[4];
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int b = 0; b < 4; ++b) glide::mbar_init(&bar[b], 1);
    abort_flag = 0;
    glide::fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 96) glide::mbar_arrive(&bar[3]);
  const uint64_t t0 = glide::global_timer_ns();
  int ok = 2;
  if (warp == 0 && lane == 0) ok = glide::mbar_wait_small(&bar[0], 0, &abort_flag, kLimitNs);
  if (warp == 1 && lane == 0) ok = glide::mbar_wait_small(&bar[1], 0, &abort_flag, 100 * kLimitNs);
  if (warp == 2) ok = glide::warp_wait_small(&bar[2], 0, &abort_flag);  // the kernels' own limit
  if (warp == 3) ok = glide::warp_wait_small(&bar[3], 0, &abort_flag);
  __syncwarp();
  if (lane == 0) ns[warp] = glide::global_timer_ns() - t0;
  const bool same = __all_sync(0xffffffffu, ok == __shfl_sync(0xffffffffu, ok, 0));
  if (lane == 0) saw[warp] = warp >= 2 && !same ? -1 : ok;
  __syncthreads();
  // a completed phase is seen whatever the flag says
  if (warp == 3) {
    ok = glide::warp_wait_small(&bar[3], 0, &abort_flag);
    if (lane == 0) saw[4] = ok;
  }
  if (threadIdx.x == 0) glide::record_abort(&abort_flag, status);
}

}  // namespace

int main() {
  struct Out {
    unsigned long long ns[4];
    unsigned status[4];
    int saw[8];
  }* out;
  if (cudaMallocManaged(&out, sizeof(Out)) != cudaSuccess) return 2;
  *out = Out{};
  wait_kernel<<<1, 128>>>(out->status, out->saw, out->ns);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  std::printf("%d %d %d %d %d %u", out->saw[0], out->saw[1], out->saw[2], out->saw[3], out->saw[4], out->status[0]);
  for (int w = 0; w < 4; ++w) std::printf(" %llu", out->ns[w] / 1000);
  std::printf("\n");
  return cudaFree(out) == cudaSuccess ? 0 : 2;
}
