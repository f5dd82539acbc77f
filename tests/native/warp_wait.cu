// One warp whose lanes wait on different barriers: the even ones' completes,
// the odd ones' never does.  Prints how many lanes of warp_wait saw the phase
// complete (mixed, then with every barrier complete), how many of warp_flag saw
// a flag that only one lane's word holds, and how many lanes got past elect_one
// afterwards.  Built and run by tests/test_gpu_warp_wait.py.
#include <cstdio>

#include "fo_common.cuh"
#include "fo_ptx.cuh"

__global__ void probe(int* out) {
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ volatile int flag[32];
  const int lane = threadIdx.x;
  if (lane == 0) {
    fo::mbar_init(&bar[0], 1);
    fo::mbar_init(&bar[1], 1);
    fo::mbar_arrive(&bar[0]);
  }
  flag[lane] = lane == 5;
  __syncwarp();
  const bool mixed = fo::warp_wait(&bar[lane % 2], 0);   // half of the lanes give up after the limit
  const bool one = fo::elect_one();
  const bool same = fo::warp_wait(&bar[0], 0);
  const bool seen = fo::warp_flag(&flag[lane]), none = fo::warp_flag(&flag[0]);
  const bool two = fo::elect_one();
  atomicAdd(&out[0], mixed);
  atomicAdd(&out[1], same);
  atomicAdd(&out[2], seen);
  atomicAdd(&out[3], none);
  atomicAdd(&out[4], one + two);
}

int main() {
  int* d = nullptr;
  int h[5] = {-1, -1, -1, -1, -1};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
  probe<<<1, 32>>>(d);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  std::printf("%d %d %d %d %d\n", h[0], h[1], h[2], h[3], h[4]);
  return 0;
}
