// Two threads that launch the classifier head over and over, one with 1000 and
// one with 600 classes (different amounts of shared memory of one kernel), each
// on its own stream.  Prints how many launches of each were refused.  Built
// with k_head.cu and run by tests/test_gpu_head_threads.py.
#include <cstdio>
#include <thread>

#include "fo_common.cuh"
#include "fo_kernels.h"

namespace fo {
bool pdl_enabled() { return false; }
}  // namespace fo

constexpr int kRows = 128, kWidth = 64, kLaunches = 4000;

static void drive(int classes, int* refused) {
  float *x, *w, *logits, *dz, *loss;
  int32_t* labels;
  cudaStream_t st;
  *refused = -1;
  if (cudaStreamCreate(&st) != cudaSuccess || cudaMalloc(&x, 4 * kRows * kWidth) != cudaSuccess ||
      cudaMalloc(&w, 4 * classes * kWidth) != cudaSuccess || cudaMalloc(&logits, 4 * kRows * classes) != cudaSuccess ||
      cudaMalloc(&dz, 4 * kRows * classes) != cudaSuccess || cudaMalloc(&loss, 4 * kRows) != cudaSuccess ||
      cudaMalloc(&labels, 4 * kRows) != cudaSuccess)
    return;
  cudaMemsetAsync(x, 0, 4 * kRows * kWidth, st);
  cudaMemsetAsync(w, 0, 4 * classes * kWidth, st);
  cudaMemsetAsync(labels, 0, 4 * kRows, st);
  int n = 0;
  for (int i = 0; i < kLaunches; ++i) {
    fo::head_forward_loss(x, fo::kF32, w, nullptr, labels, kRows, kWidth, classes, logits, dz, loss, st);
    n += cudaGetLastError() != cudaSuccess;
  }
  if (cudaStreamSynchronize(st) == cudaSuccess) *refused = n;
}

int main() {
  int a = 0, b = 0;
  if (cudaFree(nullptr) != cudaSuccess) return 1;
  std::thread t1(drive, 1000, &a), t2(drive, 600, &b);
  t1.join();
  t2.join();
  std::printf("%d %d\n", a, b);
  return 0;
}
