// The finalize step's table log2 (lamp_fin.cuh) beside CUDA's, element by element, for
// tests/test_gpu_fin.py.
#include "lamp_fin.cuh"

__global__ void k_log2(const double* x, int n, double* got, double* want) {
  __shared__ lamp::LogEntry tab[128];
  if (threadIdx.x < 128) tab[threadIdx.x] = lamp::kLogTab[threadIdx.x];
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  got[i] = lamp::log2_table(x[i], tab);
  want[i] = log2(x[i]);
}

extern "C" int probe_log2(const double* x, int n, double* got, double* want) {
  k_log2<<<(n + 255) / 256, 256>>>(x, n, got, want);
  return (int)cudaDeviceSynchronize();
}
