// The twiddles w^1 .. w^15 of every job step of a line of n points, as the FP32 transforms form them
// (test_gpu_twiddles.py).
#include "rd_fft.cuh"

using namespace rd;

__global__ void k_twiddles(const cx<float>* tw, cx<float>* out, int steps) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= steps) return;
  cx<float> w[16];
  rf_twiddles<float, 16>(tw, s, w);
  for (int r = 1; r < 16; ++r) out[16 * s + r] = w[r];
}

// tw: n complex entries; out: 16 (n / 16) complex entries, [step][r]
extern "C" __attribute__((visibility("default"))) int twiddle_probe(int n, const float* tw, float* out) {
  const size_t bytes = (size_t)n * sizeof(cx<float>);
  cx<float>*dt = nullptr, *dout = nullptr;
  cudaError_t e = cudaMalloc(&dt, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&dout, bytes);
  if (e == cudaSuccess) e = cudaMemset(dout, 0, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(dt, tw, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_twiddles<<<(n / 16 + 127) / 128, 128>>>(dt, dout, n / 16);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, dout, bytes, cudaMemcpyDeviceToHost);
  cudaFree(dt);
  cudaFree(dout);
  return (int)e;
}
