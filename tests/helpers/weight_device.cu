// Device driver around the Wiener filters' pixel weight, used only by the GPU tests. Reads lines "lt inb" (FP32 as hexadecimal
// floats, "inf" too) from stdin and prints the device's weights as hexadecimal floats.
#include <cstdio>
#include <vector>

#include "../../paper_1810_02821_gb300/csrc/wf_gibbs.cuh"

__global__ void k_weights(const float2* in, float* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = wf::wf_weight(in[i].x, in[i].y);
}

int main() {
  std::vector<float2> in;
  float2 v;
  while (std::scanf("%f %f", &v.x, &v.y) == 2) in.push_back(v);
  const int n = int(in.size());
  std::vector<float> out(in.size());
  float2* din = nullptr;
  float* dout = nullptr;
  if (n == 0 || cudaMalloc(&din, n * sizeof(float2)) != cudaSuccess || cudaMalloc(&dout, n * sizeof(float)) != cudaSuccess)
    return 1;
  if (cudaMemcpy(din, in.data(), n * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess) return 2;
  k_weights<<<(n + 255) / 256, 256>>>(din, dout, n);
  if (cudaMemcpy(out.data(), dout, n * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  for (float w : out) std::printf("%a\n", double(w));
  return 0;
}
