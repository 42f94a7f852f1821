// Counts the fp32 inputs for which silu() of common.cuh and the division operator give other bits.
#include "common.cuh"

__global__ void silu_bits(unsigned long long* differ) {
  const unsigned low = blockIdx.x * 256 + threadIdx.x;  // 2^24 threads, the high byte in a loop
  unsigned bad = 0;
  for (unsigned high = 0; high < 256; ++high) {
    const float g = __uint_as_float(low | high << 24);
    const float a = hydra::silu(g), b = g / (1.0f + expf(-g));
    bad += __float_as_uint(a) != __float_as_uint(b) && !(isnan(a) && isnan(b));
  }
  if (bad) atomicAdd(differ, static_cast<unsigned long long>(bad));
}

extern "C" int count_silu_bits(unsigned long long* differ, void* stream) {
  silu_bits<<<1 << 16, 256, 0, static_cast<cudaStream_t>(stream)>>>(differ);
  return cudaPeekAtLastError();
}
