// Prints how many of a 5 x 3 x 2 grid's CTAs left a stamp of their own (start and end) in timeline
// mode, and how many other words were written.
#include <cstdio>

#include "../paper_2607_12287_gb300/csrc/ptx.cuh"

__global__ void stamped(unsigned long long* s) {
  ivit::stamp_begin(s);
  ivit::stamp_end(s);
}

int main() {
  const size_t n = 2 * ivit::kStampCtas;
  unsigned long long *d = nullptr, h[n];
  if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
  stamped<<<dim3(5, 3, 2), 64>>>(d);
  if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  int own = 0, other = 0;
  for (size_t b = 0; b < n / 2; ++b)
    if (b < 30) own += h[2 * b] && h[2 * b + 1]; else other += (h[2 * b] != 0) + (h[2 * b + 1] != 0);
  std::printf("%d %d\n", own, other);
  return 0;
}
