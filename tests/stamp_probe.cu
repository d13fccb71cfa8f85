// The few-row GEMM of 40 rows x 96 features in two row groups, in timeline mode: prints its CTAs, how
// many of them left a stamp of their own (start and end), and how many other words were written.
#include <cstdio>

#include "../paper_2607_12287_gb300/csrc/internal.h"
#include "../paper_2607_12287_gb300/csrc/ptx.cuh"

#define CK(call)                                                   \
  do {                                                             \
    const cudaError_t e = (call);                                  \
    if (e != cudaSuccess) {                                        \
      std::fprintf(stderr, "%s: %s\n", #call, cudaGetErrorString(e)); \
      return 1;                                                    \
    }                                                              \
  } while (0)

int main() {
  constexpr int rows = 40, features = 96, k = 64, words = 2 * ivit::kStampCtas;
  char* d = nullptr;  // weights, rows, bias, result, error word, stamps: 4 KB blocks and more
  constexpr size_t block = 64 * 1024;
  CK(cudaMalloc(&d, 6 * block));
  CK(cudaMemset(d, 0, 6 * block));
  ivit::GemmArgs a;
  a.n_out = features;
  a.k = k;
  a.m_static = rows;
  a.row_groups = 2;
  a.w = reinterpret_cast<const ivit::bf16*>(d);
  a.x = reinterpret_cast<const ivit::bf16*>(d + block);
  a.err = reinterpret_cast<int*>(d + 4 * block);
  a.epi.kind = ivit::kEpiResid;
  a.epi.bias = reinterpret_cast<const float*>(d + 2 * block);
  a.epi.out_f32 = reinterpret_cast<float*>(d + 3 * block);
  a.epi.ld_out = features;
  ivit::g_stamp = reinterpret_cast<unsigned long long*>(d + 5 * block);
  CK(ivit::gemm_rows_setup());
  CK(ivit::launch_gemm_rows(1, a, nullptr));
  static unsigned long long h[words];
  CK(cudaMemcpy(h, d + 5 * block, sizeof h, cudaMemcpyDeviceToHost));
  const int ctas = features / 8 * 2;
  int own = 0, other = 0;
  for (int b = 0; b < words / 2; ++b) {
    if (b < ctas)
      own += h[2 * b] != 0 && h[2 * b + 1] != 0;
    else
      other += (h[2 * b] != 0) + (h[2 * b + 1] != 0);
  }
  std::printf("%d %d %d\n", ctas, own, other);
  return 0;
}
