// Work items of the attention kernels: (view, head, query tile), from the device-resident row
// offsets.
#pragma once

#include "internal.h"

namespace ivit {

constexpr int MAX_VIEWS = 4096;

struct AttnItem {
  int v, h, r0, nq;  // view, head, first packed row, rows
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// cum[v] = items before view v (cum[sv]: all of them), for query tiles of `tile` rows; by the
// first warp of the block.
__device__ __forceinline__ void attention_items(const AttnTcArgs& a, int tile, int* cum) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  int before = 0;
  for (int v0 = 0; v0 < a.sv; v0 += 32) {
    const int v = v0 + lane;
    int n = v < a.sv ? (a.cu_rows[v + 1] - a.cu_rows[v] + tile - 1) / tile * a.heads : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, n, o);
      if (lane >= o) n += up;
    }
    if (v < a.sv) cum[v + 1] = before + n;
    before += __shfl_sync(0xffffffffu, n, 31);
  }
  if (lane == 0) cum[0] = 0;
}

// Item g of the call: views in order, in a view the heads, in a head the query tiles, so that
// the tiles that share keys and values run at the same time (their K and V come from L2).
__device__ __forceinline__ AttnItem attention_item(int g, int tile, const int* cum, const AttnTcArgs& a) {
  int lo = 0, hi = a.sv - 1;  // last view with cum[view] <= g
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cum[mid] <= g) lo = mid; else hi = mid - 1;
  }
  AttnItem it;
  it.v = lo;
  const int rb = a.cu_rows[lo], m = a.cu_rows[lo + 1] - rb;
  const int tiles = (m + tile - 1) / tile, rem = g - cum[lo];
  it.h = rem / tiles;
  const int qt = rem - it.h * tiles;
  it.r0 = rb + qt * tile;
  it.nq = min(tile, m - qt * tile);
  return it;
}

}  // namespace ivit
