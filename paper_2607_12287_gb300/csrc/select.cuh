// Token selection of one view by a thread block, one token per thread (shared by the encoder's
// selection kernel and the selection without allocation).
#pragma once

#include <stdint.h>

namespace ivit {

constexpr unsigned kFullWarp = 0xffffffffu;

// Exclusive prefix count of `flag` over the block in thread order; `total` gets the count.
// `scratch`: 33 ints of shared memory.  Every thread of the block calls it.
__device__ __forceinline__ int block_rank(bool flag, int* scratch, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const unsigned ballot = __ballot_sync(kFullWarp, flag);
  __syncthreads();  // the scratch's last use is over
  if (lane == 0) scratch[warp] = __popc(ballot);
  __syncthreads();
  if (warp == 0) {
    const int x = lane < nwarps ? scratch[lane] : 0;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFullWarp, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane < nwarps) scratch[lane] = incl - x;
    if (lane == 31) scratch[32] = incl;
  }
  __syncthreads();
  total = scratch[32];
  return scratch[warp] + __popc(ballot & ((1u << lane) - 1u));
}

// Whether this thread's score is among the k lowest of the block's valid ones, in the order
// (score ascending, thread ascending).  A NaN is below nothing and nothing is below it: with
// k > 0 it is selected, beside the k lowest of the others.  The k-th lowest is found by radix
// selection, eight bits at a time (a histogram of the candidates' digits and a scan of its 256
// bins per step), instead of comparing every score with every other one: the selection of 32
// views of 1024 tokens took 81 us that way, 51 this way, of which 47 are its scores' 302 MB.
// `hist`: 256 ints, `scratch`: 33 ints of shared memory.
__device__ __forceinline__ bool among_lowest(float s, bool valid, int k, int* hist, int* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool nan = valid && s != s;
  // order-preserving bits; -0 and +0 compare equal
  const uint32_t u = __float_as_uint(s == 0.f ? 0.f : s);
  const uint32_t key = (u >> 31) ? ~u : (u | 0x80000000u);
  bool cand = valid && !nan;
  int n;
  block_rank(cand, scratch, n);
  if (k <= 0) return false;
  if (k >= n) return valid;
  uint32_t prefix = 0;  // the k-th lowest key's digits so far
  int left = k;         // its rank among the candidates, from 1
#pragma unroll 1
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    const unsigned in = __ballot_sync(kFullWarp, cand);
    if (cand) {  // scores crowd into few bins: one addition per warp and bin
      const uint32_t digit = (key >> shift) & 255u;
      const unsigned same = __match_any_sync(in, digit);
      if (lane == __ffs(same) - 1) atomicAdd(hist + digit, __popc(same));
    }
    __syncthreads();
    if (warp == 0) {  // the bin that holds rank `left`: eight bins per lane
      int c[8], sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += c[j] = hist[8 * lane + j];
      int incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFullWarp, incl, o);
        if (lane >= o) incl += y;
      }
      int before = incl - sum;
      if (before < left && left <= incl) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (before < left && left <= before + c[j]) {
            scratch[0] = 8 * lane + j;
            scratch[1] = left - before;
          }
          before += c[j];
        }
      }
    }
    __syncthreads();
    const uint32_t digit = static_cast<uint32_t>(scratch[0]);
    left = scratch[1];
    prefix |= digit << shift;
    cand = cand && ((key >> shift) & 255u) == digit;
    __syncthreads();  // scratch and histogram are read before the next step writes them
  }
  // everything below the k-th lowest key, and the first `left` of those equal to it
  int equal;
  const int r = block_rank(cand, scratch, equal);
  return nan || (valid && (key < prefix || (cand && r < left)));
}

}  // namespace ivit
