// Attention of a few updated queries per view (see attention.cu for the operation), as a chain
// of as few dependent steps as the work allows.
//
// Work item = (view, head, tile of up to 16 packed updated rows); CTAs walk the items with a
// stride.  The eight warps split the view's keys, 32 at a time: queries, keys and values go
// from L2 straight into registers, in one round trip, in an order that makes them the
// fragments of mma.m16n8k16 --
//   S = Q K^T: a lane's 16 bytes of a row are 8 consecutive dims, taken in the same order on
//     both sides (as in gemm.cu);
//   O = P V: P's fragments are S's; V's want two keys of one dim in a register, so a lane loads
//     dims 8 g .. 8 g + 7 of the keys 2 t, 2 t + 1, 2 t + 8, 2 t + 9 and interleaves them: the
//     eight MMAs of a 64-dim block then each cover every eighth dim.  One or two 8-dim groups
//     past a block (heads of 72 and 80) come in single elements.
// Each warp keeps its own running maximum, sum and output; they meet once in shared memory.  In
// the exact form a probability is three bf16 terms that together hold all 24 bits of its fp32
// value, multiplied by V in turn.
//
// Bound: latency at small row counts (wait, one round trip, MMAs, one exchange); mma.sync's
// rate at larger ones, where attention.cu is the faster one (the rule is attention_few in
// engine.cu).  Heads of up to 64 have a form for two CTAs on an SM (128 registers; wider heads would
// spill, 8.8 -> 11.6 us), taken when there are more items than SMs: six views of 196 x 196, 3 heads
// of 64, 5.6 -> 4.9 us (a full encode of 12 layers in the exact form: 8 us less than with one CTA).  16 heads of 72, 256 keys, 26 queries: 3.9 us back to back against 6.1 there, whose
// 128-query tile walks the keys in three dependent steps.
#include "attention.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace ivit {
namespace {

constexpr int WARPS = 8, THREADS = WARPS * 32;
constexpr int TQ = 16;       // queries per item
constexpr int KW = 32;       // keys per warp and step

__device__ __forceinline__ uint4 load16(const bf16* p, bool ok) {
  return ok ? __ldcg(reinterpret_cast<const uint4*>(p)) : make_uint4(0, 0, 0, 0);
}

__device__ __forceinline__ uint32_t word(const uint4& v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&b);
}

// (bf16 widens to fp32 by its bits)
__device__ __forceinline__ float2 unpack_bf16(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// NC: 32-dim chunks of a head (rounded up); NB: 64-dim blocks of V; R: 8-dim groups past them;
// CTAS: CTAs per SM; TERMS: bf16 terms of a probability in P V, 1 (rounded, and the normaliser
// sums the rounded values) or 3 (all 24 bits of the fp32 value).
template <int NC, int NB, int R, int CTAS, int TERMS>
__global__ void __launch_bounds__(THREADS, CTAS) attention_rows_kernel(const AttnTcArgs a) {
  constexpr int NT = 8 * NB + R;             // output n-tiles
  constexpr int DW = 64 * NB + 8 * R + 4;    // floats of a partial output row
  extern __shared__ __align__(16) float sm[];
  float* po = sm;                            // [WARPS][TQ][DW]
  float* pm = po + WARPS * TQ * DW;          // [WARPS][TQ]
  float* pl = pm + WARPS * TQ;
  int* cum = reinterpret_cast<int*>(pl + WARPS * TQ);  // [sv + 1] items before each view
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int N = a.n_tok, D = a.dim, dh = a.dh;

  // The row offsets come from the selection kernel, at least two launches back.
  attention_items(a, TQ, cum);
  __syncthreads();
  const int n_items = cum[a.sv];
  pdl_wait();  // queries and this call's K/V rows (QKV kernel) are visible from here
  pdl_launch_dependents();
  stamp_begin(a.stamp);

  const float sc = rsqrtf(static_cast<float>(dh)) * 1.4426950408889634f;  // log2(e) / sqrt(dh)
  for (int s = blockIdx.x; s < n_items; s += gridDim.x) {
    const AttnItem it = attention_item(s, TQ, cum, a);
    const size_t head = static_cast<size_t>(it.h) * dh;
    const bf16* kbase = a.k + static_cast<size_t>(it.v) * N * D + head;
    const bf16* vbase = a.v + static_cast<size_t>(it.v) * N * D + head;
    uint4 q[NC][2];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int r = 0; r < 2; ++r)
        q[c][r] = load16(a.q + static_cast<size_t>(it.r0 + g + 8 * r) * D + head + 32 * c + 8 * t,
                         g + 8 * r < it.nq && 32 * c + 8 * t < dh);
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    float o[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[j][e] = 0.f;

    for (int k0 = warp * KW; k0 < N; k0 += WARPS * KW) {
      uint4 kf[4][NC];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int key = k0 + 8 * j + g;
          kf[j][c] = load16(kbase + static_cast<size_t>(key) * D + 32 * c + 8 * t, key < N && 32 * c + 8 * t < dh);
        }
      uint4 vf[2][4][NB];
      uint32_t vr[2][4][R > 0 ? R : 1];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const int key = k0 + 16 * u + 2 * t + (w & 1) + 8 * (w >> 1);
          const bf16* row = vbase + static_cast<size_t>(key) * D;
#pragma unroll
          for (int b = 0; b < NB; ++b) vf[u][w][b] = load16(row + 64 * b + 8 * g, key < N && 64 * b + 8 * g < dh);
#pragma unroll
          for (int x = 0; x < R; ++x)
            vr[u][w][x] = key < N ? __ldcg(reinterpret_cast<const unsigned short*>(row + 64 * NB + 8 * x + g)) : 0u;
        }
      float sv[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int e = 0; e < 4; ++e) sv[j][e] = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          mma_bf16_16816(sv[j], q[c][0].x, q[c][1].x, q[c][0].y, q[c][1].y, kf[j][c].x, kf[j][c].y);
          mma_bf16_16816(sv[j], q[c][0].z, q[c][1].z, q[c][0].w, q[c][1].w, kf[j][c].z, kf[j][c].w);
        }
      }
      if (k0 + KW > N) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (k0 + 8 * j + 2 * t + (e & 1) >= N) sv[j][e] = -INFINITY;
      }
      uint32_t p[4][2];  // P of (keys 8 j + 2 t, + 1) of rows g and g + 8
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) mx = fmaxf(mx, fmaxf(sv[j][2 * r], sv[j][2 * r + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m[r], mx), m_fin = m_new == -INFINITY ? 0.f : m_new;  // (scores of -inf alone so far:
        const float alpha = ex2((m[r] - m_fin) * sc), mo = m_fin * sc;                  // P = 0, nothing to rescale)
        m[r] = m_new;
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float2 f = make_float2(ex2(fmaf(sv[j][2 * r], sc, -mo)), ex2(fmaf(sv[j][2 * r + 1], sc, -mo)));
          if (TERMS == 1) {
            p[j][r] = pack_bf16(f.x, f.y);
            f = unpack_bf16(p[j][r]);
          } else {
            sv[j][2 * r] = f.x;
            sv[j][2 * r + 1] = f.y;
          }
          sum += f.x + f.y;  // the normaliser sums the values the MMA multiplies
        }
        l[r] = l[r] * alpha + sum;
        if (k0 >= WARPS * KW) {
#pragma unroll
          for (int j = 0; j < NT; ++j) {
            o[j][2 * r] *= alpha;
            o[j][2 * r + 1] *= alpha;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        uint32_t pa[TERMS][4];
#pragma unroll
        for (int x = 0; x < TERMS; ++x)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = 2 * u + (e >> 1), r = e & 1;
            if (TERMS == 1) {
              pa[x][e] = p[j][r];
            } else {  // the next 8 bits of both probabilities
              pa[x][e] = pack_bf16(sv[j][2 * r], sv[j][2 * r + 1]);
              const float2 f = unpack_bf16(pa[x][e]);
              sv[j][2 * r] -= f.x;
              sv[j][2 * r + 1] -= f.y;
            }
          }
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
            const uint32_t b0 = __byte_perm(word(vf[u][0][b], j >> 1), word(vf[u][1][b], j >> 1), sel),
                           b1 = __byte_perm(word(vf[u][2][b], j >> 1), word(vf[u][3][b], j >> 1), sel);
#pragma unroll
            for (int x = 0; x < TERMS; ++x) mma_bf16_16816(o[8 * b + j], pa[x][0], pa[x][1], pa[x][2], pa[x][3], b0, b1);
          }
#pragma unroll
        for (int y = 0; y < R; ++y)
#pragma unroll
          for (int x = 0; x < TERMS; ++x)
            mma_bf16_16816(o[8 * NB + y], pa[x][0], pa[x][1], pa[x][2], pa[x][3], vr[u][0][y] | (vr[u][1][y] << 16),
                           vr[u][2][y] | (vr[u][3][y] << 16));
      }
    }

    // this warp's (m, l, O) of rows g, g + 8 to shared memory
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
      l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
      const int row = warp * TQ + g + 8 * r;
      if (t == 0) {
        pm[row] = m[r];
        pl[row] = l[r];
      }
      float* d = po + row * DW;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          // the eight tiles of a block hold dims 8 (2 t + e) + 0 .. 7 of it
          float4* d4 = reinterpret_cast<float4*>(d + 64 * b + 8 * (2 * t + e));
          d4[0] = make_float4(o[8 * b][2 * r + e], o[8 * b + 1][2 * r + e], o[8 * b + 2][2 * r + e], o[8 * b + 3][2 * r + e]);
          d4[1] = make_float4(o[8 * b + 4][2 * r + e], o[8 * b + 5][2 * r + e], o[8 * b + 6][2 * r + e],
                              o[8 * b + 7][2 * r + e]);
        }
#pragma unroll
        for (int x = 0; x < R; ++x) d[64 * NB + 8 * x + 2 * t + e] = o[8 * NB + x][2 * r + e];
      }
    }
    __syncthreads();
    const int c8 = dh >> 3;
    for (int e = tid; e < it.nq * c8; e += THREADS) {
      const int row = e / c8, c = e - row * c8;
      float M = pm[row];
#pragma unroll
      for (int w = 1; w < WARPS; ++w) M = fmaxf(M, pm[w * TQ + row]);
      float L = 0.f, acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        const float f = ex2((pm[w * TQ + row] - M) * sc);  // a warp without keys: m = -inf, 0
        L += f * pl[w * TQ + row];
        const float4* x = reinterpret_cast<const float4*>(po + (w * TQ + row) * DW + 8 * c);
        const float4 x0 = x[0], x1 = x[1];
        acc[0] += f * x0.x;
        acc[1] += f * x0.y;
        acc[2] += f * x0.z;
        acc[3] += f * x0.w;
        acc[4] += f * x1.x;
        acc[5] += f * x1.y;
        acc[6] += f * x1.z;
        acc[7] += f * x1.w;
      }
      const float inv = 1.f / L;
      uint4 u;
      uint32_t* w4 = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(acc[2 * k] * inv, acc[2 * k + 1] * inv);
        w4[k] = *reinterpret_cast<const uint32_t*>(&b);
      }
      *reinterpret_cast<uint4*>(a.o + static_cast<size_t>(it.r0 + row) * D + head + 8 * c) = u;
    }
    __syncthreads();  // the partials are read before the next item's
  }
  stamp_end(a.stamp);
}

template <int NB, int R>
constexpr size_t smem_bytes() {
  return static_cast<size_t>(WARPS) * TQ * (64 * NB + 8 * R + 4 + 2) * 4;
}

}  // namespace

cudaError_t attention_rows_setup() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kern, size_t bytes) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(bytes + 4 * (MAX_VIEWS + 1)));
  };
  auto both = [&](auto rounded, auto exact, size_t bytes) {
    set(rounded, bytes);
    set(exact, bytes);
  };
  both(attention_rows_kernel<1, 1, 0, 1, 1>, attention_rows_kernel<1, 1, 0, 1, 3>, smem_bytes<1, 0>());
  both(attention_rows_kernel<2, 1, 0, 1, 1>, attention_rows_kernel<2, 1, 0, 1, 3>, smem_bytes<1, 0>());
  both(attention_rows_kernel<1, 1, 0, 2, 1>, attention_rows_kernel<1, 1, 0, 2, 3>, smem_bytes<1, 0>());
  both(attention_rows_kernel<2, 1, 0, 2, 1>, attention_rows_kernel<2, 1, 0, 2, 3>, smem_bytes<1, 0>());
  set(attention_rows_kernel<3, 1, 1, 1, 1>, smem_bytes<1, 1>());
  both(attention_rows_kernel<3, 1, 2, 1, 1>, attention_rows_kernel<3, 1, 2, 1, 3>, smem_bytes<1, 2>());
  both(attention_rows_kernel<3, 2, 0, 1, 1>, attention_rows_kernel<3, 2, 0, 1, 3>, smem_bytes<2, 0>());
  both(attention_rows_kernel<4, 2, 0, 1, 1>, attention_rows_kernel<4, 2, 0, 1, 3>, smem_bytes<2, 0>());
  return e;
}

cudaError_t launch_attention_rows(const AttnTcArgs& a, int num_sms, int ctas, bool exact, cudaStream_t s) {
  if (a.sv > MAX_VIEWS || a.dh % 8 || a.dh > 128) return cudaErrorInvalidValue;
  const bool two = ctas == 2 && a.dh <= 64;
  const int grid = max(1, min(a.sv * a.heads * ((a.n_tok + TQ - 1) / TQ), two ? 2 * num_sms : num_sms));
  auto launch = [&](auto rounded, auto full, size_t bytes) {
    return launch_ex(exact ? full : rounded, dim3(grid), dim3(THREADS), bytes + 4 * (a.sv + 1), s, 1, a);
  };
  if (two && a.dh <= 32)
    return launch(attention_rows_kernel<1, 1, 0, 2, 1>, attention_rows_kernel<1, 1, 0, 2, 3>, smem_bytes<1, 0>());
  if (two) return launch(attention_rows_kernel<2, 1, 0, 2, 1>, attention_rows_kernel<2, 1, 0, 2, 3>, smem_bytes<1, 0>());
  if (a.dh <= 32)
    return launch(attention_rows_kernel<1, 1, 0, 1, 1>, attention_rows_kernel<1, 1, 0, 1, 3>, smem_bytes<1, 0>());
  if (a.dh <= 64)
    return launch(attention_rows_kernel<2, 1, 0, 1, 1>, attention_rows_kernel<2, 1, 0, 1, 3>, smem_bytes<1, 0>());
  if (a.dh == 72) {  // (an encoder with such heads is at least 576 wide: no exact form)
    if (exact) return cudaErrorInvalidValue;
    return launch(attention_rows_kernel<3, 1, 1, 1, 1>, attention_rows_kernel<3, 1, 1, 1, 1>, smem_bytes<1, 1>());
  }
  if (a.dh == 80)
    return launch(attention_rows_kernel<3, 1, 2, 1, 1>, attention_rows_kernel<3, 1, 2, 1, 3>, smem_bytes<1, 2>());
  if (a.dh <= 96)
    return launch(attention_rows_kernel<3, 2, 0, 1, 1>, attention_rows_kernel<3, 2, 0, 1, 3>, smem_bytes<2, 0>());
  return launch(attention_rows_kernel<4, 2, 0, 1, 1>, attention_rows_kernel<4, 2, 0, 1, 3>, smem_bytes<2, 0>());
}

}  // namespace ivit
