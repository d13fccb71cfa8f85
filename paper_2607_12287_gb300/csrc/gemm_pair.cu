// Tensor-core GEMM over CTA pairs (tcgen05 cta_group::2), for every GEMM of more than about
// 64 rows: Y[r][f] = sum_k X[r][k] W[f][k] for the packed rows, then an epilogue of
// GemmEpilogue.
//
// A cluster of two CTAs computes a tile of 256 output features x BN rows: each CTA stages
// its 128 features of W and its half of the BN rows of X, the leader's MMA warp multiplies
// 256 x BN from both shared memories, and each CTA's tensor memory receives its 128 features
// (lanes) x BN rows (columns).  A CTA fetches (128 + BN / 2) x 128 bytes per 64-wide k-block
// where a CTA on its own fetches (128 + BN) x 128 for the same MMA work.
//
// What bounds it: at large row counts the tensor pipe under the power limit; at a few
// hundred rows the chain of one tile (prologue, 18 to 68 k-blocks, epilogue).  What the
// single-CTA kernels before it spent their time on, and what is done about it here:
//   - the loops that issue TMA and MMA run as whole warps with one elected lane, so their
//     operands stay in uniform registers; one diverged lane needed 0.31 us per k-block of a
//     64-row tile whatever the number of stages, this form 0.19;
//   - X comes in one box of BN / 2 rows per stage, not in boxes of 32 (down-projection of
//     32768 rows 260 -> 226 us);
//   - one epilogue per instantiation, through shared memory and 16-byte accesses: the
//     epilogue that stored column by column behind a switch took 7.5 us for 64 rows x 128
//     features, most of it on instruction fetch.  The residual is added in L2 (red.v4.f32),
//     so it is never loaded.
// Measured back to back (whole launches, prologue included), random bf16 data, before -> now:
// 32768 rows QKV 422 -> 149 us (1750 TFLOP/s), up 497 -> 195, out 154 -> 78, down 324 -> 218; 3080
// rows QKV 65 -> 23, up 60 -> 27, down 53 -> 29; 768 rows QKV 29 -> 12, up 27 -> 13; 256 rows QKV
// 16 -> 6.9, up 16 -> 7.6.
#include "gelu.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace ivit {
namespace {

constexpr int BM = 128;   // output features per CTA (a pair's MMA has M = 256)
constexpr int BK = 64;    // K per stage: 128-byte rows, 128-byte swizzle
constexpr int W_BYTES = BM * BK * 2;
constexpr int EPI_WARPS = 8;
constexpr int THREADS = (EPI_WARPS + 2) * 32;
constexpr int EPI_HALF = 8192;  // a staging buffer: 32 rows of 128 bf16 or 16 of fp32

// As many stages as fit for the two smaller tiles: the first ones hold weights requested before
// the wait on the previous kernel.  64-row tiles with 2 / 3 / 4 / 5 stages: four-layer 224 px
// full encode 221 / 200 / 192 / 189 us.
template <int BN>
struct PairCfg {
  // k-blocks per stage: 64-row tiles are bound by the issuing warps, not by the MMAs, so they
  // take two per barrier (0.20 -> 0.16 us per k-block; up of 256 rows 8.5 -> 7.8 us)
  static constexpr int KS = BN == 64 ? 2 : 1;
  static constexpr int STAGES = BN == 64 ? 5 : BN == 128 ? 8 : 6;
  static constexpr int X_BYTES = BN / 2 * BK * 2;
  static constexpr int X_OFFSET = KS * W_BYTES;
  static constexpr int KB_BYTES = W_BYTES + X_BYTES;
  static constexpr int STAGE_BYTES = KS * KB_BYTES;
  static constexpr int EPI_OFFSET = STAGES * STAGE_BYTES;
  static constexpr int BUFS = BN == 256 ? 2 : 1;  // staging buffers per row half
  static constexpr int BAR_OFFSET = EPI_OFFSET + 2 * BUFS * EPI_HALF;
  static constexpr int TOTAL = BAR_OFFSET + 256 + 1024;  // barriers, flags, 1 KB alignment slack
  static_assert(TOTAL <= 227 * 1024, "shared memory of one CTA");
};

// Sums over a warp of three values of four rows each (v[row]): lanes 8 k .. 8 k + 7 get row k's.
__device__ __forceinline__ float3 sum_rows4(const float3 (&v)[4], int lane) {
  auto fold = [&](const float3& keep, const float3& send, int o) {
    return make_float3(keep.x + __shfl_xor_sync(0xffffffffu, send.x, o), keep.y + __shfl_xor_sync(0xffffffffu, send.y, o),
                       keep.z + __shfl_xor_sync(0xffffffffu, send.z, o));
  };
  const bool hi = lane & 16, mid = lane & 8;
  const float3 p = fold(hi ? v[2] : v[0], hi ? v[0] : v[2], 16), q = fold(hi ? v[3] : v[1], hi ? v[1] : v[3], 16);
  float3 s = fold(mid ? q : p, mid ? p : q, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s = fold(s, s, o);
  return s;
}

// Drains rows [c_lo, c_hi) of the tile (columns of this CTA's accumulator) on the four
// warps of one row half: chunks of 32 rows (16 when fp32) go from tensor memory (lane =
// feature) through shared memory (row-major) to global memory with 16-byte accesses, 128
// features of a row at a time.  `ready` waits for the accumulator (false: nothing is stored),
// `release` is called once, when it has been read.  The next chunk's accumulators and rows are
// requested before this one is stored, and the staging has two buffers if there is room (`buf`:
// the one to use, kept over the tiles of a CTA), so that a chunk costs one barrier and no round
// trip.
template <int KIND, int BUFS, class Ready, class Release>
__device__ __forceinline__ void drain(const GemmArgs& a, uint32_t acc, uint8_t* stg, int bar_id, int wq, int lane,
                                      int row0, int c_lo, int c_hi, int ft, float* slot, int& buf, Ready ready,
                                      Release release) {
  constexpr bool kGelu = KIND == kEpiGelu || KIND == kEpiGeluTanhf, kBf16 = KIND == kEpiQKV || kGelu;
  constexpr int CHUNK = kBf16 ? 32 : 16;
  constexpr bool kAhead = BUFS == 2, kByTok = KIND == kEpiQKV || KIND == kEpiScatterF32;
  const int f0 = ft * BM, fl = wq * 32 + lane;
  float bias = 0.f;
  if (KIND != kEpiPartial && f0 + fl < a.n_out) bias = __ldg(a.epi.bias + f0 + fl);
  // this thread's part of a row in the second step: 8 bf16 features (two rows per warp
  // and access) or 4 fp32 features (one row)
  constexpr int FPT = kBf16 ? 8 : 4, LPR = BM / FPT, RPW = 32 / LPR, ITERS = CHUNK / (4 * RPW);
  const int sub = lane % LPR, rsub = wq * RPW + lane / LPR;
  const int f = f0 + FPT * sub;
  bf16* dst16 = nullptr;
  float* dst32 = nullptr;
  bool by_tok = KIND == kEpiScatterF32;
  int ld = a.epi.ld_out;
  if (KIND == kEpiQKV) {
    const int D = a.epi.dim;  // D % 64 == 0: 8 features never straddle Q, K and V
    dst16 = f < D ? a.epi.out_bf16 + f : f < 2 * D ? a.epi.cache_k + (f - D) : a.epi.cache_v + (f - 2 * D);
    by_tok = f >= D;
    ld = D;
  } else if (kGelu) {
    dst16 = a.epi.out_bf16 + f;
  } else if (KIND == kEpiPartial) {
    dst32 = slot + FPT * sub;
    ld = BM;
  } else {
    dst32 = a.epi.out_f32 + f;
  }
  // kEpiScore: the rows' previous content, four chunks ahead (the first ones under the main
  // loop): one chunk at a time was bound by their latency
  constexpr int AHEAD = 4;
  float4 old[KIND == kEpiScore ? AHEAD : 1][ITERS];
  auto load_old = [&](int c0, float4 (&d)[ITERS]) {
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int c = c0 + i * 4 * RPW + rsub;
      d[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < c_hi && f < a.n_out)
        d[i] = __ldcg(reinterpret_cast<const float4*>(dst32 + static_cast<size_t>(row0 + c) * ld));
    }
  };
  if constexpr (KIND == kEpiScore) {
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) load_old(c_lo + k * CHUNK, old[k]);
  }
  int rr[ITERS];  // destination rows, -1 past the tile's end
  auto load_rows = [&](int c0, int (&d)[ITERS]) {
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int c = c0 + i * 4 * RPW + rsub;
      d[i] = -1;
      if (c < c_hi && f < a.n_out)
        d[i] = KIND == kEpiPartial ? c : by_tok ? __ldcg(a.epi.rowtok + row0 + c) : row0 + c;
    }
  };
  // (the rows' tokens: a round trip under the main loop and not after it, QKV of 1176 rows x 192
  // 3.6 -> 3.3 us)
  if (kAhead || kByTok) load_rows(c_lo, rr);
  const bool ok = ready();
  uint32_t v[CHUNK];
  auto load_acc = [&](int c0) {
    if constexpr (kBf16)
      tmem_ld32_async(acc + c0, v);
    else
      tmem_ld16_async(acc + c0, v);
  };
  if (kAhead) load_acc(c_lo);
  auto chunk = [&](int c0, const float4 (&prev)[ITERS]) {
    if (!kAhead) {
      if (!kByTok || c0 != c_lo) load_rows(c0, rr);
      load_acc(c0);
    }
    if constexpr (kBf16) {
      tmem_ld_wait_regs(v);
    } else {
      tmem_ld_wait();
      tmem_regs_after_wait16(v);
    }
    const bool last = c0 + CHUNK >= c_hi;
    if (last) release();
    uint8_t* sb = stg + buf * EPI_HALF;
    if (BUFS == 2)
      buf ^= 1;
    else
      named_barrier(bar_id, 128);  // the previous chunk has left the staging buffer
    if (kBf16) {
      bf16* st = reinterpret_cast<bf16*>(sb) + fl;
#pragma unroll
      for (int j = 0; j < CHUNK; ++j) {
        float y = __uint_as_float(v[j]) + bias;
        if (kGelu) y = gelu_f<KIND>(y, a.epi.gelu_mode);
        st[j * BM] = __float2bfloat16_rn(y);
      }
    } else {
      float* st = reinterpret_cast<float*>(sb) + fl;
#pragma unroll
      for (int j = 0; j < CHUNK; ++j) st[j * BM] = __uint_as_float(v[j]) + bias;
    }
    int next[ITERS];
    if (kAhead && !last) {
      load_acc(c0 + CHUNK);
      load_rows(c0 + CHUNK, next);
    }
    named_barrier(bar_id, 128);
    float3 sums[KIND == kEpiScore ? ITERS : 1];
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const uint4 u = *reinterpret_cast<const uint4*>(sb + ((i * 4 * RPW + rsub) * LPR + sub) * 16);
      if constexpr (KIND == kEpiScore) sums[i] = make_float3(0.f, 0.f, 0.f);
      if (rr[i] < 0 || !ok) continue;
      const size_t off = static_cast<size_t>(rr[i]) * ld;
      if (kBf16)
        *reinterpret_cast<uint4*>(dst16 + off) = u;
      else if (KIND == kEpiResid)
        red_add_f32x4(dst32 + off, *reinterpret_cast<const float4*>(&u));
      else
        *reinterpret_cast<uint4*>(dst32 + off) = u;
      if constexpr (KIND == kEpiScore) {
        const float4 x = *reinterpret_cast<const float4*>(&u), y = prev[i];
        sums[i] = make_float3(x.x * y.x + x.y * y.y + x.z * y.z + x.w * y.w,
                              x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w,
                              y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w);
      }
    }
    if constexpr (KIND == kEpiScore) {  // (a warp holds 128 features of one row per iteration)
      const float3 s = sum_rows4(sums, lane);
      const int c = c0 + (lane >> 3) * 4 + wq;
      if ((lane & 7) == 0 && c < c_hi && ok)
        a.epi.score[static_cast<size_t>(ft) * a.m_static + row0 + c] = make_float4(s.x, s.y, s.z, 0.f);
    }
    if (kAhead && !last) {
#pragma unroll
      for (int i = 0; i < ITERS; ++i) rr[i] = next[i];
    }
  };
  if constexpr (KIND == kEpiScore) {
    for (int c0 = c_lo; c0 < c_hi; c0 += AHEAD * CHUNK) {
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) {
        if (c0 + k * CHUNK >= c_hi) break;
        chunk(c0 + k * CHUNK, old[k]);
        load_old(c0 + (AHEAD + k) * CHUNK, old[k]);
      }
    }
  } else {
    for (int c0 = c_lo; c0 < c_hi; c0 += CHUNK) chunk(c0, old[0]);
  }
}

// The same for a half of a 64-row tile, where it is faster: at most 32 rows of this warp's 32
// features straight from the registers, 64 or 128 bytes per access, without the exchange through
// shared memory and its barriers.  256 rows of the So400m shapes in the replayed graph, from a
// launch's wait on the kernel before to its last store (without the prologue of the figures above),
// staged -> direct: out and down 5.9 -> 5.7 us, QKV 5.4 -> 5.3, but up with GELU 6.2 -> 7.1 and the
// embedding 4.5 -> 4.7.
template <int KIND>
constexpr bool kDirect = KIND == kEpiResid || KIND == kEpiPartial || KIND == kEpiQKV || KIND == kEpiScatterF32;

template <int KIND, class Ready, class Release>
__device__ __forceinline__ void drain_direct(const GemmArgs& a, uint32_t acc, int wq, int lane, int row0, int c_lo,
                                             int c_hi, int ft, float* slot, Ready ready, Release release) {
  const int fl = wq * 32 + lane, f = ft * BM + fl;
  const bool f_ok = f < a.n_out;
  const float bias = KIND != kEpiPartial && f_ok ? __ldg(a.epi.bias + f) : 0.f;
  constexpr bool kByTok = KIND == kEpiQKV || KIND == kEpiScatterF32;
  bool by_tok = kByTok;
  size_t ld = KIND == kEpiPartial ? BM : a.epi.ld_out;
  bf16* dst16 = nullptr;
  float* dst32 = nullptr;
  if (KIND == kEpiQKV) {
    const int D = a.epi.dim;  // D % 64 == 0: a warp's features never straddle Q, K and V
    dst16 = f < D ? a.epi.out_bf16 + f : f < 2 * D ? a.epi.cache_k + (f - D) : a.epi.cache_v + (f - 2 * D);
    by_tok = f >= D;
    ld = D;
  } else {
    dst32 = KIND == kEpiPartial ? slot + fl - static_cast<ptrdiff_t>(row0) * BM : a.epi.out_f32 + f;
  }
  int row = row0 + c_lo + lane;  // of the lane's turn
  if (by_tok && c_lo + lane < c_hi) row = __ldcg(a.epi.rowtok + row);
  const int n = ready() && f_ok ? c_hi - c_lo : 0;
  uint32_t v[32];
  tmem_ld32_async(acc + c_lo, v);
  tmem_ld_wait_regs(v);
  release();
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int r = kByTok ? __shfl_sync(0xffffffffu, row, j) : row0 + c_lo + j;
    const float y = __uint_as_float(v[j]) + bias;
    if (j < n) {
      if (KIND == kEpiQKV)
        dst16[r * ld] = __float2bfloat16_rn(y);
      else if (KIND == kEpiResid)
        atomicAdd(dst32 + r * ld, y);
      else
        dst32[r * ld] = y;
    }
  }
}

// What L2 is to keep.  A few row tiles read the weights about once: the rows, which every
// feature pair reads, stay.  256-row tiles come in many rounds and read the weights in each,
// while a tile's rows are done with after one round and may exceed L2 altogether: the weights
// stay.  32768 rows of the So400m shapes: QKV 153 -> 149 us, up 203 -> 198.
template <int BN>
__device__ __forceinline__ uint64_t weight_policy() {
  return BN == 256 ? l2_policy_evict_last() : l2_policy_evict_first();
}

template <int BN, int KIND>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                     const GemmArgs a) {
  using C = PairCfg<BN>;
  constexpr int STAGES = C::STAGES, KS = C::KS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::BAR_OFFSET);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
  volatile int* sh_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t smem_base = smem_u32(smem), bar_base = smem_u32(bars);
  const uint32_t accf = bar_base + 8 * (2 * STAGES), acce = accf + 16;
  const int rank = static_cast<int>(cluster_ctarank());
  const uint64_t desc0 = sdesc_kmajor_sw128(smem_base);

  if (tid == 0) {
    for (int st = 0; st < STAGES; ++st) {
      mbar_init(bar_base + 8 * st, 1);             // full: the leader's expected bytes of both CTAs
      mbar_init(bar_base + 8 * (STAGES + st), 1);  // empty: the pair's MMAs have read the stage
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf + 8 * b, 1);
      mbar_init(acce + 8 * b, 2 * EPI_WARPS);  // the epilogue warps of both CTAs
    }
    fence_mbar_init();
    tma_prefetch_desc(&tm_w);
    tma_prefetch_desc(&tm_x);
    *sh_abort = 0;
  }
  if (warp == EPI_WARPS + 1) tmem_alloc_pair(smem_u32(tmem_slot), 2 * BN);
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before any copy or arrival reaches them
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // The row count comes from the selection kernel, at least two launches back.
  const int M = a.d_rows ? *a.d_rows : a.m_static;
  const int n_ft = (a.n_out + BM - 1) / BM, n_fp = (n_ft + 1) / 2;
  const int n_tt = (M + BN - 1) / BN;
  const int n_kb = (a.k + BK - 1) / BK;
  const int splits = KIND == kEpiPartial ? a.vsplit : 1;
  const int units = n_fp * n_tt * splits;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  // unit u: K split u % splits of feature pair (u / splits) % n_fp, row tile the rest
  auto rows_of = [&](int tt) { return min(BN, M - tt * BN); };
  auto half_of = [&](int rows) { return ((rows + 31) >> 5) << 4; };  // rows of X per CTA (MMA N / 2)

  int n_pre = 0;
  if (warp == EPI_WARPS && pair < units) {
    // the first unit's weight stages do not depend on earlier kernels
    const int sp = pair % splits, ft = 2 * (pair / splits % n_fp) + rank;
    const int kb0 = sp * n_kb / splits, kb1 = (sp + 1) * n_kb / splits;
    n_pre = min(STAGES * KS, kb1 - kb0);
    if (elect_one()) {
      const uint64_t pol_w = weight_policy<BN>();
      for (int i = 0; i < n_pre; ++i) {
        const int st = i / KS, j = i - st * KS;
        if (rank == 0 && j == 0) mbar_arrive_expect_tx(bar_base + 8 * st, 2 * min(KS, n_pre - i) * C::KB_BYTES);
        tma_load_2d_pair(smem_base + st * C::STAGE_BYTES + j * W_BYTES, &tm_w, (kb0 + i) * BK, ft * BM,
                         mapa_shared(bar_base + 8 * st, 0), pol_w);
      }
    }
    __syncwarp();
  }
  pdl_wait();
  pdl_launch_dependents();
  stamp_begin(a.stamp);

  if (warp == EPI_WARPS) {
    const uint64_t pol_w = weight_policy<BN>();
    const uint64_t pol_x = BN == 256 ? l2_policy_evict_normal() : l2_policy_evict_last();
    uint32_t stage = 0, phase = 0;
    bool first = true, ok = true;
    const uint32_t full0 = mapa_shared(bar_base, 0);
    for (int u = pair; u < units && ok; u += n_pairs) {
      const int sp = u % splits, tile = u / splits;
      const int ft = 2 * (tile % n_fp) + rank, tt = tile / n_fp;
      const int half = half_of(rows_of(tt));
      const int xrow = tt * BN + rank * half;
      const int kb0 = sp * n_kb / splits, kb1 = (sp + 1) * n_kb / splits;
      for (int kb = kb0; kb < kb1; kb += KS) {
        const int nk = min(KS, kb1 - kb);
        const uint32_t full = full0 + 8 * stage;
        const uint32_t st = smem_base + stage * C::STAGE_BYTES;
        const bool pre = first && kb - kb0 < n_pre;
        if (!pre) ok = __all_sync(0xffffffffu, mbar_wait(bar_base + 8 * (STAGES + stage), phase ^ 1));
        if (!ok) break;
        if (elect_one()) {
          if (!pre) {
            if (rank == 0) mbar_arrive_expect_tx(bar_base + 8 * stage, 2 * nk * C::KB_BYTES);
#pragma unroll
            for (int j = 0; j < KS; ++j)
              if (j < nk) tma_load_2d_pair(st + j * W_BYTES, &tm_w, (kb + j) * BK, ft * BM, full, pol_w);
          }
#pragma unroll
          for (int j = 0; j < KS; ++j)
            if (j < nk)
              tma_load_2d_pair(st + C::X_OFFSET + j * C::X_BYTES, &tm_x, (kb + j) * BK, xrow, full, pol_x);
        }
        __syncwarp();
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
      first = false;
    }
    if (!ok) {
      atomicExch(a.err, kErrWaitSlotEmpty);
      *sh_abort = 1;
    }
  } else if (warp == EPI_WARPS + 1) {
    if (rank == 0) {
      uint32_t stage = 0, phase = 0;
      int iter = 0;
      for (int u = pair; u < units; u += n_pairs, ++iter) {
        const int sp = u % splits, tt = u / splits / n_fp;
        const uint32_t idesc = idesc_bf16_f32(2 * BM, 2 * half_of(rows_of(tt)));
        const int kb0 = sp * n_kb / splits, kb1 = (sp + 1) * n_kb / splits;
        const int b = iter & 1;
        bool ok = mbar_wait(acce + 8 * b, ((iter >> 1) & 1) ^ 1);
        tc_fence_after();
        const uint32_t acc = tmem + static_cast<uint32_t>(b * BN);
        for (int kb = kb0; kb < kb1; kb += KS) {
          ok = ok && mbar_wait(bar_base + 8 * stage, phase);
          if (!__all_sync(0xffffffffu, ok)) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t da = desc0 + static_cast<uint64_t>(stage * (C::STAGE_BYTES >> 4));
            const uint64_t db = da + (C::X_OFFSET >> 4);
#pragma unroll
            for (int j = 0; j < KS; ++j) {
              if (kb + j >= kb1) break;
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                umma_bf16_pair(acc, da + j * (W_BYTES >> 4) + 2 * k, db + j * (C::X_BYTES >> 4) + 2 * k, idesc,
                               (kb > kb0 || j > 0 || k > 0) ? 1u : 0u);
            }
            umma_commit_pair(bar_base + 8 * (STAGES + stage));
          }
          __syncwarp();
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (!__all_sync(0xffffffffu, ok)) {
          atomicExch(a.err, kErrWaitTmaFull);
          *sh_abort = 1;
          break;
        }
        if (elect_one()) umma_commit_pair(accf + 8 * b);
        __syncwarp();
      }
    }
  } else {
    const int wq = warp & 3, hf = warp >> 2;
    const uint32_t trow = tmem + (static_cast<uint32_t>(wq * 32) << 16);
    uint8_t* stg = smem + C::EPI_OFFSET + hf * C::BUFS * EPI_HALF;
    int iter = 0, buf = 0;
    for (int u = pair; u < units; u += n_pairs, ++iter) {
      const int sp = u % splits, tile = u / splits;
      const int ft = 2 * (tile % n_fp) + rank, tt = tile / n_fp;
      const int rows = rows_of(tt), hrows = ((rows + 63) >> 6) << 5;
      const int b = iter & 1;
      const uint32_t acc = trow + static_cast<uint32_t>(b * BN);
      const uint32_t freed = mapa_shared(acce + 8 * b, 0);
      // (after an expired wait the loop runs on without waiting or storing, so that the
      // warps of a half still meet at their named barriers)
      auto ready = [&]() {
        const bool aborted = *sh_abort != 0;
        const bool done = !aborted && mbar_wait(accf + 8 * b, (iter >> 1) & 1);
        if (!done && !aborted) {
          atomicExch(a.err, kErrWaitAccum);
          *sh_abort = 1;
        }
        tc_fence_after();
        return done;
      };
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(freed);
      };
      const int c_lo = hf * hrows, c_hi = min(rows, c_lo + hrows);
      float* slot = nullptr;
      if (KIND == kEpiPartial)
        slot = a.partials + (static_cast<size_t>(ft + n_ft * tt) * splits + sp) * BN * BM;
      if (c_lo < c_hi && ft < n_ft) {
        if constexpr (BN == 64 && kDirect<KIND>)
          drain_direct<KIND>(a, acc, wq, lane, tt * BN, c_lo, c_hi, ft, slot, ready, release);
        else
          drain<KIND, C::BUFS>(a, acc, stg, 1 + hf, wq, lane, tt * BN, c_lo, c_hi, ft, slot, buf, ready, release);
      } else {
        ready();
        release();
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the peer's copies, MMAs and arrivals on this CTA's memory are done
  if (warp == EPI_WARPS + 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 2 * BN);
  }
  stamp_end(a.stamp);
}

template <int BN, int KIND>
cudaError_t launch_one(const CUtensorMap& tm_w, const CUtensorMap& tm_x, const GemmArgs& a, int n_pairs,
                       cudaStream_t s) {
  return launch_ex(gemm_pair_kernel<BN, KIND>, dim3(2 * n_pairs), dim3(THREADS), PairCfg<BN>::TOTAL, s, 2, tm_w, tm_x,
                   a);
}

template <int BN>
cudaError_t launch_bn(const CUtensorMap& tm_w, const CUtensorMap& tm_x, const GemmArgs& a, int n_pairs,
                      cudaStream_t s) {
  if (a.defer) return launch_one<BN, kEpiPartial>(tm_w, tm_x, a, n_pairs, s);
  switch (a.epi.kind) {
    case kEpiF32Bias: return launch_one<BN, kEpiF32Bias>(tm_w, tm_x, a, n_pairs, s);
    case kEpiQKV: return launch_one<BN, kEpiQKV>(tm_w, tm_x, a, n_pairs, s);
    case kEpiResid: return launch_one<BN, kEpiResid>(tm_w, tm_x, a, n_pairs, s);
    case kEpiGelu: return launch_one<BN, kEpiGelu>(tm_w, tm_x, a, n_pairs, s);
    case kEpiGeluTanhf: return launch_one<BN, kEpiGeluTanhf>(tm_w, tm_x, a, n_pairs, s);
    case kEpiScatterF32: return launch_one<BN, kEpiScatterF32>(tm_w, tm_x, a, n_pairs, s);
    case kEpiScore: return launch_one<BN, kEpiScore>(tm_w, tm_x, a, n_pairs, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int BN>
cudaError_t setup_bn() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kern) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<BN>::TOTAL);
  };
  set(gemm_pair_kernel<BN, kEpiF32Bias>);
  set(gemm_pair_kernel<BN, kEpiQKV>);
  set(gemm_pair_kernel<BN, kEpiResid>);
  set(gemm_pair_kernel<BN, kEpiGelu>);
  set(gemm_pair_kernel<BN, kEpiGeluTanhf>);
  set(gemm_pair_kernel<BN, kEpiScatterF32>);
  set(gemm_pair_kernel<BN, kEpiScore>);
  set(gemm_pair_kernel<BN, kEpiPartial>);
  return e;
}

}  // namespace

cudaError_t gemm_pair_setup() {
  cudaError_t e = setup_bn<64>();
  if (e == cudaSuccess) e = setup_bn<128>();
  if (e == cudaSuccess) e = setup_bn<256>();
  return e;
}

cudaError_t launch_gemm_pair(int bn, const CUtensorMap& tm_w, const CUtensorMap& tm_x, const GemmArgs& args,
                             int n_pairs, cudaStream_t s) {
  GemmArgs a = args;
  a.stamp = g_stamp;
  if (bn == 64) return launch_bn<64>(tm_w, tm_x, a, n_pairs, s);
  if (bn == 128) return launch_bn<128>(tm_w, tm_x, a, n_pairs, s);
  if (bn == 256) return launch_bn<256>(tm_w, tm_x, a, n_pairs, s);
  return cudaErrorInvalidValue;
}

}  // namespace ivit
