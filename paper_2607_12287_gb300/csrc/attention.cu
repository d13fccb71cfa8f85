// Attention of the updated queries of every view over all N keys of that view, on the
// tensor cores (Sec. III-B: attention is computed only for the updated tokens; Eq. 5:
// the keys and values of reused tokens come from the per-layer cache):
//
//   O = softmax(Q K^T / sqrt(dh)) V          per (view, head).
//
// Work item = (view v, head h, query tile of up to 128 packed updated rows).  Every CTA
// derives the list of items from the device-resident row offsets (written by the selection
// kernel) and walks it with a stride, so one launch shape serves every row count and the
// launch can sit in a CUDA graph.  Per item the keys are walked in blocks of KB (128, 96 or
// 64 by head width, so that S, P and O of a block fit in 256 tensor-memory columns) with an
// online softmax.  Two CTAs share an SM: while one's warps take exponentials the other's
// MMAs run.
//
// Bound: the exponentials and the softmax's other arithmetic (one row per thread) at large
// row counts, the chain K -> S -> softmax -> P V of an item at small ones.  Measured with 16
// heads of 72 against the kernel before it (one CTA per SM or a cluster splitting the keys,
// softmax and MMAs in turn, P through shared memory): 32 views x 1024 queries x 1024 keys
// 690 -> 218 us (709 TFLOP/s), 32 x 96 queries 158 -> 38 us.  Of that, the order of the items
// (query tiles of a head together, K/V from L2 instead of DRAM) and the narrow second slice
// took 327 to 218 us.
//
// Warps of a CTA:
//   4      TMA: Q tile of 128 rows, then K and V blocks through a ring of 4 to 7 tiles.  The
//          maps are [rows][heads][dh]: the columns past a head's dh are out of bounds, zero
//          in shared memory and not fetched.  Columns 0..63 form one slice with 128-byte
//          swizzle, the rest (8 of a 72-wide head) a second one as narrow as a swizzle
//          allows, which leaves room for two more tiles.
//   5      MMA: S = Q K^T (fp32, tensor memory) of block i+1 is issued before O += P V of
//          block i, so it runs while block i's softmax finishes; P is read from tensor
//          memory, V is the B operand in MN-major form.
//   0 - 3  softmax, thread = query row = tensor-memory lane: S into registers, P = 2^((S - m) c)
//          (c = log2(e) / sqrt(dh)) rounded to bf16 into tensor memory, l = the sum of those
//          values.  The reference m is the row's running maximum, moved (and O, l rescaled)
//          only when a block exceeds it by more than 2^8, which keeps P in bf16's and the
//          sums in fp32's range; the result does not depend on the reference.  At the end
//          O / l goes to global memory.
#include "attention.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace ivit {
namespace {

constexpr int AQ = 128;             // queries per item (MMA M)
constexpr int THREADS = 192;
constexpr int SMEM_HALF = 113 * 1024;  // two CTAs share an SM
constexpr float RESCALE = 8.f;      // log2 of the growth that moves the reference maximum

template <int DHP>
struct AttnCfg {
  static constexpr int KB = attention_key_block(DHP);
  // A row's columns past 64 form a second slice, as narrow as a swizzle allows.
  static constexpr int W2 = attention_slice2(DHP);
  static constexpr int Q1 = AQ * 128, Q2 = AQ * W2 * 2;                // bytes of the slices of Q
  static constexpr int T1 = KB * 128, TILE = (T1 + KB * W2 * 2 + 1023) / 1024 * 1024;  // of a K or V block
  static constexpr int T_BYTES = T1 + KB * W2 * 2;
  static constexpr int TM_O = KB, TM_P = KB + DHP, TM_COLS = 256;      // S at column 0
  static_assert(TM_P + KB / 2 <= TM_COLS, "tensor memory of one CTA");
  static constexpr int OFF_RING = Q1 + Q2;
  static constexpr int RING = (SMEM_HALF - OFF_RING - 1024 - 512) / TILE < 8 ? (SMEM_HALF - OFF_RING - 1024 - 512) / TILE : 8;
  static constexpr int OFF_BAR = OFF_RING + RING * TILE;
  static constexpr int OFF_CUM = OFF_BAR + 256;  // [sv + 1] items before each view
  static constexpr int BYTES = OFF_CUM + 1024;   // alignment slack
};

// 32 columns of S (bits) -> 16 packed bf16 pairs of P; l gets the rounded values.
__device__ __forceinline__ void exp_chunk(const uint32_t* s, float sc, float mo, uint32_t* pk, float2 (&l)[2]) {
  const float2 c2 = make_float2(sc, sc), m2 = make_float2(-mo, -mo);
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    const float2 t = fma_f32x2(make_float2(__uint_as_float(s[2 * u]), __uint_as_float(s[2 * u + 1])), c2, m2);
    const __nv_bfloat162 b = __floats2bfloat162_rn(ex2(t.x), ex2(t.y));
    const uint32_t w = *reinterpret_cast<const uint32_t*>(&b);
    // (bf16 widens to fp32 by its bits; the normaliser sums the values the MMA multiplies)
    l[u & 1] = add_f32x2(l[u & 1], make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)));
    pk[u] = w;
  }
}

// Shared-memory descriptor of a slice whose rows are W2 columns (and one swizzle span) wide:
// groups of 8 rows follow each other.  For a K-major operand the rows are its M or N index,
// for an MN-major one (V) its K index.
template <int W2>
__device__ __forceinline__ uint64_t sdesc_rows(uint32_t saddr) {
  constexpr uint32_t group = 8 * W2 * 2;
  uint64_t d = sdesc_sw128(saddr, group, group) & ~(static_cast<uint64_t>(7) << 61);
  return d | (static_cast<uint64_t>(W2 == 16 ? 6 : W2 == 32 ? 4 : 2) << 61);  // 32-, 64-, 128-byte swizzle
}

template <int DHP>
__global__ void __launch_bounds__(THREADS, 2)
    attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                        const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_q2,
                        const __grid_constant__ CUtensorMap tm_k2, const __grid_constant__ CUtensorMap tm_v2,
                        const AttnTcArgs a) {
  using C = AttnCfg<DHP>;
  constexpr int KB = C::KB, RING = C::RING, W2 = C::W2;
  extern __shared__ uint8_t at_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(at_raw) + 1023) &
                                           ~static_cast<uintptr_t>(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = a.n_tok;
  const int nb = (N + KB - 1) / KB;  // key blocks of an item
  const uint32_t sb = smem_u32(sm), bar = sb + C::OFF_BAR;
  const uint32_t q_full = bar, q_empty = bar + 8, s_full = bar + 16, s_free = bar + 24, p_ready = bar + 32,
                 o_done = bar + 40, o_free = bar + 48, t_full = bar + 56, t_empty = t_full + 8 * RING;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + C::OFF_BAR + 56 + 16 * RING);
  volatile int* sh_abort = reinterpret_cast<volatile int*>(tslot + 1);
  int* cum = reinterpret_cast<int*>(sm + C::OFF_CUM);

  if (tid == 0) {
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    mbar_init(s_full, 1);
    mbar_init(s_free, 4);
    mbar_init(p_ready, 4);
    mbar_init(o_done, 1);
    mbar_init(o_free, 4);
    for (int i = 0; i < RING; ++i) {
      mbar_init(t_full + 8 * i, 1);
      mbar_init(t_empty + 8 * i, 1);
    }
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
    if (W2 > 0) {
      tma_prefetch_desc(&tm_q2);
      tma_prefetch_desc(&tm_k2);
      tma_prefetch_desc(&tm_v2);
    }
    *sh_abort = 0;
  }
  // The row offsets come from the selection kernel, at least two launches back (every kernel
  // of the library triggers its dependents only after its own wait).
  attention_items(a, AQ, cum);
  if (warp == 5) {
    tmem_alloc(smem_u32(tslot), C::TM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  pdl_wait();  // queries and this call's K/V rows (QKV kernel) are visible from here
  pdl_launch_dependents();
  stamp_begin(a.stamp);

  // Every wait is bounded; after one has expired no role waits again and all leave.
  auto wait = [&](uint32_t b, uint32_t parity) {
    if (*sh_abort) return false;
    if (mbar_wait(b, parity)) return true;
    atomicExch(a.err, kErrWaitTmaFull);
    *sh_abort = 1;
    return false;
  };

  const int n_items = cum[a.sv];
  int s = blockIdx.x;
  if (warp == 4) {
    const uint64_t pol_q = l2_policy_evict_first(), pol_kv = l2_policy_evict_last();
    uint32_t t = 0;  // K / V tiles so far
    for (uint32_t n = 0; s < n_items; ++n, s += gridDim.x) {
      const AttnItem it = attention_item(s, AQ, cum, a);
      if (!__all_sync(0xffffffffu, wait(q_empty, (n & 1) ^ 1))) break;
      if (elect_one()) {
        mbar_arrive_expect_tx(q_full, C::Q1 + C::Q2);
        tma_load_3d(sb, &tm_q, 0, it.h, it.r0, q_full, pol_q);
        if (W2 > 0) tma_load_3d(sb + C::Q1, &tm_q2, 64, it.h, it.r0, q_full, pol_q);
      }
      __syncwarp();
      bool ok = true;
      for (int i = 0; i < 2 * nb && ok; ++i, ++t) {  // K and V of block i / 2
        const uint32_t slot = t % RING;
        ok = __all_sync(0xffffffffu, wait(t_empty + 8 * slot, ((t / RING) & 1) ^ 1));
        if (ok && elect_one()) {
          const uint32_t dst = sb + C::OFF_RING + slot * C::TILE, full = t_full + 8 * slot;
          const int row = it.v * N + (i >> 1) * KB;
          mbar_arrive_expect_tx(full, C::T_BYTES);
          tma_load_3d(dst, (i & 1) ? &tm_v : &tm_k, 0, it.h, row, full, pol_kv);
          if (W2 > 0) tma_load_3d(dst + C::T1, (i & 1) ? &tm_v2 : &tm_k2, 64, it.h, row, full, pol_kv);
        }
        __syncwarp();
      }
      if (!ok) break;
    }
  } else if (warp == 5) {
    uint32_t j0 = 0;  // key blocks of the earlier items
    bool ok = true;
    for (uint32_t n = 0; ok && s < n_items; ++n, s += gridDim.x, j0 += nb) {
      ok = __all_sync(0xffffffffu, wait(q_full, n & 1));
      for (int i = 0; i <= nb && ok; ++i) {
        if (i < nb) {  // S of block i
          const uint32_t j = j0 + i, t = 2 * j, slot = t % RING;
          ok = __all_sync(0xffffffffu, wait(t_full + 8 * slot, (t / RING) & 1) && wait(s_free, (j & 1) ^ 1));
          if (!ok) break;
          tc_fence_after();
          const uint32_t id = idesc_bf16_f32(AQ, (min(KB, N - i * KB) + 15) & ~15);
          if (elect_one()) {
            const uint32_t kt = sb + C::OFF_RING + slot * C::TILE;
#pragma unroll
            for (int u = 0; u < DHP / 16; ++u)
              umma_bf16(tmem,
                        u < 4 ? sdesc_kmajor_sw128(sb + u * 32) : sdesc_rows<W2>(sb + C::Q1 + (u - 4) * 32),
                        u < 4 ? sdesc_kmajor_sw128(kt + u * 32) : sdesc_rows<W2>(kt + C::T1 + (u - 4) * 32), id, u > 0);
            umma_commit(t_empty + 8 * slot);
            umma_commit(s_full);
            if (i == nb - 1) umma_commit(q_empty);
          }
          __syncwarp();
        }
        if (i > 0) {  // O += P V of block i - 1
          const uint32_t j = j0 + i - 1, t = 2 * j + 1, slot = t % RING;
          ok = __all_sync(0xffffffffu, wait(t_full + 8 * slot, (t / RING) & 1) && wait(p_ready, j & 1) &&
                                           (i > 1 || wait(o_free, (n & 1) ^ 1)));
          if (!ok) break;
          tc_fence_after();
          const int steps = (min(KB, N - (i - 1) * KB) + 15) >> 4;
          if (elect_one()) {
            const uint32_t vt = sb + C::OFF_RING + slot * C::TILE;
            const uint32_t id0 = idesc_bf16_f32_bmn(AQ, DHP > 64 ? 64 : DHP);
            const uint32_t id1 = idesc_bf16_f32_bmn(AQ, DHP > 64 ? DHP - 64 : 16);
            for (int u = 0; u < steps; ++u) {
              const uint32_t acc = (i > 1 || u > 0) ? 1u : 0u;
              umma_bf16_ts(tmem + C::TM_O, tmem + C::TM_P + u * 8, sdesc_sw128(vt + u * 2048, 1024, 1024), id0, acc);
              if (DHP > 64)
                umma_bf16_ts(tmem + C::TM_O + 64, tmem + C::TM_P + u * 8,
                             sdesc_rows<W2>(vt + C::T1 + u * 32 * W2), id1, acc);
            }
            umma_commit(t_empty + 8 * slot);
            umma_commit(o_done);
          }
          __syncwarp();
        }
      }
    }
  } else {
    const uint32_t trow = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    const float sc = rsqrtf(static_cast<float>(a.dh)) * 1.4426950408889634f;  // log2(e) / sqrt(dh)
    uint32_t j = 0;  // key blocks so far
    bool ok = true;
    auto arrive = [&](uint32_t b) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b);
    };
    for (; ok && s < n_items; s += gridDim.x) {
      const AttnItem it = attention_item(s, AQ, cum, a);
      const bool wrow = warp * 32 < it.nq;  // warp-uniform: a warp of padding rows only keeps step
      float m_ref = -INFINITY;
      float2 l[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      for (int i = 0; i < nb; ++i, ++j) {
        if (!(ok = __all_sync(0xffffffffu, wait(s_full, j & 1)))) break;
        tc_fence_after();
        if (!wrow) {
          arrive(s_free);
          if (!(ok = __all_sync(0xffffffffu, j == 0 || wait(o_done, (j & 1) ^ 1)))) break;
          arrive(p_ready);
          continue;
        }
        uint32_t r[KB];
#pragma unroll
        for (int c = 0; c < KB; c += 32) tmem_ld32_async(trow + c, *reinterpret_cast<uint32_t(*)[32]>(r + c));
#pragma unroll
        for (int c = 0; c < KB; c += 32) tmem_ld_wait_regs(*reinterpret_cast<uint32_t(*)[32]>(r + c));
        arrive(s_free);
        const int gn = N - i * KB;
        if (gn < KB) {
#pragma unroll
          for (int c = 0; c < KB; ++c)
            if (c >= gn) r[c] = 0xff800000u;  // -inf: P = 0
        }
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < KB; ++c) mx[c & 3] = fmaxf(mx[c & 3], __uint_as_float(r[c]));
        const float m_blk = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        float alpha = 1.f;
        const bool grow = i > 0 && (m_blk - m_ref) * sc > RESCALE;
        if (i == 0 || grow) {
          alpha = ex2((m_ref - m_blk) * sc);
          m_ref = m_blk;
        }
        const float mo = m_ref == -INFINITY ? 0.f : m_ref * sc;  // (scores of -inf alone so far: P = 0)
        const bool rescale = __any_sync(0xffffffffu, grow);
        if (rescale) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            l[e].x *= alpha;
            l[e].y *= alpha;
          }
        }
        uint32_t pk[KB / 2];
#pragma unroll
        for (int c = 0; c < KB; c += 32) exp_chunk(r + c, sc, mo, pk + c / 2, l);
        // P and O are free once the previous block's (or item's) P V has run
        if (!(ok = __all_sync(0xffffffffu, j == 0 || wait(o_done, (j & 1) ^ 1)))) break;
        tc_fence_after();
        if (rescale) {
#pragma unroll
          for (int d = 0; d < DHP; d += 16) {
            uint32_t o[16];
            tmem_ld16_async(trow + C::TM_O + d, o);
            tmem_ld_wait();
            tmem_regs_after_wait16(o);
#pragma unroll
            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st16(trow + C::TM_O + d, o);
          }
        }
#pragma unroll
        for (int c = 0; c < KB / 2; c += 16) tmem_st16(trow + C::TM_P + c, pk + c);
        tmem_st_wait();
        arrive(p_ready);
      }
      if (!ok || !(ok = __all_sync(0xffffffffu, wait(o_done, (j & 1) ^ 1)))) break;
      tc_fence_after();
      if (wrow) {
        const float inv = 1.f / ((l[0].x + l[0].y) + (l[1].x + l[1].y));
        const int row = warp * 32 + lane;
        bf16* orow = a.o + static_cast<size_t>(it.r0 + row) * a.dim + it.h * a.dh;
#pragma unroll
        for (int d = 0; d < DHP; d += 16) {
          uint32_t o[16];
          tmem_ld16_async(trow + C::TM_O + d, o);
          tmem_ld_wait();
          tmem_regs_after_wait16(o);
#pragma unroll
          for (int h8 = 0; h8 < 16; h8 += 8) {
            uint4 u;
            uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(o[h8 + 2 * e]) * inv,
                                                             __uint_as_float(o[h8 + 2 * e + 1]) * inv);
              w[e] = *reinterpret_cast<const uint32_t*>(&b);
            }
            if (row < it.nq && d + h8 < a.dh) *reinterpret_cast<uint4*>(orow + d + h8) = u;
          }
        }
      }
      arrive(o_free);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 5) tmem_dealloc(tmem, C::TM_COLS);
  stamp_end(a.stamp);
}

}  // namespace

cudaError_t attention_tc_setup() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kern, int bytes) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes + 4 * (MAX_VIEWS + 1));
  };
  set(attention_tc_kernel<16>, AttnCfg<16>::BYTES);
  set(attention_tc_kernel<32>, AttnCfg<32>::BYTES);
  set(attention_tc_kernel<48>, AttnCfg<48>::BYTES);
  set(attention_tc_kernel<64>, AttnCfg<64>::BYTES);
  set(attention_tc_kernel<80>, AttnCfg<80>::BYTES);
  set(attention_tc_kernel<96>, AttnCfg<96>::BYTES);
  set(attention_tc_kernel<112>, AttnCfg<112>::BYTES);
  set(attention_tc_kernel<128>, AttnCfg<128>::BYTES);
  return e;
}

cudaError_t launch_attention_tc(const AttnMaps& q, const AttnMaps& k, const AttnMaps& v, const AttnTcArgs& a,
                                int num_sms, cudaStream_t s) {
  if (a.sv > MAX_VIEWS) return cudaErrorInvalidValue;
  const int grid = max(1, min(a.sv * a.heads * ((a.n_tok + AQ - 1) / AQ), 2 * num_sms));
  auto launch = [&](auto kern, size_t bytes) {
    return launch_ex(kern, dim3(grid), dim3(THREADS), bytes + 4 * (a.sv + 1), s, 1, q.lo, k.lo, v.lo, q.hi, k.hi, v.hi,
                     a);
  };
  switch ((a.dh + 15) & ~15) {
    case 16: return launch(attention_tc_kernel<16>, AttnCfg<16>::BYTES);
    case 32: return launch(attention_tc_kernel<32>, AttnCfg<32>::BYTES);
    case 48: return launch(attention_tc_kernel<48>, AttnCfg<48>::BYTES);
    case 64: return launch(attention_tc_kernel<64>, AttnCfg<64>::BYTES);
    case 80: return launch(attention_tc_kernel<80>, AttnCfg<80>::BYTES);
    case 96: return launch(attention_tc_kernel<96>, AttnCfg<96>::BYTES);
    case 112: return launch(attention_tc_kernel<112>, AttnCfg<112>::BYTES);
    case 128: return launch(attention_tc_kernel<128>, AttnCfg<128>::BYTES);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ivit
