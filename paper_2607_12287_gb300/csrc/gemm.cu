// GEMM of a few packed rows (incremental calls, up to about 64 updated tokens): Y[r][f] =
// sum_k X[r][k] W[f][k], then an epilogue of GemmEpilogue, as a chain of as few dependent
// steps as the work allows.
//
// A CTA owns 8 NT output features over the whole of K (or one of `vsplit` parts of it, when
// the next layer norm sums the partial results).  Its weights come into shared memory by
// bulk copies before the wait on the previous kernel.  The eight warps split K between them
// in chunks of 32: a lane loads 16 bytes (8 consecutive k) of each of its rows straight from
// L2 into registers, and the matching 16 bytes of each of its features from shared memory;
// taken in the same order on both sides these are the fragments of two mma.m16n8k16 (a dot
// product does not care which k is called which).  So no operand is staged, and the rows cost
// one round trip to L2.  The warps' sums meet in shared memory, in warp order.  Rows beyond
// 32 run as further passes over the resident weights; where one plan serves every row count, a
// second group of CTAs (blockIdx.y) takes every other pass and leaves at once when there is none.
// Two calls of four So400m layers took 1058 us with one group and take 696 with two when all 256
// tokens of a view change, 451 and 371 when 30 % do.  A call of one pass costs no more: two calls
// of 27 layers with 26 rows on average went from 1499 to 1419 us, by those of 33 rows and more.
//
// Bound: latency (wait, rows from L2, MMAs, sum over the warps, store).  mma.sync and not
// tcgen05 because a tcgen05.mma takes at least about 46 cycles however few rows it has, and a
// CTA's whole K in one accumulator is 72 of them in a row (K 1152); here eight warps work on
// eight parts of K at once.  The tcgen05 kernel before it split K over a cluster and paid
// partial tiles through L2, a cluster barrier and a second read.  Measured back to back at 26
// rows of the So400m shapes, before -> now: QKV 6.9 -> 4.0 us, up 7.4 -> 4.5, down (deferred)
// 5.3 -> 3.9; a further 32 rows cost 2.3 to 2.8 us, so the CTA-pair kernel takes over past
// about 64.  Fetching a next pass's rows early made one pass 0.7 us slower (the loop's code
// is on the critical path) and was left out.
#include "gelu.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace ivit {
namespace {

constexpr int WARPS = 8, THREADS = WARPS * 32;
constexpr int CK = 32;    // K of one chunk
constexpr int ROWS = 32;  // rows of one pass
constexpr int DEPTH = 3;  // chunks of rows in flight per warp

// Where feature f of row r of a warp's partial sums is ([ROWS][8 nt]): groups of 8 features are
// exchanged between rows so that the fragments' 8-byte stores of four rows cover all banks.
template <int NT>
__device__ __forceinline__ int red_at(int r, int f) {
  return r * 8 * NT + (f ^ (NT == 4 ? 8 * (r & 3) : NT == 2 ? 8 * ((r >> 1) & 1) : 0));
}
// Bytes from one feature's weights to the next in shared memory: 64 bytes past a multiple of
// 128, so that the 16-byte loads of two features by 8 lanes cover all banks.
__host__ __device__ __forceinline__ int w_pitch(int k) { return (k * 2 + 127) / 128 * 128 + 64; }

__device__ __forceinline__ uint2 pack4(float4 v) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

// K chunks [lo, hi) of split sp.
__device__ __forceinline__ void split_range(int n_chunks, int splits, int sp, int& lo, int& hi) {
  lo = sp * n_chunks / splits;
  hi = (sp + 1) * n_chunks / splits;
}

template <int NT, int KIND>
__global__ void __launch_bounds__(THREADS, 2) gemm_rows_kernel(const GemmArgs a) {
  constexpr int NF = 8 * NT, Q = NF / 4;
  extern __shared__ __align__(128) uint8_t smem[];
  float* red = reinterpret_cast<float*>(smem);  // [WARPS][ROWS][NF]
  uint8_t* ws = smem + WARPS * ROWS * NF * 4;   // [NF][pitch]
  __shared__ __align__(8) uint64_t bar;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int K = a.k, splits = KIND == kEpiPartial ? a.vsplit : 1;
  // The CTAs of the second row group take every other pass; without one they have nothing to do.
  // (The row count comes from the selection kernel, at least two launches back.)
  const int first = blockIdx.y * ROWS;
  if (first > 0 && (a.d_rows ? *a.d_rows : a.m_static) <= first) return;
  const int ft = blockIdx.x / splits, sp = blockIdx.x - ft * splits;
  int c_lo, c_hi;
  split_range((K + CK - 1) / CK, splits, sp, c_lo, c_hi);
  const int k_lo = c_lo * CK, k_hi = min(K, c_hi * CK);
  const int f0 = ft * NF, nf = min(NF, a.n_out - f0);
  const int pitch = w_pitch((c_hi - c_lo) * CK);
  const uint32_t bar_a = smem_u32(&bar), ws_a = smem_u32(ws);

  if (tid == 0) {
    mbar_init(bar_a, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(bar_a, static_cast<uint32_t>(nf * (k_hi - k_lo) * 2));
  }
  __syncwarp();
  if (warp == 0 && lane < nf)
    bulk_load_hint(ws_a + lane * pitch, a.w + static_cast<size_t>(f0 + lane) * K + k_lo,
                   static_cast<uint32_t>((k_hi - k_lo) * 2), bar_a, l2_policy_evict_first());
  // this thread's part of the epilogue: four features of a row
  const int er = tid / Q, f4 = f0 + 4 * (tid - er * Q);
  const bool e_ok = er < ROWS && f4 < a.n_out;
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
  if (KIND != kEpiPartial && e_ok) bias = __ldg(reinterpret_cast<const float4*>(a.epi.bias + f4));
  __syncthreads();  // the barrier exists before anyone waits on it
  const int M = a.d_rows ? *a.d_rows : a.m_static;
  pdl_wait();
  pdl_launch_dependents();
  stamp_begin(a.stamp, blockIdx.x + gridDim.x * blockIdx.y);

  bool ok = true;
  const int n = max(0, (c_hi - c_lo - warp + WARPS - 1) / WARPS);  // this warp's chunks
  const int stride = gridDim.y * ROWS;
  for (int row0 = first; row0 < M; row0 += stride) {
    const int rows = min(ROWS, M - row0);
    const bool two = rows > 16;  // second m16 tile in use
    uint4 x[DEPTH][4];
    const bf16* xp = a.x + static_cast<size_t>(row0 + g) * K + 8 * t;
    auto load = [&](int i, uint4 (&d)[4]) {
      const int k = (c_lo + warp + i * WARPS) * CK;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        d[j] = make_uint4(0, 0, 0, 0);
        if (i < n && g + 8 * j < rows && k + 8 * t < k_hi)
          d[j] = __ldcg(reinterpret_cast<const uint4*>(xp + static_cast<size_t>(8 * j) * K + k));
      }
    };
#pragma unroll
    for (int i = 0; i < DEPTH; ++i) load(i, x[i]);
    int tok = 0;
    const bool by_tok = KIND == kEpiScatterF32 || (KIND == kEpiQKV && f4 >= a.epi.dim);
    if (by_tok && e_ok && er < rows) tok = __ldcg(a.epi.rowtok + row0 + er);
    float acc[2][NT][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[m][j][e] = 0.f;
    if (row0 == first && !mbar_wait(bar_a, 0)) ok = false;  // the weights have landed
    for (int i0 = 0; i0 < n; i0 += DEPTH) {
#pragma unroll
      for (int d = 0; d < DEPTH; ++d) {
        const int i = i0 + d;
        if (i >= n) break;
        const int kr = (warp + i * WARPS) * CK + 8 * t;  // relative to k_lo
        const bool k_ok = k_lo + kr < k_hi;
        uint4 w[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          w[j] = make_uint4(0, 0, 0, 0);
          if (k_ok) w[j] = *reinterpret_cast<const uint4*>(ws + (8 * j + g) * pitch + kr * 2);
        }
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          mma_bf16_16816(acc[0][j], x[d][0].x, x[d][1].x, x[d][0].y, x[d][1].y, w[j].x, w[j].y);
          mma_bf16_16816(acc[0][j], x[d][0].z, x[d][1].z, x[d][0].w, x[d][1].w, w[j].z, w[j].w);
          if (two) {
            mma_bf16_16816(acc[1][j], x[d][2].x, x[d][3].x, x[d][2].y, x[d][3].y, w[j].x, w[j].y);
            mma_bf16_16816(acc[1][j], x[d][2].z, x[d][3].z, x[d][2].w, x[d][3].w, w[j].z, w[j].w);
          }
        }
        load(i + DEPTH, x[d]);
      }
    }
    float* mine = red + warp * ROWS * NF;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      if (m == 1 && !two) break;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int f = 8 * j + 2 * t;
        *reinterpret_cast<float2*>(mine + red_at<NT>(16 * m + g, f)) = make_float2(acc[m][j][0], acc[m][j][1]);
        *reinterpret_cast<float2*>(mine + red_at<NT>(16 * m + g + 8, f)) = make_float2(acc[m][j][2], acc[m][j][3]);
      }
    }
    __syncthreads();
    if (e_ok && er < rows && ok) {
      const float* p = red + red_at<NT>(er, f4 - f0);
      float4 y = *reinterpret_cast<const float4*>(p);
#pragma unroll
      for (int w = 1; w < WARPS; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(p + w * ROWS * NF);
        y.x += v.x;
        y.y += v.y;
        y.z += v.z;
        y.w += v.w;
      }
      if (KIND != kEpiPartial) {
        y.x += bias.x;
        y.y += bias.y;
        y.z += bias.z;
        y.w += bias.w;
      }
      const int r = row0 + er;
      if (KIND == kEpiPartial) {
        const int tile = f4 / 128 + (a.n_out + 127) / 128 * (row0 / ROWS);
        *reinterpret_cast<float4*>(a.partials + ((static_cast<size_t>(tile) * splits + sp) * ROWS + er) * 128 +
                                   f4 % 128) = y;
      } else if (KIND == kEpiQKV) {
        const int D = a.epi.dim;
        bf16* dst = f4 < D ? a.epi.out_bf16 + static_cast<size_t>(r) * D + f4
                           : (f4 < 2 * D ? a.epi.cache_k + static_cast<size_t>(tok) * D + (f4 - D)
                                         : a.epi.cache_v + static_cast<size_t>(tok) * D + (f4 - 2 * D));
        *reinterpret_cast<uint2*>(dst) = pack4(y);
      } else if (KIND == kEpiGelu || KIND == kEpiGeluTanhf) {
        const int mode = a.epi.gelu_mode;
        y = make_float4(gelu_f<KIND>(y.x, mode), gelu_f<KIND>(y.y, mode), gelu_f<KIND>(y.z, mode), gelu_f<KIND>(y.w, mode));
        *reinterpret_cast<uint2*>(a.epi.out_bf16 + static_cast<size_t>(r) * a.epi.ld_out + f4) = pack4(y);
      } else if (KIND == kEpiResid) {
        red_add_f32x4(a.epi.out_f32 + static_cast<size_t>(r) * a.epi.ld_out + f4, y);
      } else {  // kEpiScatterF32
        *reinterpret_cast<float4*>(a.epi.out_f32 + static_cast<size_t>(tok) * a.epi.ld_out + f4) = y;
      }
    }
    if (row0 + stride < M) __syncthreads();  // the sums are read before the next pass writes
  }
  if (M <= 0 && !mbar_wait(bar_a, 0)) ok = false;  // no copy in flight at exit
  if (!ok && tid == 0) atomicExch(a.err, kErrWaitTmaFull);
  stamp_end(a.stamp, blockIdx.x + gridDim.x * blockIdx.y);
}

size_t smem_bytes(int nt, int k, int splits) {
  const int chunks = ((k + CK - 1) / CK + splits - 1) / splits;
  return static_cast<size_t>(WARPS) * ROWS * 8 * nt * 4 + static_cast<size_t>(8 * nt) * w_pitch(chunks * CK);
}

template <int NT>
cudaError_t launch_nt(const GemmArgs& a, cudaStream_t s) {
  const int splits = a.defer ? a.vsplit : 1;
  const dim3 grid((a.n_out + 8 * NT - 1) / (8 * NT) * splits, a.row_groups);
  const size_t smem = smem_bytes(NT, a.k, splits);
  auto launch = [&](auto kern) { return launch_ex(kern, grid, dim3(THREADS), smem, s, 1, a); };
  if (a.defer) return launch(gemm_rows_kernel<NT, kEpiPartial>);
  switch (a.epi.kind) {
    case kEpiQKV: return launch(gemm_rows_kernel<NT, kEpiQKV>);
    case kEpiResid: return launch(gemm_rows_kernel<NT, kEpiResid>);
    case kEpiGelu: return launch(gemm_rows_kernel<NT, kEpiGelu>);
    case kEpiGeluTanhf: return launch(gemm_rows_kernel<NT, kEpiGeluTanhf>);
    case kEpiScatterF32: return launch(gemm_rows_kernel<NT, kEpiScatterF32>);
    default: return cudaErrorInvalidValue;
  }
}

template <int NT>
cudaError_t setup_nt() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kern) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_ROWS_SMEM_MAX);
  };
  set(gemm_rows_kernel<NT, kEpiPartial>);
  set(gemm_rows_kernel<NT, kEpiQKV>);
  set(gemm_rows_kernel<NT, kEpiResid>);
  set(gemm_rows_kernel<NT, kEpiGelu>);
  set(gemm_rows_kernel<NT, kEpiGeluTanhf>);
  set(gemm_rows_kernel<NT, kEpiScatterF32>);
  return e;
}

}  // namespace

// Many-tile form: gemm_pair.cu (CTA pairs).  Below: this kernel's entry points.

size_t gemm_rows_smem(int nt, int k, int splits) { return smem_bytes(nt, k, splits); }

cudaError_t gemm_rows_setup() {
  cudaError_t e = setup_nt<1>();
  if (e == cudaSuccess) e = setup_nt<2>();
  if (e == cudaSuccess) e = setup_nt<3>();
  if (e == cudaSuccess) e = setup_nt<4>();
  return e;
}

cudaError_t launch_gemm_rows(int nt, const GemmArgs& args, cudaStream_t s) {
  GemmArgs a = args;
  a.stamp = g_stamp;
  switch (nt) {
    case 1: return launch_nt<1>(a, s);
    case 2: return launch_nt<2>(a, s);
    case 3: return launch_nt<3>(a, s);
    case 4: return launch_nt<4>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ivit
