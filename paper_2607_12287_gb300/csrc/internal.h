// Kernel launch interfaces shared by the engine and the kernel translation units.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ivit {

using bf16 = __nv_bfloat16;

// Programmatic dependent launch for every kernel of the library (on by default; the
// IVIT_NO_PDL environment variable turns it off at handle creation).
extern bool g_use_pdl;

// Stamp block (timeline mode) the next launch of this host thread passes to its kernel:
// [kStampCtas][2] global times, or null.  Set by the engine before each launch.
extern thread_local unsigned long long* g_stamp;

// cudaLaunchKernelEx with optional cluster width and the PDL attribute.
template <typename... KArgs, typename... Args>
cudaError_t launch_ex(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                      unsigned cluster_x, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (cluster_x > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster_x;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (g_use_pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args&&>(args)...);
}

// ------------------------------------------------------------------ GEMM (tcgen05)
// Y[r][f] = sum_k X[r][k] * W[f][k] for r < M rows, f < Nout features, then an
// epilogue.  W is the weight matrix in Linear layout [Nout][K] (bf16, K-major), X the
// packed activation rows [M][K] (bf16, K-major).
enum EpiKind : int {
  kEpiF32Bias = 0,  // out_f32[r][f] = y + bias[f]
  kEpiQKV = 1,      // f <  D: out_bf16[r][f] = y + b (queries, packed rows)
                    // f < 2D: cache_k[rowtok[r]][f-D], else cache_v[rowtok[r]][f-2D]  (Eq. 5)
  kEpiResid = 2,    // out_f32[r][f] += y + bias[f]  (residual stream, fp32)
  kEpiGelu = 3,     // out_bf16[r][f] = gelu(y + bias[f])
  kEpiScatterF32 = 4,  // out_f32[rowtok[r]][f] = y + bias[f]  (per-token output cache)
  kEpiScore = 6,       // out_f32[r][f] = y + bias[f], and sums for the cosine of row r with its old
                       // content: score[feature tile of 128 * m_static + r] (Eq. 3)
  kEpiGeluTanhf = 7,   // as kEpiGelu, tanh form, with tanhf in place of the hardware's tanh
  kEpiPartial = 5,     // a K split's fp32 tile, left in the scratch (GemmArgs::defer)
};

struct GemmEpilogue {
  int kind = kEpiF32Bias;
  const float* bias = nullptr;   // [Nout]
  float* out_f32 = nullptr;      // kEpiF32Bias / kEpiResid, row stride ld_out
  bf16* out_bf16 = nullptr;      // kEpiGelu / kEpiQKV (queries), row stride ld_out
  bf16* cache_k = nullptr;       // kEpiQKV: this layer's key cache [SV*N][D]
  bf16* cache_v = nullptr;       // kEpiQKV: this layer's value cache [SV*N][D]
  const int* rowtok = nullptr;   // kEpiQKV: packed row -> token index v*N + i
  float4* score = nullptr;       // kEpiScore: (<new, old>, |new|^2, |old|^2, 0) over 128 features
  int dim = 0;                   // kEpiQKV: D
  int gelu_mode = 0;             // kEpiGelu: 0 tanh form, 1 erf form
  int ld_out = 0;
};

struct GemmArgs {
  int n_out = 0;                 // Nout
  int k = 0;                     // K
  const int* d_rows = nullptr;   // device row count M (nullptr: use m_static)
  int m_static = 0;
  int* err = nullptr;            // device error word
  float* partials = nullptr;     // scratch of a deferred launch (global memory, stays in L2)
  // With defer set, K is split over vsplit consecutive CTAs (or pairs) and
  // the partial tiles are left in the scratch, slot (tile * vsplit + split) of fp32
  // [rows per tile][128] with tile = feature tile + n_ft * row tile; the kernel neither
  // reduces them nor runs the epilogue: the next kernel sums them (layernorm_sum, for the
  // residual epilogue).
  int defer = 0;
  int vsplit = 0;
  int row_groups = 1;            // few-row GEMM: CTAs per feature tile and split, 1 or 2
  unsigned long long* stamp = nullptr;  // timeline stamps of this launch (or null)
  const bf16* w = nullptr;       // W and X themselves, for the kernel that uses no TMA maps
  const bf16* x = nullptr;       // (gemm_rows)
  GemmEpilogue epi;
};

// A residual update x += bias + sum_s partial_s still split over the scratch slots of a
// deferred GEMM (see GemmArgs::defer).
struct PendingSum {
  const float* partials = nullptr;  // the GEMM's scratch
  const float* bias = nullptr;      // [dim]
  int csize = 0;                    // splits, 2..16
  int bn = 0;                       // rows per row tile
  int n_ft = 0;                     // feature tiles of 128
};

// The GEMM over CTA pairs (cta_group::2), tiles of 256 features x bn rows (64, 128 or
// 256; tm_x boxes of bn / 2 rows), walked by n_pairs persistent pairs.  With defer set (and vsplit >= 1) K is split
// vsplit ways and the partial tiles stay in the scratch, as described at GemmArgs::defer.
cudaError_t gemm_pair_setup();
cudaError_t launch_gemm_pair(int bn, const CUtensorMap& tm_w, const CUtensorMap& tm_x, const GemmArgs& a,
                             int n_pairs, cudaStream_t s);

// The same GEMM for a few rows: CTAs of 8 nt features (nt 1..4), rows in passes of 32, every
// epilogue but kEpiF32Bias and kEpiScore, row_groups CTAs side by side for the passes.  With defer set, K is split vsplit ways and the slots have 32 rows.
// k a multiple of 8.
constexpr int GEMM_ROWS_SMEM_MAX = 160 * 1024;
size_t gemm_rows_smem(int nt, int k, int splits);
cudaError_t gemm_rows_setup();
cudaError_t launch_gemm_rows(int nt, const GemmArgs& a, cudaStream_t s);

// ------------------------------------------------------- persistent encoder (small M)
struct LayerParams {
  const float *bqkv, *bo, *b1, *b2, *ln1g, *ln1b, *ln2g, *ln2b;
};

struct PersistentArgs {
  int N, D, F, H, dh, L, SV, M_max;
  float eps;
  int gelu;
  const int* cu_rows;             // [SV+1], cu_rows[SV] = updated rows M
  const int* rowtok;              // [M] packed row -> token v*N + i
  const CUtensorMap* wmaps;       // [L][4] weight maps (qkv, out, up, down), device memory
  const CUtensorMap* xmaps;       // [3] activation maps (xn, o, h), device memory
  const CUtensorMap* kvmaps;      // [L][2] key/value cache maps, box [N rows][dh], device memory
  const LayerParams* layers;      // [L], device memory
  const float *lnfg, *lnfb;
  float* x;                       // fp32 residual stream [M_max][D]
  bf16 *xn, *q, *o, *h, *cacheK, *cacheV, *tok_out;
  float* part;                    // K-split partial tiles
  unsigned* gbar;                 // [count, generation, abort], zero at launch
  int* err;
  unsigned long long* trace;      // optional: [0] count, then phase-exit times of CTA 0
};

size_t persistent_smem_bytes(int n_tok, int head_dim);
size_t persistent_part_floats(int max_items);
cudaError_t persistent_setup(size_t smem);
int persistent_max_ctas(size_t smem);
// Cooperative launch (all CTAs resident); fails if the grid cannot be resident.
cudaError_t launch_persistent(const PersistentArgs& a, int grid, size_t smem, cudaStream_t s);

// ------------------------------------------------ weight-streaming encoder (small M)
struct StreamArgs {
  int N, D, F, H, dh, L, SV, M_max;
  float eps;
  int gelu;
  int ring_stages;                // weight ring depth (16 KB stages), >= the k-blocks of a task
  int region_bytes;               // activation operand / attention region of shared memory
  int att_groups;                 // query groups per (view, head)
  int splits[4];                  // K splits of the QKV, out-proj, MLP-up and MLP-down GEMMs
  int qkv_tiles;                  // 128-feature tiles of the QKV GEMM
  int n_barriers;                 // grid barriers per launch (7 L)
  const int* cu_rows;             // [SV+1], cu_rows[SV] = updated rows M
  const int* rowtok;              // [M] packed row -> token v*N + i
  const CUtensorMap* wmaps;       // [L][4] weights (qkv, out, up, down), box 64 x 128, 128B swizzle
  const CUtensorMap* bmaps;       // [3] LN output xn, attention output o, MLP hidden h; box 64 x 32
  const CUtensorMap* kvmaps;      // [L][2] key / value caches, box dh x N, no swizzle
  const LayerParams* layers;      // [L], device memory
  const float *lnfg, *lnfb;
  float* x;                       // fp32 residual stream [M_max][D] (packed rows)
  bf16 *xn, *q, *o, *h, *cacheK, *cacheV, *tok_out;
  float* part;                    // split partials [splits][M_max][n_out] of the current GEMM
  unsigned* sync;                 // [0] barrier count, [2] abort, [4 + ...] tile counters of the
                                  // QKV and MLP-up GEMMs [L][tiles][passes]; zeroed per launch
  int* err;
  // Optional timeline (IVIT_TRACE): [n_barriers][G] barrier arrival times,
  // [n_barriers] barrier exit times of CTA 0, [G][8][8] per-CTA accumulators.
  unsigned long long* trace;
};

// k-blocks (64 wide) of one task of a GEMM with K = k split `splits` ways.
int stream_task_kblocks(int k, int splits);
// Bytes of the activation operand / attention region (1 KB multiple).
size_t stream_region_bytes(int max_task_kblocks, int n_tok, int head_dim);
// Dynamic shared memory of one CTA with `ring_stages` 16 KB weight stages.
size_t stream_smem_bytes(int ring_stages, size_t region);
// Most weight stages that fit beside the region within `smem_limit` bytes (<= 16).
int stream_ring_stages_for(size_t smem_limit, size_t region);
// Largest model width a row stage holds in registers.
int stream_max_dim();
// Updated rows per pass of a GEMM task.
int stream_rows_per_pass();
cudaError_t stream_setup(size_t smem);
int stream_max_ctas(size_t smem);
// Cooperative launch (all CTAs resident); fails if the grid cannot be resident.
cudaError_t launch_stream(const StreamArgs& a, int grid, size_t smem, cudaStream_t s);

// ------------------------------------------------------------------- other kernels
struct ColdMask {
  uint32_t bits[128];  // bit v set: view v is cold (updates every token); up to 4096 views
};

cudaError_t launch_patchify(const uint8_t* frames, bf16* patches, int sv, int img_h, int img_w,
                            int patch, int kpad, cudaStream_t s);

cudaError_t launch_score(const float* e_t, float* e_ref, float* sims, int rows, int dim,
                         int copy_ref, cudaStream_t s);

// (scores from sims, or with parts from n_parts sums [n_parts][sv * n_tok] as the embedding GEMM leaves them)
cudaError_t launch_select(const float* sims, const float4* parts, int n_parts, int n_tok, int sv, int mode, float tau, int topk,
                          const ColdMask& cold, int* idx, int* counts, int* cu_rows, int* done_ctr,
                          cudaStream_t s);

// Copies the final tokens (bytes a multiple of 16, out aligned to 16) and the views' counts to the
// caller, both in this GPU's memory; either destination may be null.
cudaError_t launch_outputs(const bf16* tok, void* out, size_t bytes, const int* counts, int* user_counts, int sv,
                           int num_sms, cudaStream_t s);

// The selection's ascending token lists idx [sv][n_tok] and the views' packed-row offsets
// cu_rows [sv + 1]; idx null: none.
struct RowLists {
  const int* idx = nullptr;
  const int* cu_rows = nullptr;
  int sv = 0, n_tok = 0;
};

// Row-count bands of an incremental call's CUDA graph: the launch plans of band b are
// made for at most ub[b] updated rows; the graph's switch node runs the body of the
// smallest band that holds the call's row count.
struct RowBands {
  unsigned long long handle = 0;  // cudaGraphConditionalHandle of the switch node (0: none)
  int n = 0;
  int ub[4] = {0, 0, 0, 0};
};

// x[r] = e_t[tok] + pos[tok % N] for the packed rows r, tok = rowtok[r] or, with lists, looked
// up there and written to rowtok; refreshes e_ref[tok] from
// ref_src[tok] for refreshed tokens (last-refresh reference or cold view).  With
// bands.handle set, thread 0 of CTA 0 also selects the band of the row count.
cudaError_t launch_gather(const int* cu_rows_total, int* rowtok, const RowLists& lists, const float* e_t,
                          const float* pos, float* x, const float* ref_src, float* e_ref, int n_tok,
                          int dim, int ref_last_refresh, const ColdMask& cold, int max_rows, int grid,
                          cudaStream_t s, const RowBands& bands = RowBands());

// y[r] = LN(x[r]) (bf16) for r < *rows; when dst_rowtok is set, row r is written to
// row dst_rowtok[r] of y instead (final-token cache scatter).
cudaError_t launch_layernorm(const int* rows, const float* x, const float* gamma, const float* beta,
                             bf16* y, const int* dst_rowtok, int dim, float eps, int max_rows,
                             int grid, cudaStream_t s);
// The same, reading row src_rowtok[r] of x when src_rowtok is set, and when `add` is set
// first adding row src_rowtok[r] (or r) of `add` to x in place: x += add; y = LN(x).
cudaError_t launch_layernorm_ex(const int* rows, float* x, const float* add, const int* src_rowtok,
                                const float* gamma, const float* beta, bf16* y, const int* dst_rowtok, int dim,
                                float eps, int max_rows, int grid, cudaStream_t s);

// x[r] += bias + sum_s partial_s[r] (splits in order), written back to x, then y = LN(x[r])
// (row dst_rowtok[r] of y when set), for r < *rows.  With src_rowtok, row r is row
// src_rowtok[r] of x and of the partials, and x is left as it is; with add (not both), row r
// of add is added to x too.  dim a multiple of 4, at most 4096.
cudaError_t launch_layernorm_sum(const int* rows, float* x, const PendingSum& ps, const float* add,
                                 const int* src_rowtok, const float* gamma, const float* beta, bf16* y,
                                 const int* dst_rowtok, int dim, float eps, int max_rows, int grid, cudaStream_t s);

// One-time function attributes of the attention kernel (dynamic shared memory opt-in).
cudaError_t attention_setup();

// O[r] = softmax(Q[r] K_v^T / sqrt(dh)) V_v per head, for the packed query rows r of
// each view v (cu_rows), over the N cached keys/values of that view.
// Keys per CTA of the attention kernel for N tokens per view (the key-split width).
int attention_keys_per_split(int n_tok);
// tm_k / tm_v: this layer's key / value cache, bf16 [SV*N][D], box [kps rows][dh], no
// swizzle.  rowtok lists the updated tokens (packed row -> v*N + i): their keys are
// re-read after the wait on the QKV kernel, every other key is loaded before it.
// query_blocks: clusters per (view, head) along the queries (each loops over blocks of
// 32 queries with its key tile resident); any value is correct, it sets parallelism.
cudaError_t launch_attention(const CUtensorMap& tm_k, const CUtensorMap& tm_v, const bf16* q,
                             const bf16* cache_k, const bf16* cache_v, const int* cu_rows,
                             const int* rowtok, bf16* o, int sv, int n_tok, int dim, int heads,
                             int query_blocks, cudaStream_t s);

// ----------------------------------------------------------- attention (tcgen05)
struct AttnTcArgs {
  const int* cu_rows = nullptr;  // [SV+1] packed-row offsets of the views' updated rows
  const bf16* q = nullptr;       // packed queries [rows][D] and this layer's caches [SV*N][D],
  const bf16* k = nullptr;       // for the kernel that uses no TMA maps (attention_rows)
  const bf16* v = nullptr;
  bf16* o = nullptr;             // [rows][D] attention output, packed rows
  int* err = nullptr;            // device error word
  int n_tok = 0, dim = 0, dh = 0, heads = 0, sv = 0;
  unsigned long long* stamp = nullptr;  // timeline stamps of this launch (or null)
};

// One-time function attributes of the tensor-core attention kernel.
cudaError_t attention_tc_setup();

// Keys per block for a head width padded to 16: the widest whose S (a column per key), P (half
// a column) and O (dhp columns) fit in 256 tensor-memory columns.
constexpr int attention_key_block(int dhp) { return dhp <= 64 ? 128 : dhp <= 80 ? 96 : 64; }
// Columns of the second slice of a row, past the first 64 (0: none): one swizzle span wide.
constexpr int attention_slice2(int dhp) { return dhp <= 64 ? 0 : dhp <= 80 ? 16 : dhp <= 96 ? 32 : 64; }

// TMA maps of a [rows][H][dh] array for the attention: boxes of 1 head x 128 rows (queries) or
// attention_key_block rows (caches), `lo` of 64 columns with 128-byte swizzle, `hi` (when
// attention_slice2 > 0) of that many columns with a swizzle span of their size.
struct AttnMaps {
  CUtensorMap lo, hi;
};

// O[r] = softmax(Q[r] K_v^T / sqrt(dh)) V_v per head on the tensor cores, for the packed
// query rows r of each view v, over the N cached keys/values of that view (q, k, v: the packed
// queries, this layer's caches [SV*N]).  Two CTAs per SM walk the (view, head, query tile)
// items.  At most 4096 views.
cudaError_t launch_attention_tc(const AttnMaps& q, const AttnMaps& k, const AttnMaps& v, const AttnTcArgs& a,
                                int num_sms, cudaStream_t s);

// The same for a few queries per view, without TMA maps: CTAs walk (view, head, 16-query tile)
// items, `ctas` (1, or 2 for heads of up to 64) per SM; with `exact` the probabilities are not
// rounded to bf16.
cudaError_t attention_rows_setup();
cudaError_t launch_attention_rows(const AttnTcArgs& a, int num_sms, int ctas, bool exact, cudaStream_t s);

}  // namespace ivit
