// Engine behind the C ABI of include/ivit.h: weight upload, per-view caches,
// workspaces, TMA descriptors and the per-frame launch chain of temporal token reuse
// (Sec. III-B): embed -> score (Eq. 3) -> select/compact -> gather -> per layer
// {LN1, QKV + K/V cache scatter (Eq. 4-5), attention of updated queries over all
// tokens, out-proj + residual, LN2, MLP up + GELU, MLP down + residual} -> final LN
// scattered into the final-token cache -> output copy.
#include <cudaTypedefs.h>

#include <cmath>
#include <cstdlib>
#include <cstdio>
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/ivit.h"
#include "internal.h"
#include "ptx.cuh"

using ivit::bf16;

namespace {

struct LayerW {
  bf16 *wqkv, *wo, *w1, *w2;
  float *bqkv, *bo, *b1, *b2, *ln1g, *ln1b, *ln2g, *ln2b;
  CUtensorMap tm_qkv, tm_o, tm_1, tm_2;
  CUtensorMap tm_ck, tm_cv;  // this layer's key / value cache, SIMT attention key-split tiles (if selected)
  ivit::AttnMaps tm_ak, tm_av;  // the same caches for the tcgen05 attention
};

// Kernel families of the timeline.
enum Family : int { kFamGemm = 0, kFamAttn = 1, kFamLN = 2, kFamOther = 3, kFamilies = 4 };

struct TimelineSlot {
  int family = kFamOther;
  int n_out = 0, k = 0, kind = 0;  // GEMM shape and epilogue
  int m_static = -1;               // GEMM rows when fixed, -1 when read from the device
};

// Launch shape of one GEMM.  Over CTA pairs (nt = 0): tiles of bn rows, walked by n_pairs
// pairs.  Else the few-row kernel: CTAs of 8 nt features, passes of bn = 32 rows.  K is split
// `splits` ways, more than one only when deferred.
struct GemmPlan {
  int nt = 0, bn = 64, splits = 1, n_pairs = 1;
  bool defer = false;  // residual GEMMs: leave the split partials to the next layer norm
};

// One activation buffer: its TMA maps with boxes of 64 columns x 32, 64 and 128 rows.
struct ActMaps {
  const bf16* base = nullptr;
  CUtensorMap b32, b64, b128;
  const CUtensorMap& of(const GemmPlan& pl) const { return pl.bn <= 64 ? b32 : pl.bn == 128 ? b64 : b128; }
};

enum GemmSlot { kGemmEmbed = 0, kGemmQKV, kGemmO, kGemmUp, kGemmDown, kGemmSlots };

thread_local std::string g_create_error;

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// bf16 2-D tensor [rows][inner] with the given row stride; box = box_inner x box_rows,
// 128-byte swizzle (box_inner * 2 == 128) or dense rows, out-of-bounds elements read as 0.
bool make_map(CUtensorMap* m, const void* base, uint64_t inner, uint64_t rows, uint64_t stride_bytes,
              uint32_t box_inner, uint32_t box_rows, bool swizzle = true) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {inner, rows};
  cuuint64_t strides[1] = {stride_bytes};
  cuuint32_t box[2] = {box_inner, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The attention's maps of a [rows][heads][dh] array, boxes of box_rows rows.
bool make_attn_maps(ivit::AttnMaps* m, const void* base, uint64_t dh, uint64_t heads, uint64_t rows,
                    uint32_t box_rows) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  auto make = [&](CUtensorMap* map, uint32_t cols) {
    cuuint64_t dims[3] = {dh, heads, rows};
    cuuint64_t strides[2] = {dh * 2, dh * heads * 2};
    cuuint32_t box[3] = {cols, 1, box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    const auto swizzle = cols == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                         : cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                      : CU_TENSOR_MAP_SWIZZLE_32B;
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  const int hi = ivit::attention_slice2(static_cast<int>((dh + 15) & ~15ull));
  if (!make(&m->lo, 64)) return false;
  m->hi = m->lo;
  return hi == 0 || make(&m->hi, static_cast<uint32_t>(hi));
}

// Bump allocator over one device allocation; every sub-buffer 256-byte aligned.
struct Arena {
  size_t size = 0;
  char* base = nullptr;
  size_t take(size_t bytes) {
    const size_t off = size;
    size += (bytes + 255) & ~static_cast<size_t>(255);
    return off;
  }
  template <class T>
  T* at(size_t off) const {
    return reinterpret_cast<T*>(base + off);
  }
};

inline float bf16_bits_to_float(uint16_t b) {
  uint32_t u = static_cast<uint32_t>(b) << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

}  // namespace

namespace ivit {
void set_create_error(const char* msg) { g_create_error = msg ? msg : ""; }
}  // namespace ivit

struct ivit_handle {
  ivit_config cfg{};
  int N = 0, D = 0, F = 0, H = 0, L = 0, SV = 0, Kp = 0, KPAD = 0, M_max = 0;
  int device = 0, num_sms = 0;
  int row_grid = 0;
  GemmPlan plan_full[kGemmSlots], plan_inc[kGemmSlots], plan_keys;
  // Row-count bands of the incremental graph (band 0 = plan_inc): launch plans made for at
  // most band_ub[b] updated rows; a switch node picks the band of each call's device-resident
  // row count.
  int n_bands = 1;
  int row_groups = 1;  // of the few-row GEMM
  int band_ub[4] = {0, 0, 0, 0};
  GemmPlan plan_band[4][kGemmSlots];
  bool capture_bands = false;  // set while the incremental graph is captured with bands
  ivit::RowBands bands;        // the switch node's handle and the bands' row bounds
  cudaStream_t cap_stream2 = nullptr;  // captures the band bodies

  void* wmem = nullptr;  // weights (device)
  void* smem = nullptr;  // state + workspaces (device)
  bf16* w_pe = nullptr;
  float *b_pe = nullptr, *pos = nullptr, *lnfg = nullptr, *lnfb = nullptr;
  std::vector<LayerW> layers;
  CUtensorMap tm_pe;
  ActMaps tm_patches, tm_xn, tm_o, tm_h;
  ivit::AttnMaps tm_qa;  // packed queries (tcgen05 attention)
  bool attn_tc = true;   // tensor-core attention (IVIT_ATTN=simt selects the SIMT kernel)
  int attn_forced = -1;  // which of the two (IVIT_ATTN=tc 0, rows 1), -1: attention_few decides

  bf16* patches = nullptr;
  // Where the reference is the previous frame's patch embeddings, e_t and e_ref are one buffer:
  // the embedding GEMM's epilogue takes the scores against the content that it overwrites.
  bool one_ref = false;
  float4* score_parts = nullptr;  // its sums [feature tiles of 128][M_max]
  float *e_t = nullptr, *e_ref = nullptr, *sims = nullptr, *x = nullptr;
  float* key_t = nullptr;          // first-layer keys of every token (score_source KEY0)
  float* acache = nullptr;         // [L][M_max][D] attention-block outputs (mlp_tokens ALL)
  float* gemm_partials = nullptr;  // split-K partial tiles of the deferred GEMMs (global scratch)
  int* rowtok_all = nullptr;       // identity row -> token map, all SV*N rows
  int* m_all = nullptr;            // device copy of SV*N
  CUtensorMap tm_wk0;              // layer 0's key projection (rows D..2D-1 of W_qkv)
  long long chunk = 0;             // ivit_encode_incremental calls (odd/even schedule)
  int *idx = nullptr, *counts = nullptr, *cu_rows = nullptr, *rowtok = nullptr, *done_ctr = nullptr;
  int* err = nullptr;
  bf16 *xn = nullptr, *q = nullptr, *o = nullptr, *hbuf = nullptr, *cacheK = nullptr,
       *cacheV = nullptr, *tok_out = nullptr;

  std::vector<uint8_t> cold;
  int64_t launches = 0;

  // Persistent encoder (all blocks in one cooperative launch), on request.
  bool persistent = false;
  size_t pt_smem = 0;
  int pt_grid = 0;
  void* pt_mem = nullptr;  // device: tensor maps, layer parameters, partials, barrier words
  ivit::PersistentArgs pt_args{};

  // Weight-streaming kernel (every block of an incremental call in one cooperative
  // launch, weights streamed through a shared-memory ring) for small updated-row counts.
  bool stream_ok = false;
  size_t sk_smem = 0;
  int sk_grid = 0;
  void* sk_mem = nullptr;  // device: tensor maps, layer parameters, partials, sync words
  size_t sk_sync_bytes = 0;
  ivit::StreamArgs sk_args{};

  // CUDA graphs of the full and the steady-state incremental chain.  The kernels that see the
  // caller's pointers (patchify before it, the output copy after it) are launched outside the
  // graph, so its kernel parameters never change.
  bool use_graphs = true;
  uint8_t* frames_buf = nullptr;  // frames that patchify cannot read where they are
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t graph_full = nullptr, graph_inc = nullptr;
  int64_t graph_full_launches = 0, graph_inc_launches = 0;

  // Timeline mode (ivit_timeline): every launch of a call writes per-CTA start/end
  // stamps into its slot of `stamps`; `slots_*` record each slot's kernel family and,
  // for GEMMs, the shape that gives its algorithmic bytes.
  bool timeline = false;
  unsigned long long* stamps = nullptr;
  int stamp_cap = 0, stamp_used = 0;
  std::vector<TimelineSlot> slots_cur, slots_full, slots_inc, slots_last;

  std::string error;

  int fail(int code, const std::string& msg) {
    error = msg;
    return code;
  }
  int cuda_fail(const char* what, cudaError_t e) {
    error = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? IVIT_ERR_OOM : IVIT_ERR_CUDA;
  }
};

#define IVIT_CK(h, call)                                 \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return (h)->cuda_fail(#call, e_); \
  } while (0)

namespace {

const char* validate(const ivit_config* c) {
  if (!c) return "null config";
  if (c->patch <= 0 || c->img_h <= 0 || c->img_w <= 0) return "patch and image size must be positive";
  if (c->img_h % c->patch || c->img_w % c->patch) return "patch must divide img_h and img_w";
  const long long n = static_cast<long long>(c->img_h / c->patch) * (c->img_w / c->patch);
  if (n > 1024) return "at most 1024 tokens per view";
  if (c->dim <= 0 || c->dim % 64 || c->dim > 2048) return "dim must be a multiple of 64 in [64, 2048]";
  if (c->heads <= 0 || c->dim % c->heads) return "heads must divide dim";
  const int dh = c->dim / c->heads;
  if (dh % 8 || dh > 128) return "head_dim must be a multiple of 8 and at most 128";
  if (c->depth <= 0) return "depth must be positive";
  if (c->mlp_dim <= 0 || c->mlp_dim % 8) return "mlp_dim must be a positive multiple of 8";
  if (c->n_streams <= 0 || c->n_views <= 0) return "n_streams and n_views must be positive";
  if (static_cast<long long>(c->n_streams) * c->n_views > 4096) return "at most 4096 views";
  if (!(c->ln_eps > 0.f)) return "ln_eps must be positive";
  if (c->gelu != IVIT_GELU_TANH && c->gelu != IVIT_GELU_ERF) return "bad gelu";
  if (c->select_mode != IVIT_SEL_THRESHOLD && c->select_mode != IVIT_SEL_TOPK) return "bad select_mode";
  if (c->ref_mode != IVIT_REF_PREV_FRAME && c->ref_mode != IVIT_REF_LAST_REFRESH) return "bad ref_mode";
  if (c->select_mode == IVIT_SEL_TOPK && c->topk < 0) return "topk must be >= 0";
  if (!std::isfinite(c->threshold)) return "threshold must be finite";
  if (c->score_source != IVIT_SCORE_EMBED && c->score_source != IVIT_SCORE_KEY0) return "bad score_source";
  if (c->schedule != IVIT_SCHED_INCREMENTAL && c->schedule != IVIT_SCHED_ODD_EVEN) return "bad schedule";
  if (c->mlp_tokens != IVIT_MLP_UPDATED && c->mlp_tokens != IVIT_MLP_ALL) return "bad mlp_tokens";
  return nullptr;
}

size_t weights_count(const ivit_config* c) {
  const size_t D = c->dim, F = c->mlp_dim, N = static_cast<size_t>(c->img_h / c->patch) * (c->img_w / c->patch);
  const size_t Kp = static_cast<size_t>(c->patch) * c->patch * 3;
  const size_t per_layer = 2 * D + 3 * D * D + 3 * D + D * D + D + 2 * D + F * D + F + D * F + D;
  return D * Kp + D + N * D + per_layer * c->depth + 2 * D;
}

// Scratch slots (fp32 [bn][128]) a deferred plan needs for up to m_bound rows.
size_t defer_slots(const GemmPlan& pl, int n_out, int m_bound) {
  return static_cast<size_t>((n_out + 127) / 128) * ((m_bound + pl.bn - 1) / pl.bn) * pl.splits;
}

// Launch shape of a GEMM expected to see m_expected rows, as wide as m_bound rows can use (any
// count runs): the cheapest candidate of a cost model in microseconds per launch, fitted to back-to-back
// launches on GB300 of the SigLIP-So400m and ViT-Tiny shapes at 16 to 32768 rows.
//   CTA pairs: a fixed part (prologue, first loads, last tile's epilogue) plus a k-block
//     (64 wide) rate per round of units over the 76 pairs; 64-, 128- and 256-row tiles
//     measured 4.3 / 4.8 / 6.2 us + 0.165 / 0.24 / 0.33 us per k-block, and 0.7 us for the
//     prologue that its shared memory keeps from running under the previous kernel.
//   Few rows (`few`: the epilogues that kernel has): 1.1 us, then per pass of 32 rows and
//     round of CTAs over the SMs 0.9 us and 0.15 to 0.36 us per chunk (32 wide) of a warp for 8
//     to 32 features per CTA.  QKV of 26 rows 4.0 us against 7.2 in pairs, of 64 rows 6.6
//     against 7.2, of 128 rows 11.1 against 7.2.
//   Deferred (residual GEMMs, `defer`): the next layer norm sums the partial tiles: no
//     epilogue, but every split's fp32 tile is written and read once (about 10 TB/s, in L2, hence
//     at most 64 MB of them for m_bound rows; the scratch itself has room for every row).
GemmPlan plan_gemm(int num_sms, int n_out, int k, int m_expected, int m_bound, bool few, bool defer) {
  GemmPlan best;
  double best_cost = 1e30;
  defer = defer && !std::getenv("IVIT_NO_DEFER");
  auto consider = [&](const GemmPlan& pl, double cost) {
    if (pl.defer) {
      if (defer_slots(pl, n_out, m_bound) * pl.bn * 128 * 4 > (64ull << 20)) return;
      cost += pl.splits * (8.0 * n_out) * m_expected / 1.0e7;
    }
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = pl;
    }
  };
  const int n_ft = (n_out + 127) / 128, n_kb = (k + 63) / 64, max_pairs = num_sms / 2;
  for (int bn : {64, 128, 256}) {
    const double fixed = bn == 64 ? 5.0 : bn == 128 ? 5.5 : 6.9, per_kb = bn == 64 ? 0.165 : bn == 128 ? 0.24 : 0.33;
    const int tiles = std::max(1, (n_ft + 1) / 2 * ((m_expected + bn - 1) / bn));
    for (int c = 1; c <= std::min(defer ? 16 : 1, n_kb); ++c) {
      GemmPlan pl;
      pl.bn = bn;
      pl.splits = c;
      pl.defer = c > 1;
      // (a call may bring more rows than expected: the launch is as wide as m_bound can use)
      pl.n_pairs = std::min(max_pairs, (n_ft + 1) / 2 * ((m_bound + bn - 1) / bn) * c);
      const int rounds = (tiles * c + max_pairs - 1) / max_pairs;
      consider(pl, fixed + rounds * per_kb * ((n_kb + c - 1) / c));
    }
  }
  if (!few) return best;
  const int n_ck = (k + 31) / 32, passes = std::max(1, (m_expected + 31) / 32);
  for (int nt = 1; nt <= 4; ++nt) {
    for (int c = 1; c <= std::min(defer ? 16 : 1, n_ck); ++c) {
      GemmPlan pl;
      pl.nt = nt;
      pl.bn = 32;
      pl.splits = c;
      pl.defer = c > 1;
      if (ivit::gemm_rows_smem(nt, k, c) > ivit::GEMM_ROWS_SMEM_MAX) continue;
      const int ctas = (n_out + 8 * nt - 1) / (8 * nt) * c, rounds = (ctas + num_sms - 1) / num_sms;
      const int per_warp = ((n_ck + c - 1) / c + 7) / 8;
      consider(pl, 1.1 + passes * rounds * (0.9 + per_warp * (0.08 + 0.07 * nt)));
    }
  }
  return best;
}

int attention_few(const ivit_handle* h, int m_expected, bool exact = false);

// Updated rows to expect of a call in row band b: a tenth of the tokens in the first, the
// middle of the others.
int band_rows(const ivit_handle* h, int b) {
  return b == 0 ? std::max(1, h->M_max / 10) : (h->band_ub[b - 1] + h->band_ub[b]) / 2;
}

// Prepares the persistent encoder (IVIT_PATH=persistent: every call runs it) when its shared
// memory fits (attention keeps a whole view's keys and values of one head resident, so
// N * head_dim is bounded).  It is not the default anywhere: its SIMT attention phase and
// 64-row GEMM tiles lose to the kernel chain also on the full encodes of small encoders
// (six 196-token views of ViT-Tiny 1.40 ms against 0.38 ms for the chain).
int setup_persistent(ivit_handle* h) {
  const char* path = std::getenv("IVIT_PATH");
  if (!path || std::strcmp(path, "persistent") != 0) return IVIT_OK;
  if (h->cfg.mlp_tokens == IVIT_MLP_ALL) return IVIT_OK;  // the kernel chain runs that reading
  const int dh = h->D / h->H;
  const size_t smem = ivit::persistent_smem_bytes(h->N, dh);
  if (smem > 227 * 1024 || h->D > 2048 || h->N > 256) return IVIT_OK;
  IVIT_CK(h, ivit::persistent_setup(smem));
  const int grid = std::min(h->num_sms, ivit::persistent_max_ctas(smem));
  if (grid < 1) return IVIT_OK;
  const int L = h->L;
  // partial slots: at most one item per CTA with K split, else one per tile
  const int n_tt = (h->M_max + 63) / 64;
  const int max_tiles = std::max({(3 * h->D + 127) / 128, (h->F + 127) / 128}) * n_tt;
  const int max_items = std::max(grid, max_tiles);
  Arena pa;
  const size_t o_w = pa.take(sizeof(CUtensorMap) * 4 * L), o_x = pa.take(sizeof(CUtensorMap) * 3);
  const size_t o_kv = pa.take(sizeof(CUtensorMap) * 2 * L);
  const size_t o_lp = pa.take(sizeof(ivit::LayerParams) * L);
  const size_t o_part = pa.take(ivit::persistent_part_floats(max_items) * sizeof(float));
  const size_t o_bar = pa.take(4 * sizeof(unsigned));
  IVIT_CK(h, cudaMalloc(&h->pt_mem, pa.size));
  IVIT_CK(h, cudaMemset(h->pt_mem, 0, pa.size));
  pa.base = static_cast<char*>(h->pt_mem);
  std::vector<CUtensorMap> wm(4 * L);
  std::vector<ivit::LayerParams> lp(L);
  for (int l = 0; l < L; ++l) {
    const LayerW& w = h->layers[l];
    wm[4 * l + 0] = w.tm_qkv;
    wm[4 * l + 1] = w.tm_o;
    wm[4 * l + 2] = w.tm_1;
    wm[4 * l + 3] = w.tm_2;
    lp[l] = ivit::LayerParams{w.bqkv, w.bo, w.b1, w.b2, w.ln1g, w.ln1b, w.ln2g, w.ln2b};
  }
  const CUtensorMap xm[3] = {h->tm_xn.b32, h->tm_o.b32, h->tm_h.b32};
  std::vector<CUtensorMap> kvm(2 * L);
  for (int l = 0; l < L; ++l) {
    const size_t off = static_cast<size_t>(l) * h->M_max * h->D;
    if (!make_map(&kvm[2 * l], h->cacheK + off, h->D, h->M_max, h->D * 2, dh, h->N, false) ||
        !make_map(&kvm[2 * l + 1], h->cacheV + off, h->D, h->M_max, h->D * 2, dh, h->N, false))
      return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for a cache tile");
  }
  IVIT_CK(h, cudaMemcpy(pa.base + o_kv, kvm.data(), sizeof(CUtensorMap) * 2 * L, cudaMemcpyHostToDevice));
  IVIT_CK(h, cudaMemcpy(pa.base + o_w, wm.data(), sizeof(CUtensorMap) * 4 * L, cudaMemcpyHostToDevice));
  IVIT_CK(h, cudaMemcpy(pa.base + o_x, xm, sizeof(xm), cudaMemcpyHostToDevice));
  IVIT_CK(h, cudaMemcpy(pa.base + o_lp, lp.data(), sizeof(ivit::LayerParams) * L, cudaMemcpyHostToDevice));
  ivit::PersistentArgs& a = h->pt_args;
  a.N = h->N;
  a.D = h->D;
  a.F = h->F;
  a.H = h->H;
  a.dh = dh;
  a.L = L;
  a.SV = h->SV;
  a.M_max = h->M_max;
  a.eps = h->cfg.ln_eps;
  a.gelu = h->cfg.gelu;
  a.cu_rows = h->cu_rows;
  a.rowtok = h->rowtok;
  a.wmaps = pa.at<CUtensorMap>(o_w);
  a.xmaps = pa.at<CUtensorMap>(o_x);
  a.kvmaps = pa.at<CUtensorMap>(o_kv);
  a.layers = pa.at<ivit::LayerParams>(o_lp);
  a.lnfg = h->lnfg;
  a.lnfb = h->lnfb;
  a.x = h->x;
  a.xn = h->xn;
  a.q = h->q;
  a.o = h->o;
  a.h = h->hbuf;
  a.cacheK = h->cacheK;
  a.cacheV = h->cacheV;
  a.tok_out = h->tok_out;
  a.part = pa.at<float>(o_part);
  a.gbar = pa.at<unsigned>(o_bar);
  a.err = h->err;
  a.trace = nullptr;
  if (std::getenv("IVIT_TRACE")) {
    IVIT_CK(h, cudaMalloc(&a.trace, 4096 * sizeof(unsigned long long)));
    IVIT_CK(h, cudaMemset(a.trace, 0, 4096 * sizeof(unsigned long long)));
  }
  h->pt_smem = smem;
  h->pt_grid = grid;
  h->persistent = true;
  return IVIT_OK;
}

// Prepares the weight-streaming kernel (IVIT_PATH=stream: every incremental call without
// a cold view runs it).  It is not the default: on the So400m camera stream it measured
// 1.5 ms per frame against the kernel chain's 1.0 ms (seven grid barriers per layer and
// the dependent latencies inside each stage cost more than the chain's launch handoffs).
int setup_stream(ivit_handle* h) {
  const ivit_config& c = h->cfg;
  const char* path = std::getenv("IVIT_PATH");
  if (!path || std::strcmp(path, "stream") != 0) return IVIT_OK;
  if (c.mlp_tokens == IVIT_MLP_ALL) return IVIT_OK;  // the kernel chain runs that reading
  const int N = h->N, D = h->D, F = h->F, H = h->H, L = h->L, SV = h->SV, dh = D / H;
  if (D > ivit::stream_max_dim() || N > 256) return IVIT_OK;
  int optin = 0;
  IVIT_CK(h, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device));
  const int grid = h->num_sms;
  // K splits: enough tasks (tile x split) to give about one to every CTA
  const int n_out[4] = {3 * D, D, F, D}, kdim[4] = {D, D, D, F};
  int splits[4], max_kb = 0;
  size_t part_floats = 0;
  for (int g = 0; g < 4; ++g) {
    const int tiles = (n_out[g] + 127) / 128, nkb = (kdim[g] + 63) / 64;
    splits[g] = std::max(1, std::min(nkb, grid / tiles));
    max_kb = std::max(max_kb, ivit::stream_task_kblocks(kdim[g], splits[g]));
    part_floats = std::max(part_floats, static_cast<size_t>(splits[g]) * h->M_max * n_out[g]);
  }
  const size_t region = ivit::stream_region_bytes(max_kb, N, dh);
  const int rs = ivit::stream_ring_stages_for(static_cast<size_t>(optin), region);
  if (rs < std::max(4, max_kb)) return IVIT_OK;
  const size_t smem = ivit::stream_smem_bytes(rs, region);
  IVIT_CK(h, ivit::stream_setup(smem));
  if (ivit::stream_max_ctas(smem) < grid) return IVIT_OK;
  const int rpp = ivit::stream_rows_per_pass();
  const int passes_max = (h->M_max + rpp - 1) / rpp;
  const int qkv_tiles = (3 * D + 127) / 128, up_tiles = (F + 127) / 128;
  const size_t sync_words = 4 + static_cast<size_t>(L) * (qkv_tiles + up_tiles) * passes_max;
  Arena ka;
  const size_t o_w = ka.take(sizeof(CUtensorMap) * 4 * L), o_b = ka.take(sizeof(CUtensorMap) * 3);
  const size_t o_kv = ka.take(sizeof(CUtensorMap) * 2 * L), o_lp = ka.take(sizeof(ivit::LayerParams) * L);
  const size_t o_part = ka.take(part_floats * sizeof(float)), o_sync = ka.take(sync_words * sizeof(unsigned));
  IVIT_CK(h, cudaMalloc(&h->sk_mem, ka.size));
  IVIT_CK(h, cudaMemset(h->sk_mem, 0, ka.size));
  ka.base = static_cast<char*>(h->sk_mem);
  std::vector<CUtensorMap> wm(4 * L), kvm(2 * L);
  std::vector<ivit::LayerParams> lp(L);
  for (int l = 0; l < L; ++l) {
    const LayerW& w = h->layers[l];
    const size_t off = static_cast<size_t>(l) * h->M_max * D;
    wm[4 * l + 0] = w.tm_qkv;
    wm[4 * l + 1] = w.tm_o;
    wm[4 * l + 2] = w.tm_1;
    wm[4 * l + 3] = w.tm_2;
    if (!make_map(&kvm[2 * l], h->cacheK + off, D, h->M_max, D * 2, dh, N, false) ||
        !make_map(&kvm[2 * l + 1], h->cacheV + off, D, h->M_max, D * 2, dh, N, false))
      return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for the weight-streaming kernel");
    lp[l] = ivit::LayerParams{w.bqkv, w.bo, w.b1, w.b2, w.ln1g, w.ln1b, w.ln2g, w.ln2b};
  }
  const CUtensorMap bm[3] = {h->tm_xn.b32, h->tm_o.b32, h->tm_h.b32};
  IVIT_CK(h, cudaMemcpy(ka.base + o_w, wm.data(), sizeof(CUtensorMap) * 4 * L, cudaMemcpyHostToDevice));
  IVIT_CK(h, cudaMemcpy(ka.base + o_b, bm, sizeof(bm), cudaMemcpyHostToDevice));
  IVIT_CK(h, cudaMemcpy(ka.base + o_kv, kvm.data(), sizeof(CUtensorMap) * 2 * L, cudaMemcpyHostToDevice));
  IVIT_CK(h, cudaMemcpy(ka.base + o_lp, lp.data(), sizeof(ivit::LayerParams) * L, cudaMemcpyHostToDevice));
  ivit::StreamArgs& a = h->sk_args;
  a.N = N;
  a.D = D;
  a.F = F;
  a.H = H;
  a.dh = dh;
  a.L = L;
  a.SV = SV;
  a.M_max = h->M_max;
  a.eps = c.ln_eps;
  a.gelu = c.gelu;
  a.ring_stages = rs;
  a.region_bytes = static_cast<int>(region);
  a.att_groups = std::max(1, std::min(16, grid / std::max(1, SV * H)));
  for (int g = 0; g < 4; ++g) a.splits[g] = splits[g];
  a.qkv_tiles = qkv_tiles;
  a.n_barriers = 7 * L;
  a.cu_rows = h->cu_rows;
  a.rowtok = h->rowtok;
  a.wmaps = ka.at<CUtensorMap>(o_w);
  a.bmaps = ka.at<CUtensorMap>(o_b);
  a.kvmaps = ka.at<CUtensorMap>(o_kv);
  a.layers = ka.at<ivit::LayerParams>(o_lp);
  a.lnfg = h->lnfg;
  a.lnfb = h->lnfb;
  a.x = h->x;
  a.xn = h->xn;
  a.q = h->q;
  a.o = h->o;
  a.h = h->hbuf;
  a.cacheK = h->cacheK;
  a.cacheV = h->cacheV;
  a.tok_out = h->tok_out;
  a.part = ka.at<float>(o_part);
  a.sync = ka.at<unsigned>(o_sync);
  a.err = h->err;
  a.trace = nullptr;
  if (std::getenv("IVIT_TRACE")) {
    const size_t n = static_cast<size_t>(a.n_barriers) * (grid + 1) + 64 * static_cast<size_t>(grid);
    IVIT_CK(h, cudaMalloc(&a.trace, n * sizeof(unsigned long long)));
    IVIT_CK(h, cudaMemset(a.trace, 0, n * sizeof(unsigned long long)));
  }
  h->sk_sync_bytes = sync_words * sizeof(unsigned);
  h->sk_smem = smem;
  h->sk_grid = grid;
  h->stream_ok = true;
  if (std::getenv("IVIT_DEBUG"))
    std::fprintf(stderr, "ivit stream kernel: grid %d, smem %zu, ring %d stages, region %zu, groups %d, "
                 "splits %d %d %d %d\n", grid, smem, rs, region, a.att_groups, splits[0], splits[1], splits[2],
                 splits[3]);
  return IVIT_OK;
}

// Whether the row counts of threshold calls commonly cross bands, so that a switch over them pays
// its fixed cost (about 10 us: no programmatic overlap across the node).  Below, one plan serves
// every count, with a second row group in the few-row GEMM.
bool rows_cross_bands(const ivit_handle* h) { return h->M_max / 10 > 32; }

// The bands of the row count and the launch plans of every GEMM, from the configuration and the
// number of SMs alone.
void make_plans(ivit_handle* h) {
  const ivit_config& c = h->cfg;
  const int D = h->D, F = h->F, m_all = h->M_max, m_inc = std::max(1, m_all / 10);
  // Row bands: the first holds a tenth of the tokens (rounded up to 16, at least 64),
  // each next one twice the previous, the last all of them; at most four.
  int ub = std::max(64, (m_all / 10 + 15) / 16 * 16);
  h->n_bands = 0;
  while (h->n_bands < 4) {
    const bool last = ub >= m_all || h->n_bands == 3;
    h->band_ub[h->n_bands++] = last ? m_all : ub;
    if (last) break;
    ub *= 2;
  }
  if (std::getenv("IVIT_NO_BANDS")) h->n_bands = 1;
  // Full encodes know M = SV*N.  Incremental calls are planned for a tenth of the
  // tokens updated (any count still runs correctly, with more or fewer tile rounds).
  const int shapes[kGemmSlots][2] = {{D, h->KPAD}, {3 * D, D}, {D, D}, {F, D}, {D, F}};
  for (int g = 0; g < kGemmSlots; ++g) {
    // (under the MLP-on-all-tokens reading the out-projection goes to a cache, not to a layer norm)
    const bool defer = g == kGemmDown || (g == kGemmO && c.mlp_tokens == IVIT_MLP_UPDATED);
    auto plan = [&](int m_expected, int m_bound) {
      return plan_gemm(h->num_sms, shapes[g][0], shapes[g][1], m_expected, m_bound, g != kGemmEmbed, defer);
    };
    h->plan_full[g] = plan(m_all, m_all);
    h->plan_inc[g] = g == kGemmEmbed ? h->plan_full[g] : plan(m_inc, m_all);
    h->plan_band[0][g] = h->plan_inc[g];
    // (the band of all rows runs the full encode's plans)
    for (int b = 1; b < h->n_bands; ++b)
      h->plan_band[b][g] = g == kGemmEmbed || h->band_ub[b] >= m_all ? h->plan_full[g]
                                                                     : plan(h->band_ub[b], h->band_ub[b]);
  }
  // (a switch between equal plans would only cost its dispatch, about 10 us)
  auto same = [](const GemmPlan& a, const GemmPlan& b) {
    return a.nt == b.nt && a.bn == b.bn && a.splits == b.splits && a.n_pairs == b.n_pairs;
  };
  bool differ = false;
  for (int b = 1; b < h->n_bands; ++b)
    for (int g = 0; g < kGemmSlots; ++g) differ = differ || !same(h->plan_band[b][g], h->plan_band[0][g]);
  for (int b = 1; b < h->n_bands; ++b)
    differ = differ || attention_few(h, band_rows(h, b)) != attention_few(h, band_rows(h, 0));
  if (!differ) h->n_bands = 1;
  // a second row group (gemm.cu) where the band of the row count is not known at launch
  const bool one_plan = c.mlp_tokens == IVIT_MLP_ALL || c.select_mode != IVIT_SEL_TOPK;
  h->row_groups = one_plan && m_all > 64 && (c.mlp_tokens == IVIT_MLP_ALL || !rows_cross_bands(h)) ? 2 : 1;
  // every row's D x D projection without a residual (first-layer key scores)
  h->plan_keys = plan_gemm(h->num_sms, D, D, m_all, m_all, false, false);
  if (std::getenv("IVIT_DEBUG")) {
    static const char* names[kGemmSlots] = {"embed", "qkv", "out", "up", "down"};
    auto show = [&](const char* when, const char* name, const GemmPlan& pl) {
      std::fprintf(stderr, "ivit gemm %-6s %-5s %s bn=%d nt=%d splits=%d\n", when, name, pl.nt ? "rows" : "pair", pl.bn,
                   pl.nt, pl.splits);
    };
    for (int g = 0; g < kGemmSlots; ++g) {
      show("full", names[g], h->plan_full[g]);
      show("inc", names[g], h->plan_inc[g]);
      for (int b = 1; b < h->n_bands; ++b) show(b == 1 ? "band 1" : b == 2 ? "band 2" : "band 3", names[g], h->plan_band[b][g]);
    }
  }
}

// Floats of the split-K scratch: slots [rows of a tile][128 features] of every plan, for every
// row of every view.  A band's bound would not do: top-k selects NaN scores beside the k lowest,
// so a call whose plans were picked for k rows a view can bring more.
size_t scratch_floats(const ivit_handle* h) {
  size_t most = 64;
  auto need = [&](const GemmPlan& pl) {
    if (pl.defer) most = std::max(most, defer_slots(pl, h->D, h->M_max) * pl.bn * 128);
  };
  for (int g = 0; g < kGemmSlots; ++g) {
    need(h->plan_full[g]);
    need(h->plan_inc[g]);
    for (int b = 0; b < h->n_bands; ++b) need(h->plan_band[b][g]);
  }
  return most;
}

int setup(ivit_handle* h, const uint16_t* wb) {
  const ivit_config& c = h->cfg;
  h->N = (c.img_h / c.patch) * (c.img_w / c.patch);
  h->D = c.dim;
  h->F = c.mlp_dim;
  h->H = c.heads;
  h->L = c.depth;
  h->SV = c.n_streams * c.n_views;
  h->Kp = c.patch * c.patch * 3;
  h->KPAD = (h->Kp + 63) / 64 * 64;
  h->M_max = h->SV * h->N;
  h->cold.assign(h->SV, 1);
  const size_t D = h->D, F = h->F, N = h->N, L = h->L, M = h->M_max;

  IVIT_CK(h, cudaGetDevice(&h->device));
  IVIT_CK(h, cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device));
  IVIT_CK(h, ivit::gemm_rows_setup());
  IVIT_CK(h, ivit::gemm_pair_setup());
  IVIT_CK(h, ivit::attention_setup());
  IVIT_CK(h, ivit::attention_tc_setup());
  IVIT_CK(h, ivit::attention_rows_setup());
  if (const char* at = std::getenv("IVIT_ATTN")) {
    h->attn_tc = std::string(at) != "simt";
    h->attn_forced = std::string(at) == "tc" ? 0 : std::string(at) == "rows" ? 1 : -1;
  }
  if (std::getenv("IVIT_NO_PDL")) ivit::g_use_pdl = false;
  if (std::getenv("IVIT_NO_GRAPH")) h->use_graphs = false;
  IVIT_CK(h, cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
  IVIT_CK(h, cudaStreamCreateWithFlags(&h->cap_stream2, cudaStreamNonBlocking));
  h->row_grid = h->num_sms * 4;
  make_plans(h);

  // ---- weights: bf16 matrices (W_pe padded to KPAD columns), fp32 vectors
  Arena wa;
  const size_t o_pe = wa.take(D * h->KPAD * 2), o_bpe = wa.take(D * 4), o_pos = wa.take(N * D * 4);
  struct LOff { size_t qkv, o, w1, w2, bqkv, bo, b1, b2, g1, be1, g2, be2; };
  std::vector<LOff> lo(L);
  for (size_t l = 0; l < L; ++l) {
    lo[l].qkv = wa.take(3 * D * D * 2);
    lo[l].o = wa.take(D * D * 2);
    lo[l].w1 = wa.take(F * D * 2);
    lo[l].w2 = wa.take(D * F * 2);
    lo[l].bqkv = wa.take(3 * D * 4);
    lo[l].bo = wa.take(D * 4);
    lo[l].b1 = wa.take(F * 4);
    lo[l].b2 = wa.take(D * 4);
    lo[l].g1 = wa.take(D * 4);
    lo[l].be1 = wa.take(D * 4);
    lo[l].g2 = wa.take(D * 4);
    lo[l].be2 = wa.take(D * 4);
  }
  const size_t o_gf = wa.take(D * 4), o_bf = wa.take(D * 4);

  std::vector<char> host(wa.size, 0);
  auto put_bf16 = [&](size_t off, const uint16_t* src, size_t rows, size_t cols, size_t ld) {
    for (size_t r = 0; r < rows; ++r) std::memcpy(&host[off + r * ld * 2], src + r * cols, cols * 2);
  };
  auto put_f32 = [&](size_t off, const uint16_t* src, size_t n) {
    float* dst = reinterpret_cast<float*>(&host[off]);
    for (size_t i = 0; i < n; ++i) dst[i] = bf16_bits_to_float(src[i]);
  };
  const uint16_t* p = wb;
  put_bf16(o_pe, p, D, h->Kp, h->KPAD); p += D * h->Kp;
  put_f32(o_bpe, p, D); p += D;
  put_f32(o_pos, p, N * D); p += N * D;
  for (size_t l = 0; l < L; ++l) {
    put_f32(lo[l].g1, p, D); p += D;
    put_f32(lo[l].be1, p, D); p += D;
    put_bf16(lo[l].qkv, p, 3 * D, D, D); p += 3 * D * D;
    put_f32(lo[l].bqkv, p, 3 * D); p += 3 * D;
    put_bf16(lo[l].o, p, D, D, D); p += D * D;
    put_f32(lo[l].bo, p, D); p += D;
    put_f32(lo[l].g2, p, D); p += D;
    put_f32(lo[l].be2, p, D); p += D;
    put_bf16(lo[l].w1, p, F, D, D); p += F * D;
    put_f32(lo[l].b1, p, F); p += F;
    put_bf16(lo[l].w2, p, D, F, F); p += D * F;
    put_f32(lo[l].b2, p, D); p += D;
  }
  put_f32(o_gf, p, D); p += D;
  put_f32(o_bf, p, D); p += D;

  IVIT_CK(h, cudaMalloc(&h->wmem, wa.size));
  IVIT_CK(h, cudaMemcpy(h->wmem, host.data(), wa.size, cudaMemcpyHostToDevice));
  wa.base = static_cast<char*>(h->wmem);
  h->w_pe = wa.at<bf16>(o_pe);
  h->b_pe = wa.at<float>(o_bpe);
  h->pos = wa.at<float>(o_pos);
  h->lnfg = wa.at<float>(o_gf);
  h->lnfb = wa.at<float>(o_bf);
  h->layers.resize(L);
  for (size_t l = 0; l < L; ++l) {
    LayerW& w = h->layers[l];
    w.wqkv = wa.at<bf16>(lo[l].qkv);
    w.wo = wa.at<bf16>(lo[l].o);
    w.w1 = wa.at<bf16>(lo[l].w1);
    w.w2 = wa.at<bf16>(lo[l].w2);
    w.bqkv = wa.at<float>(lo[l].bqkv);
    w.bo = wa.at<float>(lo[l].bo);
    w.b1 = wa.at<float>(lo[l].b1);
    w.b2 = wa.at<float>(lo[l].b2);
    w.ln1g = wa.at<float>(lo[l].g1);
    w.ln1b = wa.at<float>(lo[l].be1);
    w.ln2g = wa.at<float>(lo[l].g2);
    w.ln2b = wa.at<float>(lo[l].be2);
    if (!make_map(&w.tm_qkv, w.wqkv, D, 3 * D, D * 2, 64, 128) ||
        !make_map(&w.tm_o, w.wo, D, D, D * 2, 64, 128) ||
        !make_map(&w.tm_1, w.w1, D, F, D * 2, 64, 128) ||
        !make_map(&w.tm_2, w.w2, F, D, F * 2, 64, 128))
      return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight matrix");
  }
  if (!make_map(&h->tm_pe, h->w_pe, h->KPAD, D, h->KPAD * 2, 64, 128))
    return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for W_pe");

  // ---- state and workspaces
  Arena sa;
  h->one_ref = c.score_source == IVIT_SCORE_EMBED && c.ref_mode == IVIT_REF_PREV_FRAME;
  const size_t o_patch = sa.take(M * h->KPAD * 2), o_et = sa.take(M * D * 4);
  const size_t o_er = h->one_ref ? o_et : sa.take(M * D * 4);
  const size_t o_sp = h->one_ref ? sa.take(M * ((D + 127) / 128) * sizeof(float4)) : 0;
  const size_t o_sims = sa.take(M * 4), o_idx = sa.take(M * 4), o_cnt = sa.take(h->SV * 4);
  const size_t o_cu = sa.take((h->SV + 1) * 4), o_rt = sa.take(M * 4), o_done = sa.take(4);
  const size_t o_x = sa.take(M * D * 4), o_xn = sa.take(M * D * 2), o_q = sa.take(M * D * 2);
  const size_t o_o = sa.take(M * D * 2), o_h = sa.take(M * F * 2);
  const size_t o_ck = sa.take(L * M * D * 2), o_cv = sa.take(L * M * D * 2), o_tok = sa.take(M * D * 2);
  const size_t o_err = sa.take(4);
  const size_t o_key = c.score_source == IVIT_SCORE_KEY0 ? sa.take(M * D * 4) : 0;
  const size_t o_acache = c.mlp_tokens == IVIT_MLP_ALL ? sa.take(L * M * D * 4) : 0;
  const size_t o_gpart = sa.take(scratch_floats(h) * 4);
  const size_t o_rta = sa.take(M * 4), o_mall = sa.take(4);
  const size_t o_fb = sa.take(static_cast<size_t>(h->SV) * c.img_h * c.img_w * 3);
  IVIT_CK(h, cudaMalloc(&h->smem, sa.size));
  IVIT_CK(h, cudaMemset(h->smem, 0, sa.size));
  sa.base = static_cast<char*>(h->smem);
  h->patches = sa.at<bf16>(o_patch);
  h->e_t = sa.at<float>(o_et);
  h->e_ref = sa.at<float>(o_er);
  if (h->one_ref) h->score_parts = sa.at<float4>(o_sp);
  h->sims = sa.at<float>(o_sims);
  h->idx = sa.at<int>(o_idx);
  h->counts = sa.at<int>(o_cnt);
  h->cu_rows = sa.at<int>(o_cu);
  h->rowtok = sa.at<int>(o_rt);
  h->done_ctr = sa.at<int>(o_done);
  h->x = sa.at<float>(o_x);
  h->xn = sa.at<bf16>(o_xn);
  h->q = sa.at<bf16>(o_q);
  h->o = sa.at<bf16>(o_o);
  h->hbuf = sa.at<bf16>(o_h);
  h->cacheK = sa.at<bf16>(o_ck);
  h->cacheV = sa.at<bf16>(o_cv);
  h->tok_out = sa.at<bf16>(o_tok);
  h->err = sa.at<int>(o_err);
  if (c.score_source == IVIT_SCORE_KEY0) h->key_t = sa.at<float>(o_key);
  if (c.mlp_tokens == IVIT_MLP_ALL) h->acache = sa.at<float>(o_acache);
  h->gemm_partials = sa.at<float>(o_gpart);
  h->rowtok_all = sa.at<int>(o_rta);
  h->m_all = sa.at<int>(o_mall);
  h->frames_buf = sa.at<uint8_t>(o_fb);
  {
    std::vector<int> ident(M);
    for (size_t i = 0; i < M; ++i) ident[i] = static_cast<int>(i);
    const int m_host = static_cast<int>(M);
    IVIT_CK(h, cudaMemcpy(h->rowtok_all, ident.data(), M * sizeof(int), cudaMemcpyHostToDevice));
    IVIT_CK(h, cudaMemcpy(h->m_all, &m_host, sizeof(int), cudaMemcpyHostToDevice));
  }
  if (!make_map(&h->tm_wk0, h->layers[0].wqkv + D * D, D, D, D * 2, 64, 128))
    return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for the first-layer key projection");
  const int kps = ivit::attention_keys_per_split(h->N);
  const int dh = h->D / h->H, kb = ivit::attention_key_block((dh + 15) & ~15);
  for (size_t l = 0; l < L; ++l) {
    const size_t off = l * M * D;
    if ((!h->attn_tc && (!make_map(&h->layers[l].tm_ck, h->cacheK + off, D, M, D * 2, D / h->H, kps, false) ||
                         !make_map(&h->layers[l].tm_cv, h->cacheV + off, D, M, D * 2, D / h->H, kps, false))) ||
        !make_attn_maps(&h->layers[l].tm_ak, h->cacheK + off, dh, h->H, M, kb) ||
        !make_attn_maps(&h->layers[l].tm_av, h->cacheV + off, dh, h->H, M, kb))
      return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for a cache tile");
  }
  auto act_maps = [&](ActMaps& m, const bf16* base, size_t inner) {
    m.base = base;
    return make_map(&m.b32, base, inner, M, inner * 2, 64, 32) && make_map(&m.b64, base, inner, M, inner * 2, 64, 64) &&
           make_map(&m.b128, base, inner, M, inner * 2, 64, 128);
  };
  if (!act_maps(h->tm_patches, h->patches, h->KPAD) || !act_maps(h->tm_xn, h->xn, D) || !act_maps(h->tm_o, h->o, D) ||
      !act_maps(h->tm_h, h->hbuf, F) || !make_attn_maps(&h->tm_qa, h->q, dh, h->H, M, 128))
    return h->fail(IVIT_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation buffer");
  if (int r = setup_persistent(h)) return r;
  if (int r = setup_stream(h)) return r;
  IVIT_CK(h, cudaDeviceSynchronize());
  return IVIT_OK;
}

void release(ivit_handle* h) {
  if (h->sk_args.trace) cudaFree(h->sk_args.trace);
  h->sk_args.trace = nullptr;
  if (h->sk_mem) cudaFree(h->sk_mem);
  h->sk_mem = nullptr;
  if (h->pt_args.trace) cudaFree(h->pt_args.trace);
  h->pt_args.trace = nullptr;
  if (h->pt_mem) cudaFree(h->pt_mem);
  h->pt_mem = nullptr;
  if (h->graph_full) cudaGraphExecDestroy(h->graph_full);
  if (h->graph_inc) cudaGraphExecDestroy(h->graph_inc);
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  if (h->cap_stream2) cudaStreamDestroy(h->cap_stream2);
  h->cap_stream2 = nullptr;
  h->graph_full = h->graph_inc = nullptr;
  h->cap_stream = nullptr;
  if (h->wmem) cudaFree(h->wmem);
  if (h->smem) cudaFree(h->smem);
  if (h->stamps) cudaFree(h->stamps);
  h->stamps = nullptr;
  h->wmem = h->smem = nullptr;
}

// Algorithmic bytes of one GEMM launch at M rows (weights, input rows, output rows, bias).
double gemm_bytes(int n_out, int k, int kind, long long M) {
  const double out_b = kind == ivit::kEpiF32Bias ? 4.0 : kind == ivit::kEpiResid || kind == ivit::kEpiScore ? 8.0 : 2.0;
  return 2.0 * n_out * k + 2.0 * M * k + out_b * M * n_out + 4.0 * n_out;
}

// Before each launch: the stamp slot of the launch in timeline mode (else none).
void next_launch(ivit_handle* h, int family, const ivit::GemmArgs* ga = nullptr, int other_kind = 0) {
  ivit::g_stamp = nullptr;
  if (!h->timeline || !h->stamps || h->stamp_used >= h->stamp_cap) return;
  ivit::g_stamp = h->stamps + static_cast<size_t>(h->stamp_used++) * 2 * ivit::kStampCtas;
  TimelineSlot sl;
  sl.family = family;
  sl.kind = other_kind;
  if (ga) {
    sl.n_out = ga->n_out;
    sl.k = ga->k;
    sl.kind = ga->epi.kind;
    sl.m_static = ga->d_rows ? -1 : ga->m_static;
  }
  h->slots_cur.push_back(sl);
}

int gemm(ivit_handle* h, const GemmPlan& plan, const CUtensorMap& tw, const bf16* w, const ActMaps& x,
         ivit::GemmArgs a, cudaStream_t s) {
  a.err = h->err;
  a.partials = h->gemm_partials;
  a.defer = plan.defer ? 1 : 0;
  a.vsplit = plan.defer ? plan.splits : 0;
  a.w = w;
  a.x = x.base;
  // (one plan for every row count: more rows than expected go to two CTAs)
  a.row_groups = h->row_groups;
  next_launch(h, kFamGemm, &a);
  IVIT_CK(h, plan.nt ? ivit::launch_gemm_rows(plan.nt, a, s)
                     : ivit::launch_gemm_pair(plan.bn, tw, x.of(plan), a, plan.n_pairs, s));
  ++h->launches;
  return IVIT_OK;
}

// Debug aid (IVIT_TRACE): mean time of each phase kind of the last persistent launch.
void print_trace(ivit_handle* h, cudaStream_t s) {
  std::vector<unsigned long long> t(4096);
  if (cudaStreamSynchronize(s) != cudaSuccess) return;
  cudaMemcpy(t.data(), h->pt_args.trace, t.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost);
  const int n = static_cast<int>(t[0]);
  static const char* names[9] = {"qkv gemm", "qkv reduce", "attention", "out gemm", "out red+LN2",
                                 "up gemm", "up reduce", "down gemm", "down red+LN"};
  double acc[9] = {0};
  int cnt[9] = {0};
  for (int i = 2; i < n; ++i) {  // entry 1 = start, entry 2 = after the first LN phase
    const int k = (i - 2) % 9;
    acc[k] += 1e-3 * static_cast<double>(t[1 + i] - t[i]);
    ++cnt[k];
  }
  std::fprintf(stderr, "ivit trace: %d phases, total %.1f us, first LN %.1f us\n", n - 1,
               1e-3 * static_cast<double>(t[n] - t[1]), 1e-3 * static_cast<double>(t[2] - t[1]));
  for (int k = 0; k < 9; ++k)
    if (cnt[k]) std::fprintf(stderr, "  %-12s %6.2f us x %d\n", names[k], acc[k] / cnt[k], cnt[k]);
}

// Debug aid (IVIT_TRACE): stage durations of the last weight-streaming launch (critical
// path: the last CTA's arrival at each grid barrier after the previous barrier's exit),
// barrier latencies, and per-task phase times.
void print_stream_trace(ivit_handle* h, cudaStream_t s) {
  const int L = h->L, G = h->sk_grid, NB = h->sk_args.n_barriers;
  std::vector<unsigned long long> t(static_cast<size_t>(NB) * (G + 1) + 64 * static_cast<size_t>(G));
  if (cudaStreamSynchronize(s) != cudaSuccess) return;
  cudaMemcpy(t.data(), h->sk_args.trace, t.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost);
  static const char* names[7] = {"qkv", "attention", "out", "ln2", "up", "down", "ln1"};
  double dur[7] = {0}, lat[7] = {0}, mean_arr[7] = {0};
  int cnt[7] = {0};
  for (int k = 1; k < NB; ++k) {
    unsigned long long mx = 0;
    double sum = 0;
    for (int c = 0; c < G; ++c) {
      mx = std::max(mx, t[static_cast<size_t>(k) * G + c]);
      sum += static_cast<double>(t[static_cast<size_t>(k) * G + c]);
    }
    const double prev_exit = static_cast<double>(t[static_cast<size_t>(NB) * G + k - 1]);
    const double exit_k = static_cast<double>(t[static_cast<size_t>(NB) * G + k]);
    const int j = (k - 1) % 7;
    dur[j] += 1e-3 * (static_cast<double>(mx) - prev_exit);
    lat[j] += 1e-3 * (exit_k - static_cast<double>(mx));
    mean_arr[j] += 1e-3 * (sum / G - prev_exit);
    ++cnt[j];
  }
  std::fprintf(stderr, "ivit stream trace: %d barriers, first exit %.1f us after CTA 0 arrived, last exit %.1f us\n",
               NB, 1e-3 * static_cast<double>(t[static_cast<size_t>(NB) * G] - t[0]),
               1e-3 * static_cast<double>(t[static_cast<size_t>(NB) * G + NB - 1] - t[0]));
  for (int j = 0; j < 7; ++j)
    if (cnt[j])
      std::fprintf(stderr, "  %-9s stage %6.2f us (mean arrival %6.2f) barrier %5.2f us\n", names[j], dur[j] / cnt[j],
                   mean_arr[j] / cnt[j], lat[j] / cnt[j]);
  static const char* kinds[6] = {"qkv", "out", "up", "down", "attn", "rows"};
  static const char* slots[6][7] = {{"w-wait", "B", "mma", "acc-wait", "epilogue", "fixup", ""},
                                    {"w-wait", "B", "mma", "acc-wait", "epilogue", "fixup", ""},
                                    {"w-wait", "B", "mma", "acc-wait", "epilogue", "fixup", ""},
                                    {"w-wait", "B", "mma", "acc-wait", "epilogue", "fixup", ""},
                                    {"kv+patch", "compute", "scores", "softmax+pv", "", "", ""},
                                    {"row", "", "", "", "", "", ""}};
  const size_t base = static_cast<size_t>(NB) * (G + 1);
  for (int g = 0; g < 6; ++g) {
    double n = 0;
    for (int c = 0; c < G; ++c) n += static_cast<double>(t[base + (c * 8 + g) * 8 + 7]);
    if (n == 0) continue;
    std::fprintf(stderr, "  %-5s x%6.0f/call:", kinds[g], n);
    for (int k = 0; k < 7; ++k) {
      if (!slots[g][k][0]) continue;
      double sum = 0;
      for (int c = 0; c < G; ++c) sum += 1e-3 * static_cast<double>(t[base + (c * 8 + g) * 8 + k]);
      std::fprintf(stderr, " %s %.2f", slots[g][k], sum / n);
    }
    std::fprintf(stderr, "\n");
  }
  (void)L;
  cudaMemset(h->sk_args.trace, 0, t.size() * sizeof(unsigned long long));
}

// CTAs per SM (1, 2) of the few-query attention where it is the faster one for about m_expected
// updated rows, else 0: a cost model in microseconds per launch, fitted like plan_gemm's.  That kernel takes 2.0 us (1.3 for
// heads of up to 64) + 1.5 us per 256 keys of a 72-wide head for a round of 16-query items over
// the SMs, two rounds of heads of up to 64 on twice the CTAs 0.85 times that; the other one 4.0 us + 1.0 us per key block for a round of 128-query items over two
// CTAs per SM.  With 16 heads of 72: 26 queries x 256 keys 3.9 us against 6.1, 128 x 256 4.2
// against 6.9, 256 x 256 7.2 against 7.3 (and 4 % of a full encode slower, for its second round
// keeps the next kernel out), 100 x 1024 8.7 against 14.4, 32 views of 96 x 1024 171 against 38;
// 6 views of 196 x 196 with 3 heads of 64 5.6 (4.9 with two CTAs per SM) against 6.8.  Only this
// kernel has an exact form, which such calls take at any size.
int attention_few(const ivit_handle* h, int m_expected, bool exact) {
  const int dh = h->D / h->H;
  auto rounds = [&](int tile, int ctas) {  // a view's last tile is half full on average
    const double tiles = std::max<double>(h->SV, static_cast<double>(m_expected) / tile + 0.5 * h->SV);
    const double full = static_cast<double>(h->SV) * ((h->N + tile - 1) / tile);
    return std::ceil(h->H * std::min(tiles, full) / ctas);
  };
  const int kb = ivit::attention_key_block((dh + 15) & ~15);
  const double round = (dh <= 64 ? 1.3 : 2.0) + 1.5 * dh / 72.0 * ((h->N + 255) / 256);
  const bool two = dh <= 64 && rounds(16, h->num_sms) > 1;
  const double few = 0.4 + round * (two ? 0.85 * 2 * rounds(16, 2 * h->num_sms) : rounds(16, h->num_sms));
  const double many = 4.0 + rounds(128, 2 * h->num_sms) * ((h->N + kb - 1) / kb);
  return h->attn_forced == 0 || (h->attn_forced < 0 && !exact && few >= many) ? 0 : two ? 2 : 1;
}

// Attention of the updated queries (about m_expected) over all tokens of their view for one layer,
// with `exact` on probabilities in fp32.
int attention(ivit_handle* h, const LayerW& w, const bf16* ck, const bf16* cv, int m_expected, bool exact,
              cudaStream_t s) {
  const int N = h->N, D = h->D, SV = h->SV;
  if (h->attn_tc) {
    ivit::AttnTcArgs at;
    at.cu_rows = h->cu_rows;
    at.q = h->q;
    at.k = ck;
    at.v = cv;
    at.o = h->o;
    at.err = h->err;
    at.n_tok = N;
    at.dim = D;
    at.dh = D / h->H;
    at.heads = h->H;
    at.sv = SV;
    next_launch(h, kFamAttn);
    at.stamp = ivit::g_stamp;
    const int few = attention_few(h, m_expected, exact);
    IVIT_CK(h, few ? ivit::launch_attention_rows(at, h->num_sms, few, exact, s)
                   : ivit::launch_attention_tc(h->tm_qa, w.tm_ak, w.tm_av, at, h->num_sms, s));
  } else {
    next_launch(h, kFamAttn);
    IVIT_CK(h, ivit::launch_attention(w.tm_ck, w.tm_cv, h->q, ck, cv, h->cu_rows, h->rowtok, h->o, SV, N, D, h->H,
                                      (std::max(1, m_expected / SV) + 31) / 32, s));
  }
  ++h->launches;
  return IVIT_OK;
}

// What a residual GEMM launched with plan pl left for the next layer norm to add.
ivit::PendingSum pending_sum(ivit_handle* h, const GemmPlan& pl, const float* bias) {
  ivit::PendingSum p;
  if (!pl.defer) return p;
  p.partials = h->gemm_partials;
  p.bias = bias;
  p.csize = pl.splits;
  p.bn = pl.bn;
  p.n_ft = (h->D + 127) / 128;
  return p;
}

// The blocks under the MLP-on-all-tokens reading (Sec. III-B, after Eq. 5): x holds
// every token's residual stream (row = token v*N + i).  Per layer, the updated tokens
// (packed rows, rowtok) run LN1, QKV with the K/V scatter (Eq. 5), attention over all
// tokens and the output projection, whose result replaces their rows of the layer's
// attention-output cache; then every token adds its cached attention output to its
// stream (fused into LN2) and runs the MLP; the final LN writes every output token.
int run_layers_mlp_all(ivit_handle* h, const GemmPlan* plan, int m_expected, cudaStream_t s) {
  const ivit_config& c = h->cfg;
  const int N = h->N, D = h->D, F = h->F, SV = h->SV, M = h->M_max;
  const int* total = h->cu_rows + SV;
  // The down-projection's residual update of every token may still be split over the GEMM
  // scratch: the next layer's LN1 reads it for the updated tokens, its LN2 adds it to x.
  ivit::PendingSum pend;
  for (int l = 0; l < h->L; ++l) {
    const LayerW& w = h->layers[l];
    bf16* ck = h->cacheK + static_cast<size_t>(l) * M * D;
    bf16* cv = h->cacheV + static_cast<size_t>(l) * M * D;
    float* al = h->acache + static_cast<size_t>(l) * M * D;
    next_launch(h, kFamLN);
    if (pend.partials)
      IVIT_CK(h, ivit::launch_layernorm_sum(total, h->x, pend, nullptr, h->rowtok, w.ln1g, w.ln1b, h->xn, nullptr, D,
                                            c.ln_eps, M, h->row_grid, s));
    else
      IVIT_CK(h, ivit::launch_layernorm_ex(total, h->x, nullptr, h->rowtok, w.ln1g, w.ln1b, h->xn, nullptr, D,
                                           c.ln_eps, M, h->row_grid, s));
    ++h->launches;
    {
      ivit::GemmArgs a;
      a.n_out = 3 * D;
      a.k = D;
      a.d_rows = total;
      a.epi.kind = ivit::kEpiQKV;
      a.epi.bias = w.bqkv;
      a.epi.out_bf16 = h->q;
      a.epi.ld_out = D;
      a.epi.cache_k = ck;
      a.epi.cache_v = cv;
      a.epi.rowtok = h->rowtok;
      a.epi.dim = D;
      if (int r = gemm(h, plan[kGemmQKV], w.tm_qkv, w.wqkv, h->tm_xn, a, s)) return r;
    }
    if (int r = attention(h, w, ck, cv, m_expected, false, s)) return r;
    {
      ivit::GemmArgs a;
      a.n_out = D;
      a.k = D;
      a.d_rows = total;
      a.epi.kind = ivit::kEpiScatterF32;
      a.epi.bias = w.bo;
      a.epi.out_f32 = al;
      a.epi.ld_out = D;
      a.epi.rowtok = h->rowtok;
      if (int r = gemm(h, plan[kGemmO], w.tm_o, w.wo, h->tm_o, a, s)) return r;
    }
    next_launch(h, kFamLN);
    if (pend.partials)
      IVIT_CK(h, ivit::launch_layernorm_sum(h->m_all, h->x, pend, al, nullptr, w.ln2g, w.ln2b, h->xn, nullptr, D,
                                            c.ln_eps, M, h->row_grid, s));
    else
      IVIT_CK(h, ivit::launch_layernorm_ex(h->m_all, h->x, al, nullptr, w.ln2g, w.ln2b, h->xn, nullptr, D, c.ln_eps,
                                           M, h->row_grid, s));
    ++h->launches;
    {
      ivit::GemmArgs a;
      a.n_out = F;
      a.k = D;
      a.m_static = M;
      a.epi.kind = ivit::kEpiGelu;
      a.epi.bias = w.b1;
      a.epi.out_bf16 = h->hbuf;
      a.epi.ld_out = F;
      a.epi.gelu_mode = c.gelu;
      if (int r = gemm(h, h->plan_full[kGemmUp], w.tm_1, w.w1, h->tm_xn, a, s)) return r;
    }
    {
      ivit::GemmArgs a;
      a.n_out = D;
      a.k = F;
      a.m_static = M;
      a.epi.kind = ivit::kEpiResid;
      a.epi.bias = w.b2;
      a.epi.out_f32 = h->x;
      a.epi.ld_out = D;
      if (int r = gemm(h, h->plan_full[kGemmDown], w.tm_2, w.w2, h->tm_h, a, s)) return r;
      pend = pending_sum(h, h->plan_full[kGemmDown], w.b2);
    }
  }
  next_launch(h, kFamLN);
  if (pend.partials)
    IVIT_CK(h, ivit::launch_layernorm_sum(h->m_all, h->x, pend, nullptr, nullptr, h->lnfg, h->lnfb, h->tok_out, nullptr,
                                          D, c.ln_eps, M, h->row_grid, s));
  else
    IVIT_CK(h, ivit::launch_layernorm(h->m_all, h->x, h->lnfg, h->lnfb, h->tok_out, nullptr, D, c.ln_eps, M,
                                      h->row_grid, s));
  ++h->launches;
  (void)N;
  return IVIT_OK;
}

// Per layer {LN1, QKV + K/V cache scatter (Eq. 4-5), attention, out-proj + residual,
// LN2, MLP up + GELU, MLP down + residual}, then the final LN scattered into the
// final-token cache, with the given launch plans, made for about m_expected updated rows.
// `exact`: the softmax's probabilities and GELU's tanh to the precision of fp32.
int run_layers(ivit_handle* h, const GemmPlan* plan, int m_expected, bool exact, cudaStream_t s) {
  const ivit_config& c = h->cfg;
  const int D = h->D, F = h->F, SV = h->SV, M = h->M_max;
  const int* total = h->cu_rows + SV;
  // A residual update still split over the GEMM scratch (deferred out-projection or
  // MLP-down GEMM): the next layer norm adds it to x.
  ivit::PendingSum pend;
  auto layernorm = [&](const float* g, const float* b, bf16* y, const int* dst) -> int {
    next_launch(h, kFamLN);
    if (pend.partials) {
      IVIT_CK(h, ivit::launch_layernorm_sum(total, h->x, pend, nullptr, nullptr, g, b, y, dst, D, c.ln_eps, M,
                                            h->row_grid, s));
      pend = ivit::PendingSum();
    } else {
      IVIT_CK(h, ivit::launch_layernorm(total, h->x, g, b, y, dst, D, c.ln_eps, M, h->row_grid, s));
    }
    ++h->launches;
    return IVIT_OK;
  };
  auto residual = [&](const GemmPlan& pl, const float* bias, const CUtensorMap& tw, const bf16* wp,
                      const ActMaps& tx, int k) -> int {
    ivit::GemmArgs a;
    a.n_out = D;
    a.k = k;
    a.d_rows = total;
    a.epi.kind = ivit::kEpiResid;
    a.epi.bias = bias;
    a.epi.out_f32 = h->x;
    a.epi.ld_out = D;
    if (int r = gemm(h, pl, tw, wp, tx, a, s)) return r;
    pend = pending_sum(h, pl, bias);
    return IVIT_OK;
  };
  for (int l = 0; l < h->L; ++l) {
    const LayerW& w = h->layers[l];
    bf16* ck = h->cacheK + static_cast<size_t>(l) * M * D;
    bf16* cv = h->cacheV + static_cast<size_t>(l) * M * D;
    if (int r = layernorm(w.ln1g, w.ln1b, h->xn, nullptr)) return r;
    {
      ivit::GemmArgs a;
      a.n_out = 3 * D;
      a.k = D;
      a.d_rows = total;
      a.epi.kind = ivit::kEpiQKV;
      a.epi.bias = w.bqkv;
      a.epi.out_bf16 = h->q;
      a.epi.ld_out = D;
      a.epi.cache_k = ck;
      a.epi.cache_v = cv;
      a.epi.rowtok = h->rowtok;
      a.epi.dim = D;
      if (int r = gemm(h, plan[kGemmQKV], w.tm_qkv, w.wqkv, h->tm_xn, a, s)) return r;
    }
    if (int r = attention(h, w, ck, cv, m_expected, exact, s)) return r;
    if (int r = residual(plan[kGemmO], w.bo, w.tm_o, w.wo, h->tm_o, D)) return r;
    if (int r = layernorm(w.ln2g, w.ln2b, h->xn, nullptr)) return r;
    {
      ivit::GemmArgs a;
      a.n_out = F;
      a.k = D;
      a.d_rows = total;
      a.epi.kind = exact && c.gelu == IVIT_GELU_TANH ? ivit::kEpiGeluTanhf : ivit::kEpiGelu;
      a.epi.bias = w.b1;
      a.epi.out_bf16 = h->hbuf;
      a.epi.ld_out = F;
      a.epi.gelu_mode = c.gelu;
      if (int r = gemm(h, plan[kGemmUp], w.tm_1, w.w1, h->tm_xn, a, s)) return r;
    }
    if (int r = residual(plan[kGemmDown], w.b2, w.tm_2, w.w2, h->tm_h, F)) return r;
  }
  return layernorm(h->lnfg, h->lnfb, h->tok_out, h->rowtok);
}

// Under capture of an incremental graph with row bands: a switch node after the
// gather (which sets its value from the row count) with one body per band, each the
// layer chain with that band's launch plans, captured on a second stream.  The
// launches of one body count for the call.
int capture_band_bodies(ivit_handle* h, cudaStream_t s) {
  cudaStreamCaptureStatus st;
  cudaGraph_t graph = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  IVIT_CK(h, cudaStreamGetCaptureInfo(s, &st, nullptr, &graph, &deps, nullptr, &ndeps));
  cudaGraphNodeParams np = {};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = static_cast<cudaGraphConditionalHandle>(h->bands.handle);
  np.conditional.type = cudaGraphCondTypeSwitch;
  np.conditional.size = static_cast<unsigned>(h->n_bands);
  cudaGraphNode_t node;
  IVIT_CK(h, cudaGraphAddNode(&node, graph, deps, nullptr, ndeps, &np));
  IVIT_CK(h, cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
  const int64_t pre = h->launches;
  const int pre_stamps = h->stamp_used;
  const size_t pre_slots = h->slots_cur.size();
  for (int b = 0; b < h->n_bands; ++b) {  // (the same sequence of launches, of which one runs per call: one set of stamps)
    h->launches = pre;
    h->stamp_used = pre_stamps;
    h->slots_cur.resize(pre_slots);
    IVIT_CK(h, cudaStreamBeginCaptureToGraph(h->cap_stream2, np.conditional.phGraph_out[b], nullptr, nullptr, 0,
                                             cudaStreamCaptureModeThreadLocal));
    const int r = run_layers(h, h->plan_band[b], band_rows(h, b), false, h->cap_stream2);
    cudaGraph_t body = nullptr;
    const cudaError_t e = cudaStreamEndCapture(h->cap_stream2, &body);
    if (r) return r;
    if (e != cudaSuccess) return h->cuda_fail("cudaStreamEndCapture (band body)", e);
  }
  return IVIT_OK;
}

// The start of a call's launch record; its first launch is patchify.
void begin_record(ivit_handle* h) {
  h->launches = 0;
  h->slots_cur.clear();
  h->stamp_used = 0;
  next_launch(h, kFamOther, nullptr, 0);
}

// Whether the library's kernels may use a caller's pointer where it points: memory of the handle's
// own GPU, aligned to `align`.  The copy engine carries everything else that it can reach, another
// GPU's memory or pinned host memory, where a kernel would fault or run at the link's latency.
bool in_place(const ivit_handle* h, const void* p, uintptr_t align) {
  if (reinterpret_cast<uintptr_t>(p) & (align - 1)) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice && at.device == h->device;
}

// The call's first kernel, from the caller's frames (eager, also before a replayed graph).
int run_patchify(ivit_handle* h, const uint8_t* frames, cudaStream_t s) {
  const ivit_config& c = h->cfg;
  // (patch rows of an even number of bytes are read two at a time)
  if (!in_place(h, frames, c.patch % 2 ? 1 : 2)) {
    const size_t bytes = static_cast<size_t>(h->SV) * c.img_h * c.img_w * 3;
    IVIT_CK(h, cudaMemcpyAsync(h->frames_buf, frames, bytes, cudaMemcpyDefault, s));
    frames = h->frames_buf;
  }
  if (h->timeline && h->stamps)  // CTAs that leave early write nothing: clear the last call's stamps
    IVIT_CK(h, cudaMemsetAsync(h->stamps, 0, static_cast<size_t>(h->stamp_cap) * 2 * ivit::kStampCtas *
                                                 sizeof(unsigned long long), s));
  begin_record(h);
  IVIT_CK(h, ivit::launch_patchify(frames, h->patches, h->SV, c.img_h, c.img_w, c.patch, h->KPAD, s));
  ++h->launches;
  return IVIT_OK;
}

// Launch plans of a call, and the updated rows that it expects.  A cold view updates every token,
// a warm one k of them under top-k, so those calls take the band of that count: a cold 256-token
// So400m view, four layers, takes 194 us, and 535 (top-k) or 354 (threshold) with the plans of a
// tenth of its tokens.  Other calls' counts are known only on the device; a tenth is assumed.  (Any
// count runs correctly: top-k selects NaN scores beside its k.)
const GemmPlan* plan_of_call(const ivit_handle* h, bool full, int& m_expected) {
  m_expected = h->M_max;
  if (full) return h->plan_full;
  const bool topk = h->cfg.select_mode == IVIT_SEL_TOPK;
  const int n_cold = static_cast<int>(std::count_if(h->cold.begin(), h->cold.end(), [](uint8_t c) { return c != 0; }));
  m_expected = std::max(1, h->M_max / 10);
  if (!n_cold && (!topk || h->cfg.mlp_tokens == IVIT_MLP_ALL)) return h->plan_inc;
  const int warm = h->SV - n_cold;
  m_expected = std::max(1, n_cold * h->N + (topk ? warm * std::min(h->cfg.topk, h->N) : warm * h->N / 10));
  int b = 0;
  while (b + 1 < h->n_bands && m_expected > h->band_ub[b]) ++b;
  return h->plan_band[b];
}

// Enqueues the rest of the chain for one frame per view on `s` (eagerly or under capture).
int run_core(ivit_handle* h, bool full, cudaStream_t s) {
  const ivit_config& c = h->cfg;
  const int N = h->N, D = h->D, SV = h->SV, M = h->M_max;
  ivit::ColdMask cm;
  std::memset(&cm, 0, sizeof cm);
  for (int v = 0; v < SV; ++v)
    if (full || h->cold[v]) cm.bits[v >> 5] |= 1u << (v & 31);
  int m_expected = 0;
  const GemmPlan* plan = plan_of_call(h, full, m_expected);
  const int* total = h->cu_rows + SV;

  {
    ivit::GemmArgs a;
    a.n_out = D;
    a.k = h->KPAD;
    a.m_static = M;
    a.epi.kind = h->one_ref && !full ? ivit::kEpiScore : ivit::kEpiF32Bias;
    a.epi.bias = h->b_pe;
    a.epi.out_f32 = h->e_t;
    a.epi.ld_out = D;
    a.epi.score = h->score_parts;
    if (int r = gemm(h, plan[kGemmEmbed], h->tm_pe, h->w_pe, h->tm_patches, a, s)) return r;
  }
  const float* score_vec = h->e_t;  // what the references of updated tokens are refreshed from
  if (h->one_ref) score_vec = nullptr;  // (they hold it already)
  if (c.score_source == IVIT_SCORE_KEY0) {
    // Eq. 3 on first-layer keys of every token: W_K LN1(e + pos) + b_K (x, xn are free
    // until the updated rows are gathered below)
    next_launch(h, kFamOther, nullptr, 3);  // gather
    IVIT_CK(h, ivit::launch_gather(h->m_all, h->rowtok_all, ivit::RowLists(), h->e_t, h->pos, h->x, nullptr, h->e_ref, N, D, 0,
                                   cm, M, h->row_grid, s));
    next_launch(h, kFamLN);
    IVIT_CK(h, ivit::launch_layernorm(h->m_all, h->x, h->layers[0].ln1g, h->layers[0].ln1b, h->xn, nullptr, D,
                                      c.ln_eps, M, h->row_grid, s));
    h->launches += 2;
    ivit::GemmArgs a;
    a.n_out = D;
    a.k = D;
    a.m_static = M;
    a.epi.kind = ivit::kEpiF32Bias;
    a.epi.bias = h->layers[0].bqkv + D;
    a.epi.out_f32 = h->key_t;
    a.epi.ld_out = D;
    if (int r = gemm(h, h->plan_keys, h->tm_wk0, nullptr, h->tm_xn, a, s)) return r;
    score_vec = h->key_t;
  }
  if (!full && !h->one_ref) {
    next_launch(h, kFamOther, nullptr, 1);  // score
    IVIT_CK(h, ivit::launch_score(score_vec, h->e_ref, h->sims, M, D, c.ref_mode == IVIT_REF_PREV_FRAME, s));
    ++h->launches;
  }
  const ivit::RowLists lists{h->idx, h->cu_rows, SV, N};
  next_launch(h, kFamOther, nullptr, 2);  // select
  IVIT_CK(h, ivit::launch_select(h->sims, h->score_parts, (D + 127) / 128, N, SV, full ? IVIT_SEL_THRESHOLD : c.select_mode, c.threshold,
                                 c.topk, cm, h->idx, h->counts, h->cu_rows, h->done_ctr, s));
  ++h->launches;
  if (c.mlp_tokens == IVIT_MLP_ALL) {
    // every token's residual stream (token-indexed), then the references of the updated
    // tokens (last-refresh mode, cold views) without touching x
    next_launch(h, kFamOther, nullptr, 3);  // gather
    IVIT_CK(h, ivit::launch_gather(h->m_all, h->rowtok_all, ivit::RowLists(), h->e_t, h->pos, h->x, nullptr, h->e_ref, N, D, 0,
                                   cm, M, h->row_grid, s));
    next_launch(h, kFamOther, nullptr, 3);  // gather
    IVIT_CK(h, ivit::launch_gather(total, h->rowtok, lists, h->e_t, h->pos, nullptr, score_vec, h->e_ref, N, D,
                                   c.ref_mode == IVIT_REF_LAST_REFRESH, cm, M, h->row_grid, s));
    h->launches += 2;
    return run_layers_mlp_all(h, plan, m_expected, s);
  }
  ivit::RowBands bands;  // (no switch node: handle 0)
  if (h->capture_bands) {
    cudaStreamCaptureStatus st;
    cudaGraph_t graph = nullptr;
    IVIT_CK(h, cudaStreamGetCaptureInfo(s, &st, nullptr, &graph));
    cudaGraphConditionalHandle ch;
    IVIT_CK(h, cudaGraphConditionalHandleCreate(&ch, graph, 0, cudaGraphCondAssignDefault));
    bands.handle = static_cast<unsigned long long>(ch);
    bands.n = h->n_bands;
    for (int b = 0; b < h->n_bands; ++b) bands.ub[b] = h->band_ub[b];
    h->bands = bands;
  }
  next_launch(h, kFamOther, nullptr, 3);  // gather
  IVIT_CK(h, ivit::launch_gather(total, h->rowtok, lists, h->e_t, h->pos, h->x, score_vec, h->e_ref, N, D,
                                 c.ref_mode == IVIT_REF_LAST_REFRESH, cm, M, h->row_grid, s, bands));
  ++h->launches;

  bool any_cold = false;
  for (int v = 0; v < SV; ++v) any_cold = any_cold || (cm.bits[v >> 5] >> (v & 31)) & 1u;
  if (h->stream_ok && !full && !any_cold) {
    IVIT_CK(h, cudaMemsetAsync(h->sk_args.sync, 0, h->sk_sync_bytes, s));
    IVIT_CK(h, ivit::launch_stream(h->sk_args, h->sk_grid, h->sk_smem, s));
    ++h->launches;
    if (h->sk_args.trace) {
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      cudaStreamIsCapturing(s, &cs);
      if (cs == cudaStreamCaptureStatusNone) print_stream_trace(h, s);
    }
    return IVIT_OK;
  }
  if (h->persistent) {
    IVIT_CK(h, cudaMemsetAsync(h->pt_args.gbar, 0, 4 * sizeof(unsigned), s));
    IVIT_CK(h, ivit::launch_persistent(h->pt_args, h->pt_grid, h->pt_smem, s));
    ++h->launches;
    if (h->pt_args.trace && !h->timeline) {
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      cudaStreamIsCapturing(s, &cs);
      if (cs == cudaStreamCaptureStatusNone) print_trace(h, s);
    }
    return IVIT_OK;
  }
  if (h->capture_bands) return capture_band_bodies(h, s);
  // The full encodes of small encoders have their probabilities and tanh in fp32, where every other
  // call has bf16 and the hardware's tanh (what the persistent kernel, which these encodes once
  // took, computes): six 196-token views of ViT-Tiny take 380 us either way.
  const bool exact = full && D <= 384 && N <= 256;
  return run_layers(h, plan, m_expected, exact, s);
}

int capture_once(ivit_handle* h, bool full, cudaGraphExec_t* exec, int64_t* launches);

// The incremental graph of the kernel chain is captured with a switch over the row
// bands when there are several; if that capture fails the plain graph (band 0's plans
// for every row count) is captured instead.
int capture(ivit_handle* h, bool full, cudaGraphExec_t* exec, int64_t* launches) {
  const bool chain = h->cfg.mlp_tokens == IVIT_MLP_UPDATED && !h->stream_ok && !h->persistent;
  // threshold selection: the row count is known only on the device
  if (!full && chain && h->n_bands > 1 && h->cfg.select_mode != IVIT_SEL_TOPK && rows_cross_bands(h)) {
    h->capture_bands = true;
    const int r = capture_once(h, full, exec, launches);
    h->capture_bands = false;
    if (r == IVIT_OK) return IVIT_OK;
    if (std::getenv("IVIT_DEBUG")) std::fprintf(stderr, "ivit: row-band graph failed (%s)\n", h->error.c_str());
    cudaGetLastError();
    h->n_bands = 1;
  }
  return capture_once(h, full, exec, launches);
}

int capture_once(ivit_handle* h, bool full, cudaGraphExec_t* exec, int64_t* launches) {
  IVIT_CK(h, cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
  begin_record(h);
  const int r = run_core(h, full, h->cap_stream);
  cudaGraph_t g = nullptr;
  const cudaError_t e = cudaStreamEndCapture(h->cap_stream, &g);
  if (r != IVIT_OK) {
    if (g) cudaGraphDestroy(g);
    return r;
  }
  if (e != cudaSuccess) return h->cuda_fail("cudaStreamEndCapture", e);
  const cudaError_t ei = cudaGraphInstantiate(exec, g, 0);
  cudaGraphDestroy(g);
  if (ei != cudaSuccess) return h->cuda_fail("cudaGraphInstantiate", ei);
  *launches = h->launches;
  (full ? h->slots_full : h->slots_inc) = h->slots_cur;
  return IVIT_OK;
}

int run(ivit_handle* h, const uint8_t* frames, uint16_t* out, int32_t* user_counts, bool full,
        cudaStream_t s) {
  const int SV = h->SV;
  bool any_cold = false;
  for (int v = 0; v < SV; ++v) any_cold = any_cold || h->cold[v];
  if (h->use_graphs && (full || !any_cold)) {
    cudaGraphExec_t* exec = full ? &h->graph_full : &h->graph_inc;
    int64_t* nl = full ? &h->graph_full_launches : &h->graph_inc_launches;
    if (!*exec) {
      const int r = capture(h, full, exec, nl);
      ivit::g_stamp = nullptr;
      if (r) return r;
    }
    const int r = run_patchify(h, frames, s);
    ivit::g_stamp = nullptr;
    if (r) return r;
    h->slots_last = full ? h->slots_full : h->slots_inc;
    IVIT_CK(h, cudaGraphLaunch(*exec, s));
    h->launches += *nl;
  } else {
    int r = run_patchify(h, frames, s);
    if (!r) r = run_core(h, full, s);
    ivit::g_stamp = nullptr;
    if (r) return r;
    h->slots_last = h->slots_cur;
  }
  // every output token (updated ones recomputed, the rest from the final-token cache) and the
  // views' counts, to the caller
  const size_t tok_bytes = static_cast<size_t>(h->M_max) * h->D * 2;
  if (out && !in_place(h, out, 16)) {
    IVIT_CK(h, cudaMemcpyAsync(out, h->tok_out, tok_bytes, cudaMemcpyDefault, s));
    out = nullptr;
  }
  if (user_counts && !in_place(h, user_counts, 4)) {
    IVIT_CK(h, cudaMemcpyAsync(user_counts, h->counts, SV * sizeof(int), cudaMemcpyDefault, s));
    user_counts = nullptr;
  }
  if (out || user_counts) {
    h->slots_cur = h->slots_last;  // (a replayed graph's record, or this call's)
    h->stamp_used = static_cast<int>(h->slots_last.size());
    next_launch(h, kFamOther, nullptr, 4);
    h->slots_last = h->slots_cur;
    IVIT_CK(h, ivit::launch_outputs(h->tok_out, out, tok_bytes, h->counts, user_counts, SV, h->num_sms, s));
    ivit::g_stamp = nullptr;
    ++h->launches;
  }
  for (int v = 0; v < SV; ++v) h->cold[v] = 0;

  return IVIT_OK;
}

}  // namespace

extern "C" {

size_t ivit_weights_size(const ivit_config* cfg) {
  if (validate(cfg)) return 0;
  return weights_count(cfg);
}

int ivit_create(const ivit_config* cfg, const uint16_t* weights_bf16_host, ivit_handle** out) {
  if (!out) {
    g_create_error = "null output pointer";
    return IVIT_ERR_ARG;
  }
  *out = nullptr;
  if (const char* why = validate(cfg)) {
    g_create_error = why;
    return cfg ? IVIT_ERR_SHAPE : IVIT_ERR_ARG;
  }
  if (!weights_bf16_host) {
    g_create_error = "null weights";
    return IVIT_ERR_ARG;
  }
  ivit_handle* h = new (std::nothrow) ivit_handle();
  if (!h) {
    g_create_error = "host allocation failed";
    return IVIT_ERR_OOM;
  }
  h->cfg = *cfg;
  const int r = setup(h, weights_bf16_host);
  if (r != IVIT_OK) {
    g_create_error = h->error;
    release(h);
    delete h;
    return r;
  }
  *out = h;
  return IVIT_OK;
}

int ivit_encode_full(ivit_handle* h, const uint8_t* frames_dev, uint16_t* tokens_out_dev, void* stream) {
  if (!h) return IVIT_ERR_ARG;
  if (!frames_dev) return h->fail(IVIT_ERR_ARG, "null frames");
  return run(h, frames_dev, tokens_out_dev, nullptr, true, static_cast<cudaStream_t>(stream));
}

int ivit_encode_incremental(ivit_handle* h, const uint8_t* frames_dev, uint16_t* tokens_out_dev,
                            int32_t* changed_count_dev, void* stream) {
  if (!h) return IVIT_ERR_ARG;
  if (!frames_dev) return h->fail(IVIT_ERR_ARG, "null frames");
  // odd/even chunks (Sec. III-B): the 1st, 3rd, ... call is a full forward
  const bool full = h->cfg.schedule == IVIT_SCHED_ODD_EVEN && (h->chunk++ % 2) == 0;
  return run(h, frames_dev, tokens_out_dev, changed_count_dev, full, static_cast<cudaStream_t>(stream));
}

int ivit_get_changed(ivit_handle* h, int sv, int32_t* idx_dev, int32_t* count_dev, void* stream) {
  if (!h) return IVIT_ERR_ARG;
  if (sv < 0 || sv >= h->SV) return h->fail(IVIT_ERR_ARG, "view index out of range");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (idx_dev)
    IVIT_CK(h, cudaMemcpyAsync(idx_dev, h->idx + static_cast<size_t>(sv) * h->N, h->N * sizeof(int),
                               cudaMemcpyDeviceToDevice, s));
  if (count_dev)
    IVIT_CK(h, cudaMemcpyAsync(count_dev, h->counts + sv, sizeof(int), cudaMemcpyDeviceToDevice, s));
  return IVIT_OK;
}

int ivit_get_cache(ivit_handle* h, int which, int layer, void* dst_dev, void* stream) {
  if (!h) return IVIT_ERR_ARG;
  if (!dst_dev) return h->fail(IVIT_ERR_ARG, "null destination");
  const size_t elems = static_cast<size_t>(h->M_max) * h->D;
  const void* src = nullptr;
  size_t bytes = elems * 2;
  if (which == 0 || which == 1) {
    if (layer < 0 || layer >= h->L) return h->fail(IVIT_ERR_ARG, "layer out of range");
    src = (which == 0 ? h->cacheK : h->cacheV) + static_cast<size_t>(layer) * elems;
  } else if (which == 2) {
    src = h->tok_out;
  } else if (which == 3) {
    src = h->e_ref;
    bytes = elems * 4;
  } else if (which == 4 && h->acache) {
    if (layer < 0 || layer >= h->L) return h->fail(IVIT_ERR_ARG, "layer out of range");
    src = h->acache + static_cast<size_t>(layer) * elems;
    bytes = elems * 4;
  } else {
    return h->fail(IVIT_ERR_ARG, "bad cache selector");
  }
  IVIT_CK(h, cudaMemcpyAsync(dst_dev, src, bytes, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)));
  return IVIT_OK;
}

int ivit_reset(ivit_handle* h, int stream_index) {
  if (!h) return IVIT_ERR_ARG;
  if (stream_index < -1 || stream_index >= h->cfg.n_streams)
    return h->fail(IVIT_ERR_ARG, "stream index out of range");
  for (int v = 0; v < h->SV; ++v)
    if (stream_index == -1 || v / h->cfg.n_views == stream_index) h->cold[v] = 1;
  return IVIT_OK;
}

int ivit_timeline(ivit_handle* h, int enable) {
  if (!h) return IVIT_ERR_ARG;
  const bool on = enable != 0;
  if (on && !h->stamps) {
    h->stamp_cap = 7 * h->L + 12;  // the launches of the longest call
    IVIT_CK(h, cudaMalloc(&h->stamps, static_cast<size_t>(h->stamp_cap) * 2 * ivit::kStampCtas *
                                          sizeof(unsigned long long)));
    IVIT_CK(h, cudaMemset(h->stamps, 0, static_cast<size_t>(h->stamp_cap) * 2 * ivit::kStampCtas *
                                            sizeof(unsigned long long)));
  }
  if (on != h->timeline) {
    // the graphs are captured again, with or without the stamps
    IVIT_CK(h, cudaDeviceSynchronize());
    if (h->graph_full) cudaGraphExecDestroy(h->graph_full);
    if (h->graph_inc) cudaGraphExecDestroy(h->graph_inc);
    h->graph_full = h->graph_inc = nullptr;
    h->timeline = on;
  }
  return IVIT_OK;
}

int ivit_timeline_read(ivit_handle* h, void* stream, double* family_ms, int64_t* family_launches,
                       double* gemm_bytes_total, double* span_ms) {
  if (!h) return IVIT_ERR_ARG;
  if (!h->timeline || !h->stamps) return h->fail(IVIT_ERR_ARG, "timeline mode is off");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t n = h->slots_last.size();
  std::vector<unsigned long long> t(n * 2 * ivit::kStampCtas);
  int rows = 0;
  IVIT_CK(h, cudaMemcpyAsync(&rows, h->cu_rows + h->SV, sizeof(int), cudaMemcpyDeviceToHost, s));
  if (n) IVIT_CK(h, cudaMemcpyAsync(t.data(), h->stamps, t.size() * sizeof(unsigned long long),
                                    cudaMemcpyDeviceToHost, s));
  IVIT_CK(h, cudaStreamSynchronize(s));
  double ms[kFamilies] = {0}, bytes = 0;
  int64_t cnt[kFamilies] = {0};
  unsigned long long first = ~0ull, last = 0;
  for (size_t i = 0; i < n; ++i) {
    unsigned long long b = ~0ull, e = 0;
    for (int c = 0; c < ivit::kStampCtas; ++c) {
      const unsigned long long sb = t[(i * ivit::kStampCtas + c) * 2], se = t[(i * ivit::kStampCtas + c) * 2 + 1];
      if (sb) b = std::min(b, sb);
      if (se) e = std::max(e, se);
    }
    const TimelineSlot& sl = h->slots_last[i];
    if (b == ~0ull) continue;  // left without a stamp (no rows)
    ++cnt[sl.family];
    if (e > b) {
      ms[sl.family] += 1e-6 * static_cast<double>(e - b);
      first = std::min(first, b);
      last = std::max(last, e);
    }
    if (sl.family == kFamGemm) bytes += gemm_bytes(sl.n_out, sl.k, sl.kind, sl.m_static >= 0 ? sl.m_static : rows);
  }
  if (std::getenv("IVIT_DEBUG")) {  // mean launch time per family and GEMM epilogue kind
    double kms[kFamilies][8] = {};
    int kn[kFamilies][8] = {};
    for (size_t i = 0; i < n; ++i) {
      unsigned long long b = ~0ull, e = 0;
      for (int c = 0; c < ivit::kStampCtas; ++c) {
        const unsigned long long sb = t[(i * ivit::kStampCtas + c) * 2], se = t[(i * ivit::kStampCtas + c) * 2 + 1];
        if (sb) b = std::min(b, sb);
        if (se) e = std::max(e, se);
      }
      const TimelineSlot& sl = h->slots_last[i];
      const int k = std::min(7, std::max(0, sl.kind));
      if (e > b && b != ~0ull) {
        kms[sl.family][k] += 1e-3 * static_cast<double>(e - b);
        ++kn[sl.family][k];
      }
    }
    static const char* fam[kFamilies] = {"gemm", "attention", "layernorm", "other"};
    for (int f = 0; f < kFamilies; ++f)
      for (int k = 0; k < 8; ++k)
        if (kn[f][k])
          std::fprintf(stderr, "ivit timeline: %s%s%d: %d launches, %.2f us each\n", fam[f], f == kFamGemm ? " epilogue " : " ",
                       k, kn[f][k], kms[f][k] / kn[f][k]);
  }
  for (int f = 0; f < kFamilies; ++f) {
    if (family_ms) family_ms[f] = ms[f];
    if (family_launches) family_launches[f] = cnt[f];
  }
  if (gemm_bytes_total) *gemm_bytes_total = bytes;
  if (span_ms) *span_ms = last > first ? 1e-6 * static_cast<double>(last - first) : 0.0;
  return IVIT_OK;
}

int ivit_device_status(ivit_handle* h, void* stream) {
  if (!h) return IVIT_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int word = 0;
  IVIT_CK(h, cudaMemcpyAsync(&word, h->err, sizeof(int), cudaMemcpyDeviceToHost, s));
  IVIT_CK(h, cudaMemsetAsync(h->err, 0, sizeof(int), s));
  IVIT_CK(h, cudaStreamSynchronize(s));
  return word;
}

int64_t ivit_last_launch_count(const ivit_handle* h) { return h ? h->launches : 0; }

void ivit_destroy(ivit_handle* h) {
  if (!h) return;
  release(h);
  delete h;
}

const char* ivit_last_error(const ivit_handle* h) {
  return h ? h->error.c_str() : g_create_error.c_str();
}

}  // extern "C"
