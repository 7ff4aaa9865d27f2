// Host side of the DMTD decode library: context, weight repacking, the cycle scheduler of
// Section 2.2 of the paper, and the C ABI declared in include/dmtd.h.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <numeric>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/dmtd.h"
#include "kernels.cuh"
#include "pass_kernel.cuh"
#include "attention_kernel.cuh"
#include "gemm_tc05.cuh"
#include "attention_tc05.cuh"
#include "small_pass.cuh"

using namespace dmtd;

namespace {

thread_local std::string g_create_error;

// Clock ticks a device-side wait (grid barrier, bulk-copy or tensor-core barrier) may spin before
// it gives up and reports through the context's error word: about a second of SM clock.
constexpr long long kDeviceWaitLimitTicks = 2000000000ll;

// Captured passes that a context keeps: both kinds for four batches or cycle lengths in turn.
constexpr int kMaxGraphs = 8;

struct LayerDev {
  PackedMat qkv, o, gu, down;
  UmmaMat qkv_u{}, o_u{}, gu_u{}, down_u{};     // second copy for the tcgen05 GEMM (contexts with many rows)
  float *w_in, *w_post, *w_qn, *w_kn;
};

}  // namespace

struct dmtd_ctx {
  dmtd_model_shape s{};
  int L_d = 0, tau = 0, max_batch = 0, max_seq = 0;
  int L_e = 0;                              // encoding layers the short passes reuse as well (ExDy); 0 = none
  int device = 0, n_sms = 0;
  cudaStream_t stream = nullptr;
  cudaStream_t capture_stream = nullptr;    // graphs are recorded here (the caller's stream may be the legacy one)
  std::string err;
  std::vector<void *> allocs;
  size_t mem[4] = {0, 0, 0, 0};             // device bytes held: atom-stream weights, tcgen05 block weights, KV cache, the rest
  int mem_kind = 3;                         // category the next allocations count towards

  // model
  std::vector<LayerDev> layers;
  PackedMat embed{};
  UmmaMat embed_u{};
  bool umma_ok = false, use_umma = true;    // tcgen05 GEMM for the projections
  int gemm_stages = 0;                      // pipeline stages of its blocks; 0: chosen per launch
  uint4 *act_blocks = nullptr;              // activation blocks of the projection at hand
  uint4 *gated_blocks = nullptr;            // ... of the down projection, where gate+up writes them
  float *w_final = nullptr;
  double *inv_freq = nullptr;

  // sequence state
  void *kc = nullptr, *vc = nullptr;        // [L][max_batch][nkv][max_seq][D]
  size_t kv_layer_elems = 0;
  int *tokens = nullptr;                    // [max_batch][max_seq]
  DevState *dstate = nullptr;
  int *h_error = nullptr;                   // pinned host copy of the device error word, refreshed by calls that synchronise
  dmtd_status device_failure = DMTD_OK;     // sticky until dmtd_reset: a device-side check or wait reported an error
  dmtd_state h{};                           // host mirror
  bool prefilled = false;
  int B = 0;

  // workspace
  int ws_rows = 0, part_rows = 0;           // rows of a chunk; ... of a chunk whose attention runs over key slices
  int lda = 0, ldqkv = 0, ldgu = 0, ldl = 0, CH = 0, nsplit_max = 0;
  float *x_lo = nullptr, *x_up = nullptr, *act = nullptr, *qkv = nullptr, *gu = nullptr,
        *logits = nullptr, *part_o = nullptr, *part_ml = nullptr;
  float2 *rope_tab = nullptr;
  const float2 *rope_rows = nullptr;       // rows of rope_tab of the positions the next layers work on
  float *h_pend = nullptr;                  // [max_batch][pend_cap][hidden]: h_enc of positions the thinking layers have not seen
  float *h_base = nullptr;                  // [ws_rows][hidden]: h_emb / h_enc of a chunk of rows (literal sum, masked forward)
  int pend_cap = 0;

  // options
  bool use_graph = true, literal_sum = false, use_tc_attention = true;
  int pass_option = -1;                     // the option "fused_pass", once it is set
  bool fuse_qk_rope = true;                 // QK-norm, RoPE and the KV append inside the tensor-core attention kernel
  float temperature = 0.f;                  // > 0: tokens are drawn from softmax(logits / temperature); 0: greedy
  uint64_t sample_seed = 0;

  // fused pass kernel: one persistent launch per pass
  bool fused_ok = false;
  PassLayer *pass_layers = nullptr;         // device [n_layers]
  float *f_part_o = nullptr, *f_part_ml = nullptr, *amax_val = nullptr;
  int *amax_idx = nullptr;
  unsigned int *grid_bar = nullptr;
  float *pick_val = nullptr;                // per-step greedy pick: best of every vocabulary slice, [max_batch][ARGMAX_SLICES]
  int *pick_idx = nullptr;
  unsigned int *pick_arrived = nullptr;
  long long *pass_timing = nullptr;         // profiling builds only

  bool small_ok = false;                    // the model fits small_pass_kernel

  // captured passes: kind 1 = full (of tau pending rows), 2 = upper-only (any tau; 0 here)
  struct PassGraph {
    int kind, B, tau, forms, nodes;
    cudaGraphExec_t exec;
    cudaGraph_t graph;                      // (owns the node below)
    cudaGraphNode_t pick;                   // argmax_kernel: the pass's last launch
    int64_t used;
  };
  std::vector<PassGraph> graphs;            // at most kMaxGraphs
  int64_t graph_uses = 0;
  bool capturing = false;

  int64_t launches = 0;
};

namespace {

dmtd_status fail(dmtd_ctx *c, dmtd_status st, const char *fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (c) c->err = buf; else g_create_error = buf;
  return st;
}

#define CUDA_TRY(c, expr)                                                                   \
  do {                                                                                      \
    cudaError_t e_ = (expr);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return fail((c), DMTD_ERR_CUDA, "%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e_), \
                  __FILE__, __LINE__);                                                      \
  } while (0)

template <typename T>
dmtd_status dev_alloc(dmtd_ctx *c, T **p, size_t n) {
  void *q = nullptr;
  CUDA_TRY(c, cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(T)));
  c->allocs.push_back(q);
  c->mem[c->mem_kind] += std::max<size_t>(n, 1) * sizeof(T);
  *p = static_cast<T *>(q);
  return DMTD_OK;
}

dmtd_status check_launch(dmtd_ctx *c, const char *what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(c, DMTD_ERR_CUDA, "launch of %s failed: %s", what, cudaGetErrorString(e));
  c->launches += 1;
  return DMTD_OK;
}
#define LAUNCH_OK(c, what)                          \
  do {                                              \
    dmtd_status s_ = check_launch((c), (what));     \
    if (s_ != DMTD_OK) return s_;                   \
  } while (0)
#define TRY(expr)                                   \
  do {                                              \
    dmtd_status s_ = (expr);                        \
    if (s_ != DMTD_OK) return s_;                   \
  } while (0)

bool is_bf16(const dmtd_ctx *c) { return c->s.weight_dtype == DMTD_BF16; }
size_t wbytes(const dmtd_ctx *c) { return is_bf16(c) ? 2 : 4; }

// Largest divisor of the atom count per row that keeps a k-slab at or below `cap` atoms.
int choose_aps(int K, int cap) {
  int atoms = K / 32, best = 1;
  for (int d = 1; d <= std::min(atoms, cap); ++d)
    if (atoms % d == 0) best = d;
  return best;
}

// Build one packed matrix from up to three row blocks (e.g. q, k, v) of equal K.
dmtd_status pack_matrix(dmtd_ctx *c, PackedMat *out, int K, const void *const *srcs, const int *Ns, int n_src,
                        int aps_cap) {
  int N = 0;
  for (int i = 0; i < n_src; ++i) N += Ns[i];
  PackedMat m{};
  m.N = N; m.K = K; m.n_tiles = (N + 15) / 16;
  if (is_bf16(c)) {
    m.aps = choose_aps(K, aps_cap);
    m.n_slabs = K / 32 / m.aps;
    uint4 *dst = nullptr;
    c->mem_kind = 0;
    TRY(dev_alloc(c, &dst, (size_t)packed_atoms(m) * 64));
    c->mem_kind = 3;
    int tile0 = 0;
    for (int i = 0; i < n_src; ++i) {
      if (tile0 * 16 != (int)std::accumulate(Ns, Ns + i, 0))
        return fail(c, DMTD_ERR_SHAPE, "row blocks of a fused matrix must be multiples of 16 rows");
      long long chunks = (long long)m.n_slabs * ((Ns[i] + 15) / 16) * m.aps * 64;
      int grid = (int)std::min<long long>((chunks + 255) / 256, 65535);
      pack_bf16_kernel<<<grid, 256, 0, c->stream>>>(static_cast<const __nv_bfloat16 *>(srcs[i]), Ns[i], K, dst,
                                                    tile0, m.n_tiles, m.aps, m.n_slabs);
      LAUNCH_OK(c, "pack_bf16_kernel");
      tile0 += (Ns[i] + 15) / 16;
    }
    m.w = dst;
  } else {
    float *dst = nullptr;
    c->mem_kind = 0;
    TRY(dev_alloc(c, &dst, (size_t)N * K));
    c->mem_kind = 3;
    size_t off = 0;
    for (int i = 0; i < n_src; ++i) {
      CUDA_TRY(c, cudaMemcpyAsync(dst + off, srcs[i], (size_t)Ns[i] * K * 4, cudaMemcpyDeviceToDevice, c->stream));
      off += (size_t)Ns[i] * K;
    }
    m.wf = dst;
  }
  *out = m;
  return DMTD_OK;
}

dmtd_status vec_to_float(dmtd_ctx *c, float **out, const void *src, int n) {
  TRY(dev_alloc(c, out, (size_t)n));
  if (is_bf16(c))
    to_float_kernel<__nv_bfloat16><<<(n + 255) / 256, 256, 0, c->stream>>>(static_cast<const __nv_bfloat16 *>(src), *out, n);
  else
    to_float_kernel<float><<<(n + 255) / 256, 256, 0, c->stream>>>(static_cast<const float *>(src), *out, n);
  LAUNCH_OK(c, "to_float_kernel");
  return DMTD_OK;
}

// Second copy of a (fused) matrix in the block order of the tcgen05 GEMM; in_turn: the rows of the sources (of equal
// size) one after the other instead of source after source.  K is filled up with zeros to whole k blocks, the rows to
// `rows` of them.
dmtd_status pack_umma(dmtd_ctx *c, UmmaMat *out, int K, const void *const *srcs, const int *Ns, int n_src, bool in_turn = false, int rows = 0) {
  int N = 0;
  for (int i = 0; i < n_src; ++i) N += Ns[i];
  UmmaMat m{};
  m.N = N = std::max(N, rows); m.K = K; m.n_tiles = (N + 2 * TG_ROWS - 1) / (2 * TG_ROWS) * 2; m.n_kb = (K + TG_KB - 1) / TG_KB;
  uint4 *dst = nullptr;
  size_t units = (size_t)m.n_tiles * m.n_kb * (TG_WBLOCK / 16);
  c->mem_kind = 1;
  TRY(dev_alloc(c, &dst, units));
  c->mem_kind = 3;
  CUDA_TRY(c, cudaMemsetAsync(dst, 0, units * 16, c->stream));
  int row0 = 0;
  for (int i = 0; i < n_src; ++i) {
    long long total = (long long)Ns[i] * (K / 8);
    int grid = (int)std::min<long long>((total + 255) / 256, 65535);
    pack_umma_kernel<<<grid, 256, 0, c->stream>>>(static_cast<const __nv_bfloat16 *>(srcs[i]), Ns[i], K, row0, in_turn ? n_src : 1,
                                                  m.n_kb, dst);
    LAUNCH_OK(c, "pack_umma_kernel");
    row0 += in_turn ? 1 : Ns[i];
  }
  m.w = dst;
  *out = m;
  return DMTD_OK;
}

// ---------------------------------------------------------------------------- launches

// Launch with programmatic stream serialisation: the kernel's blocks may become resident while the
// kernel before it in the stream is still running; it calls griddepcontrol.wait before it touches
// anything that kernel (or one before it) writes.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The same for a grid of clusters of `ranks` blocks.
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int ranks, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[2]{};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ranks; attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

int gemv_smem_bytes(const PackedMat &W, int NT) {
  int KS = W.aps * 32;
  int row_bytes = ((KS * 2) % 128 == 64) ? KS * 2 : KS * 2 + 64;
  return 8 * NT * row_bytes;
}

template <int NT>
dmtd_status launch_gemv_nt(dmtd_ctx *c, const PackedMat &W, const float *act, int lda, int M, float *out, int ldo) {
  int smem = gemv_smem_bytes(W, NT);
  CUDA_TRY(c, launch_pdl(gemv_bf16_kernel<NT>, dim3(2 * c->n_sms), dim3(GEMV_THREADS), (size_t)(smem), c->stream,
                          W, act, lda, M, out, ldo));
  LAUNCH_OK(c, "gemv_bf16_kernel");
  return DMTD_OK;
}

using GemmTcKernel = void (*)(GemmTcParams);
GemmTcKernel gemm_tc05_for(bool split, int whole) {
  if (split) return whole == TG_STORE ? gemm_tc05_kernel<true, TG_STORE> : gemm_tc05_kernel<true, TG_ADD>;
  return whole == TG_STORE ? gemm_tc05_kernel<false, TG_STORE> : whole == TG_SWIGLU ? gemm_tc05_kernel<false, TG_SWIGLU>
                                                                                   : gemm_tc05_kernel<false, TG_ADD>;
}

// Where the activation blocks of a projection on the tcgen05 tensor cores come from.
struct GemmInput {
  enum Kind { ROWS, NORM, SWIGLU, SLICES, READY } kind = ROWS;
  const float *act = nullptr;               // ROWS, NORM: [rows][lda]; SWIGLU: gate and up values in turn
  int lda = 0;
  const float *norm_w = nullptr;            // NORM: RMSNorm(row) * norm_w
  int seg_rows = 0, seg_stride = 0;         // NORM: the rows come in segments (RowSegments)
  int nsplit = 0;                           // SLICES: the attention's key slices, merged on the way
  int kb0 = 0;                              // SWIGLU: the first k block that is not written yet
  uint4 *blocks = nullptr;                  // READY (and SWIGLU, for the rest): the blocks' own buffer
  GateUpParts gu{};                         // SWIGLU: the parts of gate+up's cut tiles
  // of the GEMM: outputs that do not depend on the order in which parts of tiles are added (see repeats)
  enum Sums { ANY_ORDER, TWO_PARTS, UNCUT } sums = ANY_ORDER;
  size_t part_stride = 0;                   // gate+up: its cut tiles' parts are stored this far apart
};

ActTiles projection_tiles(const dmtd_ctx *c, const UmmaMat &W, int M, bool uncut) {
  return uncut ? act_tiles_uncut(M, W.n_kb, W.n_tiles / 2, c->n_sms / 2) : act_tiles_for(M, W.n_kb);
}

// out[m][n] (+)= sum_k W[n][k] act[m][k]: the kernel that writes the activation blocks, then the GEMM.  After a norm the
// outputs are new: what the GEMM adds into is cleared beside the norm, the rest is stored (`whole`).  With `gated` the
// matrix is gate+up and the gate's result goes to the down projection's activation blocks there; `out` takes the
// values of the weight rows behind the tiles dealt out whole, [M][ldo] from row tg_whole_pairs * 256 on.
dmtd_status launch_gemm_tc05(dmtd_ctx *c, const UmmaMat &W, const GemmInput &in, int M, float *out, int ldo, uint4 *gated = nullptr,
                             const ActTiles &gated_tiles = ActTiles{}) {
  GemmTcParams P{};
  P.W = W;
  P.rows = M;
  P.T = projection_tiles(c, W, M, in.sums == GemmInput::UNCUT);
  P.out = out; P.ldo = ldo;
  P.error = &c->dstate->error; P.wait_limit = kDeviceWaitLimitTicks;
  uint4 *blocks = in.blocks ? in.blocks : c->act_blocks;
  P.act_blocks = blocks;
  const int n_pairs = c->n_sms / 2;
  // Tiles dealt out whole: gate+up where it gates, and matrices of two rounds of tiles and more (the head).  With one round (gate+up
  // of a decode pass) the part of a tile in front of it costs an epilogue more than the clearing it saves.  A pass of one
  // layer and a head of 1 / 2 / 4 / 6 rounds, stored against added: 32 rows 110.6 / 125.2 / 156.0 / 186.8 us against 108.9 / 125.3 /
  // 158.8 / 190.5, 8 rows 96.0 / 109.7 / 139.1 / 168.3 against 95.8 / 110.3 / 140.1 / 169.7, 96 rows 153.2 / 170.3 / 206.2 / 239.7
  // against 155.6 / 174.7 / 213.8 / 255.1.
  const int whole = in.kind != GemmInput::NORM ? TG_ADD : gated ? TG_SWIGLU : W.n_tiles / 2 >= 2 * n_pairs ? TG_STORE : TG_ADD;
  P.rt_whole = tg_whole_pairs(W, whole, n_pairs);
  P.whole_units = P.rt_whole / n_pairs * P.T.n_ctiles * W.n_kb;
  const int tiles = (W.n_tiles / 2 - P.rt_whole) * P.T.n_ctiles;
  P.line = in.sums == GemmInput::TWO_PARTS ? tg_line_two(tiles, W.n_kb, n_pairs)
                                           : tg_line(tiles, W.n_kb, in.sums == GemmInput::UNCUT ? tiles : n_pairs);
  P.part_stride = in.part_stride;
  const int n_whole = P.rt_whole * 2 * TG_ROWS;                                   // weight rows dealt out whole
  if (gated) { P.gated = gated; P.gated_T = gated_tiles; P.out_n0 = n_whole; }
  // shares of the k blocks per group of rows: one wave of blocks (two per SM; every block reads its rows for their sums).
  // 1 / 2 / 4 per SM: batch 32 21.8 / 21.65 / 22.4 ms for 4 cycles, batch 3 23.11 / 23.06 / 23.05 for 6
  const int n_groups = (M + NAB_ROWS - 1) / NAB_ROWS, ky = std::max(1, std::min(W.n_kb, 2 * c->n_sms / n_groups));
  if (in.kind == GemmInput::SLICES) {
    CUDA_TRY(c, launch_pdl(merge_act_blocks_kernel, dim3(n_groups, ky), dim3(256), 0, c->stream, c->part_o, c->part_ml,
                           in.nsplit, c->s.n_q_heads, c->s.head_dim, M, P.T, blocks));
    LAUNCH_OK(c, "merge_act_blocks_kernel");
  } else if (in.kind == GemmInput::NORM) {
    const int n_rest = in.part_stride ? 0 : std::max(0, W.N - n_whole);
    ZeroArea zero{gated ? out : out + n_whole, M, n_rest, (size_t)ldo};
    if (n_whole == 0 && n_rest && ldo - W.N < 16) zero.cols = ldo;                                          // whole rows, padding included
    const size_t zero_n = (size_t)zero.rows * zero.cols;
    const int n_zero = (int)std::min<size_t>((zero_n + 4095) / 4096, 2 * c->n_sms);
    CUDA_TRY(c, launch_pdl(norm_act_blocks_kernel, dim3(n_groups + (n_zero + ky - 1) / ky, ky), dim3(256), 0, c->stream,
                           in.act, in.lda, RowSegments{in.seg_rows, in.seg_stride}, in.norm_w, c->s.rms_eps, M, W.K, P.T,
                           blocks, n_groups, zero));
    LAUNCH_OK(c, "norm_act_blocks_kernel");
  } else if (in.kind != GemmInput::READY && in.kb0 < W.n_kb) {
    const int tiles = (W.n_kb - in.kb0) * ((M + AB_ROWS - 1) / AB_ROWS);
    CUDA_TRY(c, launch_pdl(in.gu.stride ? act_blocks_kernel<true, true> : in.kind == GemmInput::SWIGLU ? act_blocks_kernel<true> : act_blocks_kernel<false>,
                           dim3(std::min((tiles + AB_THREADS / 32 - 1) / (AB_THREADS / 32), 8 * c->n_sms)), dim3(AB_THREADS), 0, c->stream, in.act, in.lda, M, P.T, blocks, in.kb0, in.gu));
    LAUNCH_OK(c, "act_blocks_kernel");
  }
  // as many stages as shared memory holds, two accumulators where tensor memory does.  (Half of both for decode launches,
  // so that the next projection's blocks become resident beside this one's and fetch their first weights, was no
  // faster at 8-32 rows and slower at 96: fewer stages are in flight while a launch streams.)
  const int n_cols = P.T.split ? 2 * P.T.tile_rows : P.T.tile_rows, stage_bytes = tg_stage_units(P.T.split) * (TG_WBLOCK + P.T.tile_rows * 128);
  P.stages = std::max(2, std::min(TG_MAX_STAGES, (TG_MAX_SMEM - TG_TAIL_BYTES) / stage_bytes));
  if (c->gemm_stages >= 2) P.stages = std::min(P.stages, c->gemm_stages);
  int cols = 32;
  while (cols < n_cols) cols <<= 1;
  P.n_acc = 2 * cols <= 512 ? 2 : 1;
  P.tmem_cols = P.n_acc * cols;
  CUDA_TRY(c, launch_pdl(gemm_tc05_for(P.T.split != 0, whole), dim3(2 * n_pairs), dim3(TG_THREADS),
                         (size_t)std::max(TG_MIN_SMEM, P.stages * stage_bytes + TG_TAIL_BYTES), c->stream, P));
  LAUNCH_OK(c, "gemm_tc05_kernel");
  return DMTD_OK;
}

GemmInput rows_input(const float *act, int lda) {
  GemmInput in;
  in.act = act; in.lda = lda;
  return in;
}
GemmInput norm_input(const float *x, int ldx, const float *w) {
  GemmInput in = rows_input(x, ldx);
  in.kind = GemmInput::NORM; in.norm_w = w;
  return in;
}

// out[m][n] += sum_k W[n][k] act[m][k]
dmtd_status launch_gemv(dmtd_ctx *c, const PackedMat &W, const UmmaMat &U, const float *act, int lda, int M, float *out,
                        int ldo) {
  // the tcgen05 GEMM at every row count: the mma.sync kernel, whose warps load their weights through registers,
  // streams the tied head of the Qwen3-4B shape (778 MB, 1 - 4 rows) at 3.6 TB/s, the tcgen05 kernel at 5.9, and a
  // layer's projections at 3 rows in 82 us against 58 (kernel times)
  if (U.w && c->use_umma) return launch_gemm_tc05(c, U, rows_input(act, lda), M, out, ldo);
  if (W.wf) {
    auto launch = [&](auto kernel, int bm, int bn, int threads, int smem) {
      return launch_pdl(kernel, dim3((W.N + bn - 1) / bn, (M + bm - 1) / bm), dim3(threads), (size_t)smem, c->stream, W, act, lda, M, out, ldo);
    };
    // Small tiles up to 64 rows, large ones where they give every SM three blocks.  Layers of fp32 models, us, 16 / 32 / 64 wide
    // tiles: hidden 256, 64 rows 50 / 56 / 110, 192 rows 67 / 62 / 112, 1000 rows 213 / 137 / 156; hidden 1024, 64 rows 132 / 158 /
    // 385, 96 rows 208 / 186 / 375, 512 rows 645 / 543 / 555, 1000 rows 1249 / 1022 / 915.
    const long long large = (long long)((W.N + 63) / 64) * ((M + 63) / 64);
    if (M <= 64) CUDA_TRY(c, launch(gemm_f32_kernel<16, 16, 8>, 16, 16, 128, gemm_f32_smem<16, 16, 8>()));
    else if (large < 3ll * c->n_sms) CUDA_TRY(c, launch(gemm_f32_kernel<32, 32, 4>, 32, 32, 256, gemm_f32_smem<32, 32, 4>()));
    else CUDA_TRY(c, launch(gemm_f32_kernel<64, 64, 1>, 64, 64, 256, gemm_f32_smem<64, 64, 1>()));
    LAUNCH_OK(c, "gemm_f32_kernel");
    return DMTD_OK;
  }
  if (M <= 4) return launch_gemv_nt<1>(c, W, act, lda, M, out, ldo);
  if (M <= 8) return launch_gemv_nt<2>(c, W, act, lda, M, out, ldo);
  return launch_gemv_nt<4>(c, W, act, lda, M, out, ldo);
}

// attn_partial_kernel compiled for the fewest query rows that hold n_rows, for slices of CH keys.
template <typename KVT>
struct AttnPartialKernel {
  void (*kernel)(const float *, int, const KVT *, const KVT *, int, int, int, int, int, int, const int *, int, float *, float *, int, AttnFuse);
  int threads;
  size_t smem;
};
template <int D, typename KVT, bool FUSED, int T>
AttnPartialKernel<KVT> attn_partial_for(int n_rows, int R) {
  const int nq = n_rows <= 4 ? 4 : n_rows <= 8 ? 8 : 16, warps = attn_warps(T);
  return {nq == 4   ? attn_partial_kernel<D, KVT, 4, FUSED, T>
          : nq == 8 ? attn_partial_kernel<D, KVT, 8, FUSED, T>
                    : attn_partial_kernel<D, KVT, 16, FUSED, T>,
          warps * 32, (size_t)warps * nq * D * sizeof(float) + (FUSED ? 2 * (size_t)R * D * sizeof(KVT) : 0)};
}
// The form for slices of 64 keys (T = 1) takes more of an SM than the other and gains by latency alone: only for launches
// whose blocks are resident at once, one to an SM with 16 query rows, two with 8, four with 4.  head_dim 64, fp16 cache,
// against T = 4: 16 rows, 128 blocks 22 us (T = 4 31), 362 blocks 42 (31), 16384 blocks 1070 (670); 8 rows, 256 blocks 21
// (25), 512 blocks 30 (25); 4 rows, 362 blocks 15 (17), 1024 blocks 29 (25).
template <int D, typename KVT, bool FUSED>
AttnPartialKernel<KVT> attn_partial_for(int n_rows, int R, int CH, long long n_blocks, int n_sms) {
  const int nq = n_rows <= 4 ? 4 : n_rows <= 8 ? 8 : 16;
  if constexpr (D == 64)                    // head_dim 128: only with "tc_attention" off
    if (CH <= 64 && n_blocks * nq <= 16ll * n_sms) return attn_partial_for<D, KVT, FUSED, 1>(n_rows, R);
  return attn_partial_for<D, KVT, FUSED, 4>(n_rows, R);
}

// Does the attention of R new rows per sequence run on attn_decode_kernel?
bool tc_decode_attention(const dmtd_ctx *c) { return c->use_tc_attention && c->s.head_dim == PK_D && c->s.kv_dtype != DMTD_F32; }

// Clusters of 2, 4 and 8 attention blocks that the device holds at once (a cluster lies in one GPC).
int attn_cluster_room(int device, int ranks) {
  constexpr int kDevices = 64;
  static std::atomic<int> room[kDevices][4];
  const int i = ranks == 2 ? 1 : ranks == 4 ? 2 : 3;
  if (device < 0 || device >= kDevices) return 0;
  int n = room[device][i].load(std::memory_order_relaxed);
  if (n == 0) {
    const auto kernel = attn_decode_kernel<OpBf16, true, true>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ranks); cfg.blockDim = dim3(AD_THREADS); cfg.dynamicSmemBytes = AD_SMEM;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = ranks; attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AD_SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    room[device][i].store(n > 0 ? n : -1, std::memory_order_relaxed);
  }
  return std::max(0, n);
}
// Blocks of a cluster to an item (sequence, kv head, row block) of `units` 64-key units where the attention runs as one launch of
// clusters; 0: equal shares for one wave of blocks, and a launch behind them that merges.  As many blocks to an item as are
// resident at once; clusters of 8 up to 3/2 blocks per SM (with 32 of them a layer of 16 sequences and 2 kv heads took 5 us
// longer than without clusters: eight free places in one GPC come late).  Attention alone, 32 query and 8 kv heads, equal
// shares and merge against clusters, us: 1 x 64 / 1000 / 4000 / 16000 keys 4.9 / 8.3 / 15.0 / 24.0 against 3.9 / 5.2 / 8.7 / 24.0, 8 x 1000 14.3
// against 10.4, 32 x 1000 28.9 against 24.2, 8 x 16387 (3 rows) 87.9 against 81.3; 4 layers and the head, 3 / 16 / 32 sequences
// 355 / 373 / 408 against 345 / 358 / 396.
// More items than resident blocks: one block each, or equal shares.  Alone, ones up to three waves (two with few keys), but for a few
// items more than whole waves, which wait for another one; 128 / 300 / 1000 / 4000 keys, ones' time over equal shares': 320 items 0.80
// / 1.07 / 1.02 / 1.00, 512 0.95 / 0.95 / 0.97 / 0.98, 640 1.10 / 1.02 / 1.00 / 0.98, 832 1.02 / 1.01 / 0.99 / 0.98, 1040 1.09 / 1.02 / 1.00 / 1.01, 2000 1.16
// / 1.04 / 1.01.  In a layer, whose next launch waits for the last wave, only for short items in a well filled second wave; the
// whole layer, one row: 320 items 1.03 / 1.05 / 1.11 / 1.18, 384 1.03 / 1.01 / 1.04 / 1.09, 512 0.99 / 1.00 / 1.02 /
// 0.99 (three rows 0.98 / 0.98 / 1.01 / 1.01), 592 1.00, 640 1.05 / 1.05 / 1.07 / 1.08, 832 1.01 / 1.02 / 1.03 / 1.00, 1280 1.06 / 1.05 / 1.07 / 1.03.
// Few long items: the clusters leave places free, and where a block's piece is longer than an equal share by more than the merge's
// launch costs, shares are faster.  Layer, 8 kv heads, one row, clusters' time over equal shares', 8000 / 16000 / 32768 keys: 8 items (8 blocks each)
// 1.03 / 1.09 / 1.19, 16 0.97 / 1.00 / 1.05, 24 0.96 / 0.98 / 0.99, 32 (4 each) 0.99 / 1.07 / 1.12, 64 0.98 / 0.99; three rows 1.04 / 1.12 / 1.23, 0.95 / 1.00 /
// 1.08, 0.94 / 0.96 / 0.98, 0.99 / 1.08 / 1.18, 0.96 / 0.98: the lines cross at about 18 units of 64 keys more.  Alone, with caches read for the first
// time, 8 items 0.82 / 1.01 / 1.22 (65536 keys 1.46), 16 0.84 / 0.99 / 1.05, 32 0.94 / 1.07 / 1.05, 2 items (2 kv heads) 0.78 / 1.12 / 1.61: at about 27.
// `longest`: the units that the lengths at hand give, where `units` stands for a captured pass's longest context.
int attn_cluster_ranks(int device, int n_sms, int items, int units, int longest, bool in_layer) {
  const int slots = 2 * n_sms, over = items % slots;
  if (items > slots) {
    if (in_layer) return 2 * items > 3 * slots && items <= 2 * slots && units <= 8 ? 1 : 0;
    return (over > 0 && over < slots / 4) || items > (units > 4 ? 3 : 2) * slots ? 0 : 1;
  }
  int ranks = 1;
  while (ranks < AD_MAX_CLUSTER && ranks < units && items <= attn_cluster_room(device, 2 * ranks) && (ranks < 4 || 16 * items <= 3 * n_sms)) ranks *= 2;
  const long long free_places = slots - (long long)items * ranks;                  // longest / ranks - longest * items / slots > 18 or 27
  return longest * free_places > (in_layer ? 18ll : 27ll) * ranks * slots ? 0 : ranks;
}
// ... for R new rows per sequence in a layer, up to position pos_end.  A captured pass is replayed at other positions: its pieces are
// those of the context's last one, and the choice between the forms is part of what it is kept under (attention_forms).
int attention_ranks(const dmtd_ctx *c, int B, int R, int pos_end, bool captured) {
  if (!tc_decode_attention(c) || !c->fuse_qk_rope || R > AD_MAX_NEW || !c->use_umma || !c->umma_ok) return 0;
  const int RB = std::max(1, ATTN_QR / (c->s.n_q_heads / c->s.n_kv_heads)), n_rb = (R + RB - 1) / RB;
  return attn_cluster_ranks(c->device, c->n_sms, B * c->s.n_kv_heads * n_rb, ((captured ? c->max_seq : pos_end) + AD_UNIT - 1) / AD_UNIT,
                            (pos_end + AD_UNIT - 1) / AD_UNIT, true);
}

// Its blocks and slots: as many slots as the partial results' buffer holds (and, up to four rows at a time, the merge
// inside the O projection's activation-block kernel).
AttnDecodePlan tc_attention_plan(const dmtd_ctx *c, int B, int R, int max_slots) {
  const dmtd_model_shape &s = c->s;
  const int RB = std::max(1, ATTN_QR / (s.n_q_heads / s.n_kv_heads)), n_rb = (R + RB - 1) / RB;
  return attn_decode_plan(c->n_sms, B * s.n_kv_heads * n_rb, (c->max_seq + AD_UNIT - 1) / AD_UNIT, max_slots);
}

// Large chunks give the same bits every time, as no sum depends on the order in which blocks finish: QKV's tiles are in at most
// two parts (onto zeroed outputs), O's and the down projection's are not cut, and the parts of the few row tiles of gate+up
// that are cut keep to themselves until the gate sums them.  Where uncut tiles of more than 128 rows keep the block
// pairs busy (Qwen3-4B shape: from 897 rows, 0.84 to 0.87 of their columns in use).  Four layers on 1024 rows take 1355 us
// so and 1327 with every tile cut into equal parts, on 900 rows 1333 and 1279; the prefill of 32 x 1024 tokens 461.3 and
// 457.0 ms.  (Parts summed in order by the last block to arrive: 1497 us; three buffers for the residual rows, one to a
// part: 1430.)  Fewer rows, and decode passes, add their parts in any order.
bool repeats(const dmtd_ctx *c, int M) {
  if (!c->umma_ok || !c->use_umma || M <= TG_SPLIT_ROWS) return false;
  const LayerDev &lw = c->layers[0];
  const int n_pairs = c->n_sms / 2, n_ct = act_tiles_for(M, 1).n_ctiles;
  auto uncut = [&](const UmmaMat &W) {
    const int n_rt = W.n_tiles / 2;
    if (n_rt > n_pairs) return false;
    const int rows = act_tiles_uncut(M, W.n_kb, n_rt, n_pairs).tile_rows;
    return rows > TG_SPLIT_ROWS && rows <= TG_TILE_ROWS && n_rt * M >= 0.8 * n_pairs * rows;
  };
  const int gu_whole = tg_whole_pairs(lw.gu_u, TG_SWIGLU, n_pairs), gu_tiles = (lw.gu_u.n_tiles / 2 - gu_whole) * n_ct;
  const TgLine gu = tg_line(gu_tiles, lw.gu_u.n_kb, n_pairs);
  const size_t gu_parts = gu_tiles == 0 ? 0 : gu.q == 0 ? n_pairs : std::max(0, lw.gu_u.n_kb - 2) / gu.q + 2;
  const size_t n_rest = std::max(0, lw.gu_u.N - gu_whole * 2 * TG_ROWS);
  return lw.qkv_u.n_tiles / 2 * n_ct >= n_pairs && uncut(lw.o_u) && uncut(lw.down_u) &&
         (gu_tiles >= n_pairs || gu_parts * n_rest * M <= (size_t)c->ws_rows * c->ldgu);
}

template <int D, typename KVT>
dmtd_status launch_attention_t(dmtd_ctx *c, int layer, int B, int R, const int *pos0, int nsplit, bool merge, bool flash, int ranks) {
  const dmtd_model_shape &s = c->s;
  int M = B * R, heads = s.n_q_heads + 2 * s.n_kv_heads, G = s.n_q_heads / s.n_kv_heads;
  KVT *kc = static_cast<KVT *>(c->kc) + (size_t)layer * c->kv_layer_elems;
  KVT *vc = static_cast<KVT *>(c->vc) + (size_t)layer * c->kv_layer_elems;
  const LayerDev &lw = c->layers[layer];
  // a3 inside the attention kernel (decode-sized chunks): one launch less per layer
  const bool tiled = D == PK_D && c->use_tc_attention;                 // attn_decode_kernel or attn_f32_kernel
  const bool fused_a3 = (tiled ? !std::is_same<KVT, float>::value : D == 64) && c->fuse_qk_rope && !flash && R <= AD_MAX_NEW;
  if (!fused_a3) {
    CUDA_TRY(c, launch_pdl(qk_norm_rope_append_kernel<D, KVT>, dim3(M, (heads + 3) / 4), dim3(128), (size_t)(0), c->stream,
                             c->qkv, c->ldqkv, s.n_q_heads, s.n_kv_heads, R, lw.w_qn, lw.w_kn, s.rms_eps, c->rope_rows, pos0, kc, vc, c->max_seq));
    LAUNCH_OK(c, "qk_norm_rope_append_kernel");
  }
  if constexpr (D == PK_D && !std::is_same<KVT, float>::value) {
    if (flash) {
      // a chunk of many positions per sequence (the prefill): the causal kernel on the tcgen05 tensor cores
      using Op = typename std::conditional<std::is_same<KVT, __half>::value, OpF16, OpBf16>::type;
      const int QB = AP_M / G;
      AttnPrefillParams A{};
      A.qkv = c->qkv; A.kc = kc; A.vc = vc; A.ldq = c->ldqkv; A.max_seq = c->max_seq; A.nq = s.n_q_heads; A.nkv = s.n_kv_heads;
      A.R = R; A.pos0 = pos0; A.out = c->act; A.ld = c->lda;
      if (!merge) {                         // straight into the O projection's activation blocks
        A.blocks = c->act_blocks;
        A.T = projection_tiles(c, lw.o_u, M, repeats(c, M));
      }
      A.error = &c->dstate->error; A.wait_limit = kDeviceWaitLimitTicks;
      CUDA_TRY(c, launch_pdl(attn_prefill_kernel<Op>, dim3((R + QB - 1) / QB, s.n_kv_heads, B), dim3(AP_THREADS), (size_t)(AP_SMEM), c->stream,
                              A));
      LAUNCH_OK(c, "attn_prefill_kernel");
      return DMTD_OK;
    }
  }
  int RB = std::max(1, ATTN_QR / G), n_rb = (R + RB - 1) / RB;
  if (tiled) {
    // head_dim 128: the tensor-core kernel with a bf16 cache, the FMA kernel with an fp32 cache
    if constexpr (std::is_same<KVT, float>::value) {
      CUDA_TRY(c, launch_pdl(attn_f32_kernel, dim3(nsplit, s.n_kv_heads * n_rb, B), dim3(PK_THREADS), ATTN_F32_SMEM, c->stream,
                             c->qkv, c->ldqkv, kc, vc, c->max_seq, s.n_q_heads, s.n_kv_heads, R, RB, c->CH, pos0, 0, c->part_o,
                             c->part_ml, nsplit));
    } else {
      using Op = typename std::conditional<std::is_same<KVT, __half>::value, OpF16, OpBf16>::type;
      const AttnFuse fuse{lw.w_qn, lw.w_kn, c->rope_rows, s.rms_eps};
      if (ranks > 0) {
        CUDA_TRY(c, launch_cluster(attn_decode_kernel<Op, true, true>, dim3(B * s.n_kv_heads * n_rb * ranks), dim3(AD_THREADS), AD_SMEM, c->stream, ranks,
                                   c->qkv, c->ldqkv, kc, vc, c->max_seq, s.n_q_heads, s.n_kv_heads, B, R, RB, pos0, 0, nullptr, nullptr, 1, fuse,
                                   AttnBlocks{c->act_blocks, projection_tiles(c, lw.o_u, M, repeats(c, M))}));
        LAUNCH_OK(c, "attn_decode_kernel");
        return DMTD_OK;
      }
      const int n_blocks = tc_attention_plan(c, B, R, nsplit).n_blocks;
      CUDA_TRY(c, launch_pdl(fused_a3 ? attn_decode_kernel<Op, true> : attn_decode_kernel<Op, false>, dim3(n_blocks), dim3(AD_THREADS),
                             AD_SMEM, c->stream, c->qkv, c->ldqkv, kc, vc, c->max_seq, s.n_q_heads, s.n_kv_heads, B, R, RB, pos0, 0,
                             c->part_o, c->part_ml, nsplit, fuse, AttnBlocks{nullptr, ActTiles{}}));
    }
  } else {
    const AttnPartialKernel<KVT> ap =
        fused_a3 ? attn_partial_for<D, KVT, D == 64>(std::min(R, RB) * G, R, c->CH, (long long)nsplit * s.n_kv_heads * n_rb * B, c->n_sms)
                 : attn_partial_for<D, KVT, false>(std::min(R, RB) * G, R, c->CH, (long long)nsplit * s.n_kv_heads * n_rb * B, c->n_sms);
    CUDA_TRY(c, launch_pdl(ap.kernel, dim3(nsplit, s.n_kv_heads * n_rb, B), dim3(ap.threads), ap.smem, c->stream, c->qkv, c->ldqkv,
                           kc, vc, c->max_seq, s.n_q_heads, s.n_kv_heads, R, RB, c->CH, pos0, 0, c->part_o, c->part_ml, nsplit,
                           AttnFuse{lw.w_qn, lw.w_kn, c->rope_rows, s.rms_eps}));
  }
  LAUNCH_OK(c, "attn_partial_kernel");
  if (!merge) return DMTD_OK;               // the O projection's activation-block kernel merges the slices
  int n_rh = M * s.n_q_heads;
  CUDA_TRY(c, launch_pdl(attn_merge_kernel<D>, dim3((n_rh + 3) / 4), dim3(128), (size_t)(0), c->stream,
                          c->part_o, c->part_ml, nsplit, n_rh, s.n_q_heads, c->act, c->lda));
  LAUNCH_OK(c, "attn_merge_kernel");
  return DMTD_OK;
}

// Chunks of at least this many positions per sequence run the causal prefill kernel (16-bit cache, head_dim 128).
constexpr int kFlashMinRows = 16;
bool flash_attention_ok(const dmtd_ctx *c, int R) {
  const int G = c->s.n_q_heads / c->s.n_kv_heads;
  return c->use_tc_attention && c->s.head_dim == PK_D && c->s.kv_dtype != DMTD_F32 && R >= kFlashMinRows && AP_M % G == 0;
}

// Positions per sequence of one prefill chunk of B sequences.
int chunk_positions(const dmtd_ctx *c, int B) {
  return std::max(1, (flash_attention_ok(c, c->ws_rows / B) ? c->ws_rows : c->part_rows) / B);
}

dmtd_status launch_attention(dmtd_ctx *c, int layer, int B, int R, const int *pos0, int nsplit, bool merge = true,
                             bool flash = false, int ranks = 0) {
  const int kv = c->s.kv_dtype;
  if (c->s.head_dim == 128)
    return kv == DMTD_BF16 ? launch_attention_t<128, __nv_bfloat16>(c, layer, B, R, pos0, nsplit, merge, flash, ranks)
         : kv == DMTD_F16 ? launch_attention_t<128, __half>(c, layer, B, R, pos0, nsplit, merge, flash, ranks)
                          : launch_attention_t<128, float>(c, layer, B, R, pos0, nsplit, merge, flash, ranks);
  return kv == DMTD_BF16 ? launch_attention_t<64, __nv_bfloat16>(c, layer, B, R, pos0, nsplit, merge, flash, ranks)
       : kv == DMTD_F16 ? launch_attention_t<64, __half>(c, layer, B, R, pos0, nsplit, merge, flash, ranks)
                        : launch_attention_t<64, float>(c, layer, B, R, pos0, nsplit, merge, flash, ranks);
}

RopeTable rope_table(const dmtd_ctx *c) { return RopeTable{c->inv_freq, c->rope_tab, c->s.head_dim / 2}; }
int rope_blocks(const dmtd_ctx *c, int R) { return (R * (c->s.head_dim / 2) + 127) / 128; }

// rope_rows: the table's rows for the layers that follow; they start at row 0 unless the caller moves them
dmtd_status launch_rope_table(dmtd_ctx *c, const int *pos0, int R) {
  rope_table_kernel<<<rope_blocks(c, R), 128, 0, c->stream>>>(pos0, R, rope_table(c));
  LAUNCH_OK(c, "rope_table_kernel");
  c->rope_rows = c->rope_tab;
  return DMTD_OK;
}

// x = (accumulate: +=) the embeddings of positions *pos0 .. *pos0 + R - 1; not accumulate: their rotary table as well
dmtd_status launch_embed(dmtd_ctx *c, const int *pos0, int B, int R, float *x, bool accumulate) {
  embed_kernel<<<B * R + (accumulate ? 0 : rope_blocks(c, R)), 128, 0, c->stream>>>(c->embed, c->tokens, c->max_seq, pos0, R, B * R, x,
                                                                                    c->s.hidden, accumulate ? 1 : 0, c->dstate, rope_table(c));
  LAUNCH_OK(c, "embed_kernel");
  if (!accumulate) c->rope_rows = c->rope_tab;
  return DMTD_OK;
}

// Number of key slices of fixed length to launch: all of them while capturing a graph (the graph must stay
// valid as the context grows), else just enough for keys [0, pos_end).
int splits_for(const dmtd_ctx *c, int pos_end) {
  if (c->capturing) return c->nsplit_max;
  return std::max(1, std::min(c->nsplit_max, (pos_end + c->CH - 1) / c->CH));
}

// Key slices (slots of partial results per row and head) of a launch of B x R rows that ends at position pos_end.
int slices_for(const dmtd_ctx *c, int B, int R, int pos_end) {
  if (!tc_decode_attention(c)) return splits_for(c, pos_end);
  const long long room = (long long)c->part_rows * c->nsplit_max / ((long long)B * R);
  const int fused_merge = MAB_MAX_SLOTS / (NAB_ROWS * c->s.n_q_heads);
  return tc_attention_plan(c, B, R, (int)std::max(1ll, std::min<long long>(room, std::max(1, fused_merge)))).nsplit;
}

// fp32 weights, the few rows of a decode pass: every projection with the step in front of it.
bool f32_fused_rows(const dmtd_ctx *c, int M) {
  const dmtd_model_shape &s = c->s;
  return !is_bf16(c) && M <= F32_FUSE_ROWS && (long long)M * std::max({s.hidden, s.intermediate, s.n_q_heads * s.head_dim}) <= F32_FUSE_FLOATS;
}
template <int IN>
dmtd_status launch_gemv_f32_fused(dmtd_ctx *c, const PackedMat &W, const F32In &in, int M, float *out, int ldo, bool store) {
  CUDA_TRY(c, launch_pdl(gemv_f32_fused_kernel<IN>, dim3(std::min(4 * c->n_sms, (W.N + 7) / 8)), dim3(256),
                         (size_t)M * W.K * sizeof(float), c->stream, W, in, M, out, ldo, store ? 1 : 0));
  LAUNCH_OK(c, "gemv_f32_fused_kernel");
  return DMTD_OK;
}
// Every block of the O projection would merge all key slices again: more than 8192 values of them (of slices that hold keys; a
// captured pass keeps what held when it was captured) are merged by a kernel of their own.  Four layers of fp32 models, merged
// in front of the product against apart: 2048 values 82 us against 92, 4096 to 8192 within 5 % of each other, 32768 1.34 times
// as long, 327680 (4 rows of 16 heads x 128, 40 slices) 942 us against 360.
bool merge_apart(const dmtd_ctx *c, int M, int nsplit, int pos_end) {
  const int keys = tc_decode_attention(c) ? AD_UNIT : c->CH, live = std::min(nsplit, (pos_end + keys - 1) / keys);
  return (long long)M * c->s.n_q_heads * c->s.head_dim * live > 8192;
}
F32In f32_norm_input(const dmtd_ctx *c, const float *x, const float *w) { return F32In{x, c->s.hidden, w, c->s.rms_eps, nullptr, nullptr, 0, 0}; }

// One decoder layer (steps a2-a7) on x [B*R][hidden]; rows of sequence b sit at positions
// *pos0 .. *pos0+R-1.  pos_end = host's value of *pos0 + R.
dmtd_status run_layer(dmtd_ctx *c, int l, float *x, int B, int R, const int *pos0, int pos_end) {
  const dmtd_model_shape &s = c->s;
  const LayerDev &lw = c->layers[l];
  int M = B * R, H = s.hidden, I = s.intermediate;
  // the tcgen05 path normalises while it writes its activation blocks
  const bool tc = lw.qkv_u.w && c->use_umma;
  if (f32_fused_rows(c, M) && !flash_attention_ok(c, R)) {
    const int nsplit = slices_for(c, B, R, pos_end);
    TRY(launch_gemv_f32_fused<F32_NORM>(c, lw.qkv, f32_norm_input(c, x, lw.w_in), M, c->qkv, c->ldqkv, true));
    const bool apart = merge_apart(c, M, nsplit, pos_end);
    TRY(launch_attention(c, l, B, R, pos0, nsplit, apart));
    if (apart) TRY(launch_gemv(c, lw.o, lw.o_u, c->act, c->lda, M, x, H));
    else TRY(launch_gemv_f32_fused<F32_SLICES>(c, lw.o, F32In{nullptr, 0, nullptr, 0.f, c->part_o, c->part_ml, nsplit, s.n_q_heads}, M, x, H, false));
    TRY(launch_gemv_f32_fused<F32_NORM>(c, lw.gu, f32_norm_input(c, x, lw.w_post), M, c->gu, c->ldgu, true));
    return launch_gemv_f32_fused<F32_SWIGLU>(c, lw.down, F32In{c->gu, c->ldgu, nullptr, 0.f, nullptr, nullptr, 0, 0}, M, x, H, false);
  }
  const bool same_bits = tc && repeats(c, M);
  auto with_sums = [&](GemmInput in, GemmInput::Sums sums) {
    if (same_bits) in.sums = sums;
    return in;
  };
  if (tc) {
    TRY(launch_gemm_tc05(c, lw.qkv_u, with_sums(norm_input(x, H, lw.w_in), GemmInput::TWO_PARTS), M, c->qkv, c->ldqkv));
  } else {
    CUDA_TRY(c, launch_pdl(prep_norm_kernel, dim3(M, (c->ldqkv + PREP_ZERO_COLS - 1) / PREP_ZERO_COLS), dim3(256), (size_t)(0), c->stream,
                             x, H, lw.w_in, H, s.rms_eps, c->act, c->lda, c->qkv, c->ldqkv, c->ldqkv));
    LAUNCH_OK(c, "prep_norm_kernel");
    TRY(launch_gemv(c, lw.qkv, lw.qkv_u, c->act, c->lda, M, c->qkv, c->ldqkv));
  }
  const bool flash = flash_attention_ok(c, R);
  const int nsplit = flash ? 1 : slices_for(c, B, R, pos_end);
  // on the tcgen05 path the O projection's activation blocks come from the prefill attention itself, or from the
  // kernel that merges the key slices
  const bool fuse_merge = tc && (flash || NAB_ROWS * s.n_q_heads * nsplit <= MAB_MAX_SLOTS);
  const int ranks = tc && !flash ? attention_ranks(c, B, R, pos_end, c->capturing) : 0;       // > 0: the attention kernel merges, too
  TRY(launch_attention(c, l, B, R, pos0, nsplit, !fuse_merge && ranks == 0, flash, ranks));
  if (fuse_merge || ranks > 0) {
    GemmInput in;
    in.kind = flash || ranks > 0 ? GemmInput::READY : GemmInput::SLICES;
    in.nsplit = nsplit;
    TRY(launch_gemm_tc05(c, lw.o_u, with_sums(in, GemmInput::UNCUT), M, x, H));
  }
  else TRY(launch_gemv(c, lw.o, lw.o_u, c->act, c->lda, M, x, H));
  if (tc) {
    // more rows than a decode pass has: the GEMM gates its outputs and writes the down projection's activation blocks
    // itself, but for the few row tiles it has to share between blocks (their values go through `gu`)
    GemmInput down;
    down.kind = GemmInput::SWIGLU;
    down.act = c->gu;
    if (M > TG_SPLIT_ROWS) {
      const int n_whole = tg_whole_pairs(lw.gu_u, TG_SWIGLU, c->n_sms / 2) * 2 * TG_ROWS, n_rest = std::max(0, lw.gu_u.N - n_whole);
      down.lda = std::max(4, n_rest); down.kb0 = n_whole / 2 / TG_KB; down.blocks = c->gated_blocks;
      GemmInput gu = norm_input(x, H, lw.w_post);
      const ActTiles T = act_tiles_for(M, lw.gu_u.n_kb);
      const int tiles = (lw.gu_u.n_tiles / 2 - n_whole / (2 * TG_ROWS)) * T.n_ctiles;       // cut ones
      if (same_bits && tiles > 0 && tiles < c->n_sms / 2) {       // (a tile for every block pair: two parts at most, as QKV's)
        gu.part_stride = (size_t)M * down.lda;
        down.gu = GateUpParts{tg_line(tiles, T.n_kb, c->n_sms / 2), T.n_ctiles, T.n_kb, T.tile_rows, gu.part_stride};
      }
      TRY(launch_gemm_tc05(c, lw.gu_u, gu, M, c->gu, down.lda, c->gated_blocks, projection_tiles(c, lw.down_u, M, same_bits)));
    } else {
      down.lda = c->ldgu;
      TRY(launch_gemm_tc05(c, lw.gu_u, norm_input(x, H, lw.w_post), M, c->gu, c->ldgu));
    }
    TRY(launch_gemm_tc05(c, lw.down_u, with_sums(down, GemmInput::UNCUT), M, x, H));
  } else {
    CUDA_TRY(c, launch_pdl(prep_norm_kernel, dim3(M, (c->ldgu + PREP_ZERO_COLS - 1) / PREP_ZERO_COLS), dim3(256), (size_t)(0), c->stream,
                             x, H, lw.w_post, H, s.rms_eps, c->act, c->lda, c->gu, c->ldgu, c->ldgu));
    LAUNCH_OK(c, "prep_norm_kernel");
    TRY(launch_gemv(c, lw.gu, lw.gu_u, c->act, c->lda, M, c->gu, c->ldgu));
    CUDA_TRY(c, launch_pdl(prep_swiglu_kernel, dim3((I + 255) / 256, M), dim3(256), (size_t)(0), c->stream,
                            c->gu, c->ldgu, I, c->act, c->lda));
    LAUNCH_OK(c, "prep_swiglu_kernel");
    TRY(launch_gemv(c, lw.down, lw.down_u, c->act, c->lda, M, x, H));
  }
  return DMTD_OK;
}

SampleParams sample_params(const dmtd_ctx *c) {
  SampleParams sp{};
  sp.on = c->temperature > 0.f ? 1 : 0;
  sp.inv_temperature = sp.on ? 1.f / c->temperature : 1.f;
  sp.key0 = (unsigned)c->sample_seed; sp.key1 = (unsigned)(c->sample_seed >> 32);
  return sp;
}

// Step a9/a10/a0: final norm, tied LM head, greedy pick, token feedback, the schedule's counters.
dmtd_status run_head(dmtd_ctx *c, int B, bool write_token, int *out_argmax, float *out_logits, int kind, int P) {
  const dmtd_model_shape &s = c->s;
  if (f32_fused_rows(c, B)) {
    TRY(launch_gemv_f32_fused<F32_NORM>(c, c->embed, f32_norm_input(c, c->x_up, c->w_final), B, c->logits, c->ldl, true));
  } else if (c->embed_u.w && c->use_umma) {
    GemmInput in = norm_input(c->x_up, s.hidden, c->w_final);
    if (kind == 0) in.sums = GemmInput::TWO_PARTS;      // the first token's logits repeat as a large chunk's rows do
    TRY(launch_gemm_tc05(c, c->embed_u, in, B, c->logits, c->ldl));
  } else {
    CUDA_TRY(c, launch_pdl(prep_norm_kernel, dim3(B, (c->ldl + PREP_ZERO_COLS - 1) / PREP_ZERO_COLS), dim3(256), (size_t)(0), c->stream,
                             c->x_up, s.hidden, c->w_final, s.hidden, s.rms_eps, c->act, c->lda, c->logits, c->ldl, c->ldl));
    LAUNCH_OK(c, "prep_norm_kernel");
    TRY(launch_gemv(c, c->embed, c->embed_u, c->act, c->lda, B, c->logits, c->ldl));
  }
  if (out_logits)
    CUDA_TRY(c, cudaMemcpy2DAsync(out_logits, (size_t)s.vocab * 4, c->logits, (size_t)c->ldl * 4, (size_t)s.vocab * 4, B,
                                  cudaMemcpyDeviceToDevice, c->stream));
  CUDA_TRY(c, launch_pdl(argmax_kernel, dim3(B, ARGMAX_SLICES), dim3(256), (size_t)(0), c->stream,
                          c->logits, c->ldl, s.vocab, c->dstate, sample_params(c),
                          PickParams{c->pick_val, c->pick_idx, c->pick_arrived, write_token ? c->tokens : nullptr, c->max_seq, out_argmax, kind, P}));
  LAUNCH_OK(c, "argmax_kernel");
  return DMTD_OK;
}

// The LM head over many positions (the scoring pass): final norm and tied head of n_seg segments of seg_rows rows,
// segment i starting at row i * seg_stride of x; row m of them all to out + m * ldo.  One GEMM over all rows: a
// head launch per position streams the whole head again (Qwen3-4B shape, 2 x 187 of 2 x 250 positions: 187 x 0.25 ms
// of 59.1 ms a call; 13.4 ms now).
dmtd_status run_head_rows(dmtd_ctx *c, const float *x, int n_seg, int seg_rows, int seg_stride, float *out, int ldo) {
  const dmtd_model_shape &s = c->s;
  const int M = n_seg * seg_rows;
  if (c->embed_u.w && c->use_umma) {
    GemmInput in = norm_input(x, s.hidden, c->w_final);
    in.seg_rows = seg_rows; in.seg_stride = seg_stride;
    return launch_gemm_tc05(c, c->embed_u, in, M, out, ldo);
  }
  // segments of one row are rows of a longer stride
  int ldx = s.hidden;
  if (seg_rows == 1) { ldx *= seg_stride; seg_rows = n_seg; n_seg = 1; }
  for (int i = 0; i < n_seg; ++i) {
    CUDA_TRY(c, launch_pdl(prep_norm_kernel, dim3(seg_rows, (s.vocab + PREP_ZERO_COLS - 1) / PREP_ZERO_COLS), dim3(256), (size_t)(0), c->stream,
                             x + (size_t)i * seg_stride * s.hidden, ldx, c->w_final, s.hidden, s.rms_eps, c->act + (size_t)i * seg_rows * c->lda, c->lda,
                             out + (size_t)i * seg_rows * ldo, ldo, s.vocab));
    LAUNCH_OK(c, "prep_norm_kernel");
  }
  return launch_gemv(c, c->embed, c->embed_u, c->act, c->lda, M, out, ldo);
}

// Kernels that need more than 48 KiB of dynamic shared memory must be told so once per device
// (the attribute belongs to the device's copy of the kernel, not to the process): done at create,
// with the context's device current.
dmtd_status configure_kernels(dmtd_ctx *c) {
  const auto dyn = cudaFuncAttributeMaxDynamicSharedMemorySize;
  CUDA_TRY(c, cudaFuncSetAttribute(gemv_bf16_kernel<1>, dyn, 100 * 1024));
  CUDA_TRY(c, cudaFuncSetAttribute(gemv_bf16_kernel<2>, dyn, 100 * 1024));
  CUDA_TRY(c, cudaFuncSetAttribute(gemv_bf16_kernel<4>, dyn, 100 * 1024));
  for (int whole : {TG_ADD, TG_STORE, TG_SWIGLU})
    for (bool split : {false, true}) CUDA_TRY(c, cudaFuncSetAttribute(gemm_tc05_for(split, whole), dyn, TG_MAX_SMEM));
  if (!is_bf16(c)) {
    CUDA_TRY(c, cudaFuncSetAttribute(gemm_f32_kernel<16, 16, 8>, dyn, gemm_f32_smem<16, 16, 8>()));
    CUDA_TRY(c, cudaFuncSetAttribute(gemm_f32_kernel<64, 64, 1>, dyn, gemm_f32_smem<64, 64, 1>()));
    CUDA_TRY(c, cudaFuncSetAttribute(gemm_f32_kernel<32, 32, 4>, dyn, gemm_f32_smem<32, 32, 4>()));
    for (auto gemv : {gemv_f32_fused_kernel<F32_NORM>, gemv_f32_fused_kernel<F32_SWIGLU>, gemv_f32_fused_kernel<F32_SLICES>})
      CUDA_TRY(c, cudaFuncSetAttribute(gemv, dyn, (int)(F32_FUSE_FLOATS * sizeof(float))));
  }
  // (only the kernels of the context's cache type: the first touch of a kernel loads it)
  auto attention = [&](auto op) -> dmtd_status {
    using Op = decltype(op);
    CUDA_TRY(c, cudaFuncSetAttribute(attn_decode_kernel<Op>, dyn, AD_SMEM));
    CUDA_TRY(c, cudaFuncSetAttribute(attn_decode_kernel<Op, true>, dyn, AD_SMEM));
    CUDA_TRY(c, cudaFuncSetAttribute(attn_decode_kernel<Op, true, true>, dyn, AD_SMEM));
    CUDA_TRY(c, cudaFuncSetAttribute(attn_prefill_kernel<Op>, dyn, AP_SMEM));
    return DMTD_OK;
  };
  // 16 query rows, 128 dimensions or new rows take the key-group kernel past 48 KiB
  auto partial = [&](auto kv) -> dmtd_status {
    using KVT = decltype(kv);
    for (int rows : {8, 16}) {
      const AttnPartialKernel<KVT> forms[] = {attn_partial_for<128, KVT, false, 4>(rows, 1), attn_partial_for<64, KVT, false, 1>(rows, 1),
                                              attn_partial_for<64, KVT, false, 4>(rows, 1), attn_partial_for<64, KVT, true, 1>(rows, 1),
                                              attn_partial_for<64, KVT, true, 4>(rows, 1)};
      for (const AttnPartialKernel<KVT> &form : forms) CUDA_TRY(c, cudaFuncSetAttribute(form.kernel, dyn, 64 * 1024));
    }
    return DMTD_OK;
  };
  if (c->s.kv_dtype == DMTD_F32) {
    CUDA_TRY(c, cudaFuncSetAttribute(attn_f32_kernel, dyn, ATTN_F32_SMEM));
    return partial(0.f);
  }
  if (c->s.kv_dtype == DMTD_BF16) {
    TRY(attention(OpBf16{}));
    return partial(__nv_bfloat16{});
  }
  TRY(attention(OpF16{}));
  return partial(__half{});
}

// ---------------------------------------------------------------------------- fused pass

// Can the block-per-SM pass kernel stream this matrix?  Its k-slab must fit the staging area
// and one block's share must not reach over more than two slabs.
bool fused_matrix_ok(const PackedMat &m, int grid) {
  if (!m.w) return false;
  long long slab_atoms = (long long)m.n_tiles * m.aps, per_block = (packed_atoms(m) + grid - 1) / grid;
  // 32-bit stream arithmetic in the kernel: atoms * blocks must fit
  return m.aps * 32 <= PK_MAX_KS && per_block <= slab_atoms && packed_atoms(m) * (grid + 1) < (1ll << 31);
}

// Set up what the fused pass kernel needs; leaves fused_ok false when the model or the device
// does not fit it (the per-step kernels then run every pass).
dmtd_status setup_fused(dmtd_ctx *c) {
  const dmtd_model_shape &s = c->s;
  c->fused_ok = false;
  if (!is_bf16(c) || s.head_dim != PK_D || s.n_layers > PK_MAX_LAYERS) return DMTD_OK;
  if (s.n_q_heads / s.n_kv_heads > PK_MAX_GROUP || s.hidden % 8 || s.hidden > PK_XS_FLOATS) return DMTD_OK;
  int coop = 0;
  CUDA_TRY(c, cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, c->device));
  if (!coop) return DMTD_OK;
  if (cudaFuncSetAttribute(dmtd_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PK_SMEM_BYTES) != cudaSuccess) {
    cudaGetLastError();
    return DMTD_OK;
  }
  int per_sm = 0;
  CUDA_TRY(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, dmtd_pass_kernel, PK_THREADS, PK_SMEM_BYTES));
  if (per_sm < 1) return DMTD_OK;
  if (!fused_matrix_ok(c->embed, c->n_sms)) return DMTD_OK;
  for (const LayerDev &ld : c->layers) {
    if (!fused_matrix_ok(ld.qkv, c->n_sms) || !fused_matrix_ok(ld.o, c->n_sms) || !fused_matrix_ok(ld.gu, c->n_sms) ||
        !fused_matrix_ok(ld.down, c->n_sms))
      return DMTD_OK;
    if ((ld.o.aps * 32) % PK_D) return DMTD_OK;
    // the kernel works out every block's share of a matrix once per launch, from the first layer of the pass:
    // all layers must have the same four shapes (they do: one hidden and one intermediate size per model)
    const LayerDev &l0 = c->layers[0];
    auto same = [](const PackedMat &a, const PackedMat &b) {
      return a.N == b.N && a.K == b.K && a.n_tiles == b.n_tiles && a.aps == b.aps && a.n_slabs == b.n_slabs;
    };
    if (!same(ld.qkv, l0.qkv) || !same(ld.o, l0.o) || !same(ld.gu, l0.gu) || !same(ld.down, l0.down)) return DMTD_OK;
  }
  std::vector<PassLayer> h(s.n_layers);
  for (int l = 0; l < s.n_layers; ++l) {
    const LayerDev &ld = c->layers[l];
    h[l].qkv = ld.qkv; h[l].o = ld.o; h[l].gu = ld.gu; h[l].down = ld.down;
    h[l].w_in = ld.w_in; h[l].w_post = ld.w_post; h[l].w_qn = ld.w_qn; h[l].w_kn = ld.w_kn;
    const size_t kvb = s.kv_dtype == DMTD_F32 ? 4 : 2;
    h[l].kc = static_cast<unsigned char *>(c->kc) + (size_t)l * c->kv_layer_elems * kvb;
    h[l].vc = static_cast<unsigned char *>(c->vc) + (size_t)l * c->kv_layer_elems * kvb;
  }
  TRY(dev_alloc(c, &c->pass_layers, h.size()));
  CUDA_TRY(c, cudaMemcpyAsync(c->pass_layers, h.data(), h.size() * sizeof(PassLayer), cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  size_t slots = (size_t)PK_MAX_ROWS * s.n_q_heads * PK_NSPLIT_CAP;
  TRY(dev_alloc(c, &c->f_part_o, slots * PK_D));
  TRY(dev_alloc(c, &c->f_part_ml, slots * 2));
  TRY(dev_alloc(c, &c->amax_val, (size_t)PK_MAX_ROWS * c->n_sms));
  TRY(dev_alloc(c, &c->amax_idx, (size_t)PK_MAX_ROWS * c->n_sms));
  TRY(dev_alloc(c, &c->grid_bar, 1));
#ifdef DMTD_PASS_TIMING
  TRY(dev_alloc(c, &c->pass_timing, (size_t)2 * PK_TIMING_SLOTS));
#endif
  c->fused_ok = true;
  return DMTD_OK;
}

// The pass kernel runs where the option asks for it, and unasked where the per-step path lacks the block-ordered weights or the
// tensor-core attention (an fp32 cache): with both, a launch per step is faster at every size, since its rings fill at HBM's pace
// and the attention merges by cluster.  Cycles of 1 to 4 passes, the pass kernel's time over the per-step kernels': one sequence,
// context 64 to 3000, hidden 640 (7 MB a layer) 1.25 to 1.07, 1024 1.18 to 1.04, 2048 (100 MB) 1.09 to 1.01, 2560 (202 MB) 1.03
// to 1.05, over 36 layers 1.01 at 550 positions and 1.03 at 2500 (8 cycles 25.2 / 26.65 ms against 24.95 / 25.7); two sequences
// of 2560 1.05, three 1.08 to 1.11, four 1.11 to 1.18.  That is with captured passes.  Passes launched one by one (given tokens, "cuda_graph"
// off) take 5 to 10 % longer, and one sequence of a model with large layers is faster on the pass kernel; its time over theirs, one
// sequence: 10 MB a layer 1.06 to 1.11, 31 MB 1.01 to 1.08, 71 MB 1.00 to 1.04, 101 MB 0.95 to 1.00, 202 MB 0.96 to 0.99 (36 layers 0.945);
// two sequences of 202 MB 0.99 to 1.03, three 1.03 to 1.04.
bool fused_pass_ok(const dmtd_ctx *c, int kind, int R_lower, bool captured) {
  bool asked = c->pass_option > 0;
  if (c->pass_option < 0) {
    const LayerDev &l = c->layers[0];
    const bool per_step = c->umma_ok && c->use_umma && tc_decode_attention(c) && c->fuse_qk_rope;
    asked = !per_step || (!captured && c->B == 1 && packed_atoms(l.qkv) + packed_atoms(l.o) + packed_atoms(l.gu) + packed_atoms(l.down) >= (96 << 10));   // 1 KiB atoms
  }
  if (!c->fused_ok || !asked || c->literal_sum || c->L_e > 0) return false;
  const int lo = c->s.n_layers - c->L_d;
  const int R = (kind == 1 && lo > 0) ? R_lower : 1;
  return c->B * R <= PK_MAX_ROWS && R * (c->s.n_q_heads / c->s.n_kv_heads) <= PK_QR &&
         c->B * R * c->s.hidden <= PK_XS_FLOATS;
}

// One pass (Section 2.2) as a single cooperative launch of the persistent pass kernel.
dmtd_status enqueue_pass_fused(dmtd_ctx *c, int kind, int R_lower, bool write_token, int *out_argmax, float *out_logits) {
  const dmtd_model_shape &s = c->s;
  const int L = s.n_layers, lo = L - c->L_d;
  PassParams P{};
  P.layers = c->pass_layers; P.embed = c->embed; P.w_final = c->w_final; P.inv_freq = c->inv_freq;
  P.l_begin = (kind == 1 && lo > 0) ? 0 : lo; P.l_split = lo; P.l_end = L;
  P.R_lo = (kind == 1 && lo > 0) ? R_lower : 1; P.B = c->B;
  P.H = s.hidden; P.I = s.intermediate; P.nq = s.n_q_heads; P.nkv = s.n_kv_heads; P.vocab = s.vocab;
  P.max_seq = c->max_seq; P.ldl = c->ldl; P.eps = s.rms_eps;
  P.kind = kind; P.write_token = write_token ? 1 : 0; P.kv_f32 = s.kv_dtype == DMTD_F32 ? 1 : 0; P.kv_f16 = s.kv_dtype == DMTD_F16 ? 1 : 0;
  P.tokens = c->tokens; P.st = c->dstate;
  P.x_lo = c->x_lo; P.x_up = c->x_up; P.qkv = c->qkv; P.gu = c->gu; P.logits = c->logits;
  P.timing = c->pass_timing;
  P.part_o = c->f_part_o; P.part_ml = c->f_part_ml; P.amax_val = c->amax_val; P.amax_idx = c->amax_idx;
  P.out_argmax = out_argmax; P.barrier = c->grid_bar; P.error = &c->dstate->error;
  P.wait_limit = kDeviceWaitLimitTicks;
  P.sample = sample_params(c);
  CUDA_TRY(c, cudaMemsetAsync(c->grid_bar, 0, sizeof(unsigned int), c->stream));
  void *args[] = {&P};
  CUDA_TRY(c, cudaLaunchCooperativeKernel((const void *)dmtd_pass_kernel, dim3(c->n_sms), dim3(PK_THREADS), args,
                                          (size_t)PK_SMEM_BYTES, c->stream));
  c->launches += 1;
  if (out_logits)
    CUDA_TRY(c, cudaMemcpy2DAsync(out_logits, (size_t)s.vocab * 4, c->logits, (size_t)c->ldl * 4, (size_t)s.vocab * 4, c->B,
                                  cudaMemcpyDeviceToDevice, c->stream));
  return DMTD_OK;
}

// ---------------------------------------------------------------------------- small fp32 models

// Can passes of this model run as one launch of one cluster (small_pass_kernel)?
dmtd_status setup_small(dmtd_ctx *c) {
  const dmtd_model_shape &s = c->s;
  c->small_ok = false;
  if (is_bf16(c) || s.kv_dtype != DMTD_F32 || s.head_dim != SP_D || s.n_layers > SP_MAX_LAYERS ||
      !small_pass_fits(s.hidden, s.intermediate, s.n_q_heads, s.n_kv_heads, s.vocab))
    return DMTD_OK;
  const auto kernel = small_pass_kernel;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SP_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return DMTD_OK;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(SP_CTAS); cfg.blockDim = dim3(SP_THREADS); cfg.dynamicSmemBytes = SP_SMEM;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = SP_CTAS; attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return DMTD_OK; }
  c->small_ok = clusters >= 1;
  return DMTD_OK;
}

// ... and a pass of this kind?  At most eight rows, and as many cached keys to a block (a slice of a kv head) as it walks in
// the time that the launches of the other form take.  Cycles of the 4-layer test shape (hidden 256), launches against one
// cluster, us: 1 sequence, 3 passes, context 16 / 600 / 1800 / 7000 (875 keys to a block) 159 / 190 / 232 / 298 against 96 /
// 105 / 121 / 199; 2 sequences (6 rows), context 1800 (450 keys) 239 against 183, 7000 (1750 keys) 328 against 371; 4 sequences, 2 passes,
// 1800 (900 keys) 194 against 190; 8 sequences, 1 pass, 600 keys 130 against 122, 1800 keys 157 against 200.
bool small_pass_ok(const dmtd_ctx *c, int kind, int R_lower) {
  if (!c->small_ok || c->pass_option == 0 || c->literal_sum || c->L_e > 0) return false;
  const dmtd_model_shape &s = c->s;
  const int R = kind == 1 && s.n_layers > c->L_d ? R_lower : 1, G = s.n_q_heads / s.n_kv_heads, M = c->B * R, items = c->B * s.n_kv_heads;
  if (M > SP_MAX_ROWS || R * G > SP_MAX_ROWS || items > SP_CTAS) return false;
  if (c->h.n_known / (SP_CTAS / items) > (M <= 4 ? 900 : 500)) return false;
  return small_pass_smem(small_pass_map(s.hidden, s.intermediate, s.n_q_heads, s.n_kv_heads, s.n_layers, c->B, R)) <= SP_SMEM;
}

// n passes from here to the end of the cycle at most, as one launch.
dmtd_status enqueue_small(dmtd_ctx *c, int n, bool write_token, int *out_argmax, float *out_logits, int *out_tokens) {
  const dmtd_model_shape &s = c->s;
  const bool full = c->h.slot == 0;
  SmallParams P{};
  for (int l = 0; l < s.n_layers; ++l) {
    const LayerDev &ld = c->layers[l];
    P.layers[l] = SmallLayer{ld.qkv.wf, ld.o.wf, ld.gu.wf, ld.down.wf, ld.w_in, ld.w_post, ld.w_qn, ld.w_kn,
                             static_cast<float *>(c->kc) + (size_t)l * c->kv_layer_elems, static_cast<float *>(c->vc) + (size_t)l * c->kv_layer_elems};
  }
  P.embed = c->embed.wf; P.w_final = c->w_final; P.inv_freq = c->inv_freq;
  P.n_layers = s.n_layers; P.lo = s.n_layers - c->L_d; P.B = c->B;
  P.full = full ? 1 : 0;
  P.lower = full && P.lo > 0 ? 1 : 0;
  P.R = full && P.lo > 0 ? c->h.n_known - c->h.lo_len : 1;
  P.n_passes = n;
  P.ns = SP_CTAS / (c->B * s.n_kv_heads);
  P.H = s.hidden; P.I = s.intermediate; P.nq = s.n_q_heads; P.nkv = s.n_kv_heads; P.vocab = s.vocab; P.max_seq = c->max_seq;
  P.eps = s.rms_eps; P.write_token = write_token ? 1 : 0;
  P.tokens = c->tokens; P.st = c->dstate; P.out_logits = out_logits; P.out_argmax = out_argmax; P.out_tokens = out_tokens; P.tau = c->tau;
  P.sample = sample_params(c);
  P.map = small_pass_map(s.hidden, s.intermediate, s.n_q_heads, s.n_kv_heads, s.n_layers, P.B, P.R);
  P.error = &c->dstate->error; P.wait_limit = kDeviceWaitLimitTicks;
  CUDA_TRY(c, launch_cluster(small_pass_kernel, dim3(SP_CTAS), dim3(SP_THREADS), small_pass_smem(P.map), c->stream, SP_CTAS, P));
  c->launches += 1;
  return DMTD_OK;
}

// The passes of at most n that the next launch of small_pass_kernel takes (0: none): to the end of the cycle.  Unasked only
// for models that gain by it.
int small_passes(const dmtd_ctx *c, int n) {
  const int kind = c->h.slot == 0 ? 1 : 2, R = c->h.n_known - c->h.lo_len;
  if (!small_pass_ok(c, kind, R)) return 0;
  const dmtd_model_shape &s = c->s;
  if (c->pass_option < 0 && small_pass_gain(s.hidden, s.intermediate, s.n_q_heads, s.n_kv_heads, s.vocab, s.n_layers, c->L_d, c->B, c->tau,
                                            small_pass_ok(c, 1, c->tau)) <= 0.f)
    return 0;
  return std::min(std::min(n, c->tau - c->h.slot), SP_MAX_POSITIONS - R);
}

// One pass of the decode stage (Section 2.2).  kind 1: full pass - the R = n_known - lo_len
// pending rows through the lower layers (refill), the newest row through the decoding
// layers.  kind 2: the newest token's embedding through the decoding layers only.
dmtd_status enqueue_pass(dmtd_ctx *c, int kind, int R_lower, bool write_token, int *out_argmax, float *out_logits) {
  const int B = c->B, L = c->s.n_layers, lo = L - c->L_d, H = c->s.hidden;
  const int newest = c->h.n_known - 1;
  if (!c->capturing && fused_pass_ok(c, kind, R_lower, false))
    return enqueue_pass_fused(c, kind, R_lower, write_token, out_argmax, out_logits);
  if (c->L_e > 0) {
    // ExDy: the newest token's embedding goes through the encoding layers in every pass; their
    // output h_enc is kept until the thinking layers have seen the position
    const int Le = c->L_e;
    TRY(launch_embed(c, &c->dstate->newest, B, 1, c->x_up, false));
    for (int l = 0; l < Le; ++l) TRY(run_layer(c, l, c->x_up, B, 1, &c->dstate->newest, newest + 1));
    if (kind == 1) {
      // full pass: the pending rows' h_enc and the newest row's through the thinking layers
      gather_pending_kernel<<<B * R_lower, 256, 0, c->stream>>>(c->h_pend, c->pend_cap, c->x_up, R_lower, H, c->x_lo);
      LAUNCH_OK(c, "gather_pending_kernel");
      TRY(launch_rope_table(c, &c->dstate->lo_len, R_lower));
      for (int l = Le; l < lo; ++l) TRY(run_layer(c, l, c->x_lo, B, R_lower, &c->dstate->lo_len, c->h.n_known));
      if (c->literal_sum) {
        CUDA_TRY(c, launch_pdl(select_last_kernel, dim3(B), dim3(256), (size_t)(0), c->stream,
                                c->x_lo, R_lower, H, c->h_base));
        LAUNCH_OK(c, "select_last_kernel");
        copy_rows_kernel<<<64, 256, 0, c->stream>>>(c->h_base, c->x_up, (size_t)B * H / 4, 1);
        LAUNCH_OK(c, "copy_rows_kernel");
      } else {
        CUDA_TRY(c, launch_pdl(select_last_kernel, dim3(B), dim3(256), (size_t)(0), c->stream,
                                c->x_lo, R_lower, H, c->x_up));
        LAUNCH_OK(c, "select_last_kernel");
      }
    } else if (kind == 2) {
      save_pending_kernel<<<B, 256, 0, c->stream>>>(c->x_up, c->h_pend, c->pend_cap, H, c->dstate);
      LAUNCH_OK(c, "save_pending_kernel");
    }
  } else if (kind == 1 && lo > 0) {
    TRY(launch_embed(c, &c->dstate->lo_len, B, R_lower, c->x_lo, false));
    for (int l = 0; l < lo; ++l) TRY(run_layer(c, l, c->x_lo, B, R_lower, &c->dstate->lo_len, c->h.n_known));
    CUDA_TRY(c, launch_pdl(select_last_kernel, dim3(B), dim3(256), (size_t)(0), c->stream,
                            c->x_lo, R_lower, H, c->x_up));
    LAUNCH_OK(c, "select_last_kernel");
    if (c->literal_sum) TRY(launch_embed(c, &c->dstate->newest, B, 1, c->x_up, true));
  } else {
    TRY(launch_embed(c, &c->dstate->newest, B, 1, c->x_up, false));
  }
  // the newest position's row is the last one of a full pass's table
  if (kind == 1 && lo > 0) c->rope_rows = c->rope_tab + (size_t)(R_lower - 1) * (c->s.head_dim / 2);
  for (int l = lo; l < L; ++l) TRY(run_layer(c, l, c->x_up, B, 1, &c->dstate->newest, newest + 1));
  return run_head(c, B, write_token, out_argmax, out_logits, kind, 0);
}

void host_advance(dmtd_ctx *c, int kind) {
  dmtd_state &h = c->h;
  if (kind == 1) { h.lo_len = h.n_known; h.cycle += 1; }
  h.up_len = h.n_known;
  h.n_known += 1;
  h.slot = (h.slot + 1) % h.tau;
  h.n_emitted += 1;
}

// Calls that return results to the host synchronise the stream anyway: they bring the device's
// error word along (4 bytes into pinned memory, queued before the synchronise) and turn it into a
// status.  The word is sticky on the device and the failure is sticky here until dmtd_reset.
dmtd_status queue_error_read(dmtd_ctx *c) {
  CUDA_TRY(c, cudaMemcpyAsync(c->h_error, &c->dstate->error, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  return DMTD_OK;
}
dmtd_status device_error_status(dmtd_ctx *c, int word) {
  if (word == 0) return DMTD_OK;
  if (word == PK_ERR_TOKEN) {
    c->device_failure = DMTD_ERR_INVALID_ARG;
    return fail(c, DMTD_ERR_INVALID_ARG, "a token id outside [0, vocab) reached the embedding gather; "
                "the results since then are invalid, call dmtd_reset");
  }
  c->device_failure = DMTD_ERR_TIMEOUT;
  return fail(c, DMTD_ERR_TIMEOUT, "a device-side wait gave up (%s); the results since then are invalid, call dmtd_reset",
              word == PK_ERR_COPY_WAIT ? "weight copy" : word == PK_ERR_BARRIER_WAIT ? "grid barrier" : "tensor-core pipeline");
}
#define CHECK_NOT_FAILED(c)                                                                          \
  do {                                                                                               \
    if ((c)->device_failure != DMTD_OK)                                                              \
      return fail((c), (c)->device_failure, "the context reported a device-side error earlier; call dmtd_reset"); \
  } while (0)

void destroy_graph(const dmtd_ctx::PassGraph &g) {
  cudaGraphExecDestroy(g.exec);              // (one that still runs is released when it has)
  cudaGraphDestroy(g.graph);
}
void drop_graphs(dmtd_ctx *c) {
  for (const auto &g : c->graphs) destroy_graph(g);
  c->graphs.clear();
}

// Captured passes carry the sampling parameters as an argument of their last launch: a change replaces it (a few microseconds; another
// capture takes 0.15 to 0.7 ms.  Parameters read from memory instead cost the pick of 32 sequences 3.4 us a pass: with them as
// arguments the generator's keys are worked out once for a warp).
void update_sampling(dmtd_ctx *c) {
  SampleParams sp = sample_params(c);
  for (const auto &g : c->graphs) {
    cudaKernelNodeParams p{};
    bool ok = cudaGraphKernelNodeGetParams(g.pick, &p) == cudaSuccess;
    if (ok) {
      void *args[] = {p.kernelParams[0], p.kernelParams[1], p.kernelParams[2], p.kernelParams[3], &sp, p.kernelParams[5]};
      static_assert(std::is_same<decltype(&argmax_kernel), void (*)(const float *, int, int, DevState *, SampleParams, PickParams)>::value, "args");
      p.func = reinterpret_cast<void *>(argmax_kernel);
      p.kernelParams = args;
      p.extra = nullptr;
      ok = cudaGraphExecKernelNodeSetParams(g.exec, g.pick, &p) == cudaSuccess;
    }
    if (!ok) {                               // captured again when it is next needed
      cudaGetLastError();
      drop_graphs(c);
      return;
    }
  }
}

// Capture a steady-state pass (R_lower = tau) into a graph.  Positions come from the device
// counters and the attention grid covers max_seq, so one graph serves the whole generation.
dmtd_status capture_pass(dmtd_ctx *c, int kind, int forms) {
  cudaGraph_t graph = nullptr;
  int64_t before = c->launches;
  if (!c->capture_stream) CUDA_TRY(c, cudaStreamCreateWithFlags(&c->capture_stream, cudaStreamNonBlocking));
  cudaError_t e = cudaStreamBeginCapture(c->capture_stream, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return fail(c, DMTD_ERR_CUDA, "begin capture: %s", cudaGetErrorString(e));
  cudaStream_t user_stream = c->stream;
  c->stream = c->capture_stream;
  c->capturing = true;
  dmtd_status st = enqueue_pass(c, kind, c->tau, true, nullptr, nullptr);
  cudaGraphNode_t pick = nullptr;
  {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    const cudaGraphNode_t *last = nullptr;
    size_t n_last = 0;
    if (cudaStreamGetCaptureInfo(c->capture_stream, &status, nullptr, nullptr, &last, &n_last) == cudaSuccess && n_last == 1) pick = last[0];
  }
  e = cudaStreamEndCapture(c->capture_stream, &graph);
  c->capturing = false;
  c->stream = user_stream;
  int nodes = (int)(c->launches - before);
  c->launches = before;
  if (st != DMTD_OK) { if (graph) cudaGraphDestroy(graph); return st; }
  if (e != cudaSuccess) return fail(c, DMTD_ERR_CUDA, "end capture: %s", cudaGetErrorString(e));
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  if (e != cudaSuccess) {
    cudaGraphDestroy(graph);
    return fail(c, DMTD_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
  }
  if ((int)c->graphs.size() == kMaxGraphs) {
    const auto oldest = std::min_element(c->graphs.begin(), c->graphs.end(), [](const auto &a, const auto &b) { return a.used < b.used; });
    destroy_graph(*oldest);
    c->graphs.erase(oldest);
  }
  c->graphs.push_back({kind, c->B, kind == 1 ? c->tau : 0, forms, nodes, exec, graph, pick, 0});
  return DMTD_OK;
}

// Which of a pass's attention launches take equal shares at the position at hand (they change at most once as a context grows).
int attention_forms(const dmtd_ctx *c, int kind) {
  const auto shares = [&](int R) { return attention_ranks(c, c->B, R, c->h.n_known, true) == 0; };
  return (shares(1) ? 1 : 0) | (kind == 1 && shares(c->tau) ? 2 : 0);
}

// The graph of a kind of pass for the batch and cycle length at hand; captured: it is a new one.
dmtd_status ready_graph(dmtd_ctx *c, int kind, const dmtd_ctx::PassGraph **out, bool *captured = nullptr) {
  const int tau = kind == 1 ? c->tau : 0, forms = attention_forms(c, kind);
  auto it = std::find_if(c->graphs.begin(), c->graphs.end(),
                         [&](const auto &g) { return g.kind == kind && g.B == c->B && g.tau == tau && g.forms == forms; });
  if (captured) *captured = it == c->graphs.end();
  if (it == c->graphs.end()) {
    TRY(capture_pass(c, kind, forms));
    it = c->graphs.end() - 1;
  }
  it->used = ++c->graph_uses;
  *out = &*it;
  return DMTD_OK;
}

// The passes of few rows are captured before the first one is asked for: while the context is created, for its largest batch, and
// behind a prefill of another batch or cycle length, while the device works on it (the host takes 0.2 to 1.5 ms for each pass).  A
// failure here is left for the pass itself to meet.
void capture_ahead(dmtd_ctx *c) {
  if (!c->use_graph || !c->fused_ok || c->B > PK_MAX_ROWS || c->literal_sum || c->L_e > 0) return;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusActive;
  if (cudaStreamIsCapturing(c->stream, &status) != cudaSuccess || status != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  for (int kind = 1; kind <= (c->tau > 1 ? 2 : 1); ++kind) {
    if (fused_pass_ok(c, kind, c->tau, true)) continue;
    const dmtd_ctx::PassGraph *g = nullptr;
    bool is_new = false;
    if (ready_graph(c, kind, &g, &is_new) != DMTD_OK || (is_new && cudaGraphUpload(g->exec, c->capture_stream) != cudaSuccess)) {
      cudaGetLastError();
      return;
    }
  }
}

// Run the next pass of the schedule in greedy mode.
dmtd_status run_greedy_pass(dmtd_ctx *c) {
  int kind = c->h.slot == 0 ? 1 : 2;
  int R_lower = c->h.n_known - c->h.lo_len;
  const bool captured = c->use_graph && (kind == 2 || R_lower == c->tau);
  if (fused_pass_ok(c, kind, R_lower, captured)) {
    TRY(enqueue_pass_fused(c, kind, R_lower, true, nullptr, nullptr));
  } else if (captured) {
    const dmtd_ctx::PassGraph *g = nullptr;
    TRY(ready_graph(c, kind, &g));
    CUDA_TRY(c, cudaGraphLaunch(g->exec, c->stream));
    c->launches += g->nodes;
  } else {
    TRY(enqueue_pass(c, kind, R_lower, true, nullptr, nullptr));
  }
  host_advance(c, kind);
  return DMTD_OK;
}

dmtd_status validate_shape(const dmtd_model_shape *s, int L_d, int tau, int max_batch, int max_seq) {
  if (s->n_layers < 1 || s->hidden < 1 || s->n_q_heads < 1 || s->n_kv_heads < 1 || s->intermediate < 1 || s->vocab < 1)
    return fail(nullptr, DMTD_ERR_SHAPE, "model dimensions must be positive");
  if (L_d < 1 || L_d > s->n_layers) return fail(nullptr, DMTD_ERR_SHAPE, "L_d must be in [1, n_layers]");
  if (tau < 1) return fail(nullptr, DMTD_ERR_SHAPE, "tau must be >= 1");
  if (max_batch < 1 || max_seq < 2) return fail(nullptr, DMTD_ERR_INVALID_ARG, "max_batch >= 1 and max_seq >= 2 required");
  if (s->n_q_heads % s->n_kv_heads) return fail(nullptr, DMTD_ERR_SHAPE, "n_q_heads must be a multiple of n_kv_heads");
  if (s->n_q_heads / s->n_kv_heads > ATTN_QR) return fail(nullptr, DMTD_ERR_SHAPE, "at most 16 query heads per kv head");
  if (s->head_dim != 64 && s->head_dim != 128) return fail(nullptr, DMTD_ERR_SHAPE, "head_dim must be 64 or 128");
  if (s->weight_dtype != DMTD_F32 && s->weight_dtype != DMTD_BF16) return fail(nullptr, DMTD_ERR_SHAPE, "weight_dtype");
  if (s->kv_dtype != DMTD_F32 && s->kv_dtype != DMTD_BF16 && s->kv_dtype != DMTD_F16) return fail(nullptr, DMTD_ERR_SHAPE, "kv_dtype");
  int mult = s->weight_dtype == DMTD_BF16 ? 32 : 4;
  if (s->hidden % mult || s->intermediate % mult)
    return fail(nullptr, DMTD_ERR_SHAPE, "hidden and intermediate must be multiples of %d", mult);
  if (s->weight_dtype == DMTD_BF16 && ((s->n_q_heads * s->head_dim) % 16 || s->intermediate % 16))
    return fail(nullptr, DMTD_ERR_SHAPE, "fused row blocks must be multiples of 16");
  if (!s->tied_lm_head) return fail(nullptr, DMTD_ERR_UNSUPPORTED, "only a tied LM head is supported");
  if (!(s->rope_theta > 0.f) || !(s->rms_eps >= 0.f)) return fail(nullptr, DMTD_ERR_SHAPE, "rope_theta / rms_eps");
  return DMTD_OK;
}

}  // namespace

// ================================================================================ C ABI

extern "C" {

dmtd_status dmtd_create(const dmtd_model_shape *shape, int32_t L_d, int32_t tau, int32_t max_batch,
                        int32_t max_seq, const dmtd_weights *w, void *cuda_stream, dmtd_ctx **out) {
  if (!shape || !w || !out || !w->embed || !w->final_norm || !w->layers)
    return fail(nullptr, DMTD_ERR_INVALID_ARG, "null argument");
  if (w->lm_head) return fail(nullptr, DMTD_ERR_UNSUPPORTED, "only a tied LM head is supported (lm_head must be NULL)");
  dmtd_status vs = validate_shape(shape, L_d, tau, max_batch, max_seq);
  if (vs != DMTD_OK) return vs;

  dmtd_ctx *c = new dmtd_ctx();
  auto bail = [&](dmtd_status st) { g_create_error = c->err; dmtd_destroy(c); return st; };
#define CTRY(expr) do { dmtd_status s__ = (expr); if (s__ != DMTD_OK) return bail(s__); } while (0)
#define CCUDA(expr) do { cudaError_t e__ = (expr); if (e__ != cudaSuccess) { \
    fail(c, DMTD_ERR_CUDA, "%s failed: %s", #expr, cudaGetErrorString(e__)); return bail(DMTD_ERR_CUDA); } } while (0)

  c->s = *shape; c->L_d = L_d; c->tau = tau; c->max_batch = max_batch; c->max_seq = max_seq;
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  CCUDA(cudaGetDevice(&c->device));
  CCUDA(cudaDeviceGetAttribute(&c->n_sms, cudaDevAttrMultiProcessorCount, c->device));
  const dmtd_model_shape &s = c->s;
  const int H = s.hidden, D = s.head_dim, QD = s.n_q_heads * D, KVD = s.n_kv_heads * D, I = s.intermediate;
  const int I_pad = (I + TG_KB - 1) / TG_KB * TG_KB;

  // weights; every bf16 context whose dimensions fit also gets the copy the tcgen05 GEMM reads:
  // every pass outside the pass kernel uses it
  // (An intermediate size between two multiples of 64 is filled up: gate and up rows of zeros give the down projection's
  // last k block zeros.  6 layers of hidden 640, intermediate 1824, on the mma.sync kernels against these, us: prefill of 8 / 130 / 2000 tokens
  // 270 / 878 / 10237 against 234 / 290 / 1195; a cycle of three passes for 5 / 16 / 64 sequences 493 / 739 / 2011 against 351 / 361 / 488.)
  c->umma_ok = s.weight_dtype == DMTD_BF16 && H % TG_KB == 0 && QD % TG_KB == 0;
  // DMTD_WEIGHT_COPIES=1 in the environment keeps only the atom stream (half the weight memory):
  // every projection then runs on the mma.sync kernels, the prefill included (slower at every row count)
  if (const char *e = getenv("DMTD_WEIGHT_COPIES")) if (atoi(e) == 1) c->umma_ok = false;
  c->layers.resize(s.n_layers);
  // k-slab width of the packed matrices: contexts small enough for the pass kernel (which stages only the slabs a block's
  // share touches, and gains from short ones) get 256-wide slabs; in larger ones the layers' streams are read by the
  // mma.sync GEMV alone, which is faster with 1280-wide slabs (without the block copy, or with "tcgen05_gemm" off), and
  // the head's by the embedding gather
  const int aps = max_batch <= PK_MAX_ROWS ? 8 : 40;
  for (int l = 0; l < s.n_layers; ++l) {
    const dmtd_layer_weights &lw = w->layers[l];
    const void *ptrs[] = {lw.input_norm, lw.q_proj, lw.k_proj, lw.v_proj, lw.q_norm, lw.k_norm, lw.o_proj,
                          lw.post_norm, lw.gate_proj, lw.up_proj, lw.down_proj};
    for (const void *p : ptrs)
      if (!p) { fail(c, DMTD_ERR_INVALID_ARG, "null weight pointer in layer %d", l); return bail(DMTD_ERR_INVALID_ARG); }
    LayerDev &ld = c->layers[l];
    const void *qkv_src[3] = {lw.q_proj, lw.k_proj, lw.v_proj};
    int qkv_n[3] = {QD, KVD, KVD};
    CTRY(pack_matrix(c, &ld.qkv, H, qkv_src, qkv_n, 3, aps));
    const void *o_src[1] = {lw.o_proj}; int o_n[1] = {H};
    // k-slabs of two heads: a block of the pass kernel then merges the attention slices of few heads
    CTRY(pack_matrix(c, &ld.o, QD, o_src, o_n, 1, D == 128 ? 8 : 40));
    const void *gu_src[2] = {lw.gate_proj, lw.up_proj}; int gu_n[2] = {I, I};
    CTRY(pack_matrix(c, &ld.gu, H, gu_src, gu_n, 2, aps));
    const void *d_src[1] = {lw.down_proj}; int d_n[1] = {H};
    CTRY(pack_matrix(c, &ld.down, I, d_src, d_n, 1, aps));
    if (c->umma_ok) {
      CTRY(pack_umma(c, &ld.qkv_u, H, qkv_src, qkv_n, 3));
      CTRY(pack_umma(c, &ld.o_u, QD, o_src, o_n, 1));
      CTRY(pack_umma(c, &ld.gu_u, H, gu_src, gu_n, 2, true, 2 * I_pad));      // gate and up of one index side by side: the epilogue gates
      CTRY(pack_umma(c, &ld.down_u, I, d_src, d_n, 1));
    }
    CTRY(vec_to_float(c, &ld.w_in, lw.input_norm, H));
    CTRY(vec_to_float(c, &ld.w_post, lw.post_norm, H));
    CTRY(vec_to_float(c, &ld.w_qn, lw.q_norm, D));
    CTRY(vec_to_float(c, &ld.w_kn, lw.k_norm, D));
  }
  {
    const void *e_src[1] = {w->embed}; int e_n[1] = {s.vocab};
    CTRY(pack_matrix(c, &c->embed, H, e_src, e_n, 1, aps));
    if (c->umma_ok) CTRY(pack_umma(c, &c->embed_u, H, e_src, e_n, 1));
    CTRY(vec_to_float(c, &c->w_final, w->final_norm, H));
  }
  {
    std::vector<double> f(D / 2);
    for (int i = 0; i < D / 2; ++i) f[i] = std::pow((double)s.rope_theta, -2.0 * i / (double)D);
    CTRY(dev_alloc(c, &c->inv_freq, f.size()));
    CCUDA(cudaMemcpyAsync(c->inv_freq, f.data(), f.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    CCUDA(cudaStreamSynchronize(c->stream));
  }

  // sequence state
  size_t kvb = s.kv_dtype == DMTD_F32 ? 4 : 2;
  c->kv_layer_elems = (size_t)max_batch * s.n_kv_heads * max_seq * D;
  {
    unsigned char *p = nullptr;
    c->mem_kind = 2;
    CTRY(dev_alloc(c, &p, c->kv_layer_elems * s.n_layers * kvb)); c->kc = p;
    CTRY(dev_alloc(c, &p, c->kv_layer_elems * s.n_layers * kvb)); c->vc = p;
    c->mem_kind = 3;
  }
  CTRY(dev_alloc(c, &c->tokens, (size_t)max_batch * max_seq));
  CTRY(dev_alloc(c, &c->dstate, 1));
  CCUDA(cudaHostAlloc(reinterpret_cast<void **>(&c->h_error), sizeof(int), cudaHostAllocDefault));
  *c->h_error = 0;

  // workspace
  c->lda = std::max(H, std::max(QD, c->umma_ok ? I_pad : I));
  c->ldqkv = QD + 2 * KVD; c->ldgu = 2 * (c->umma_ok ? I_pad : I); c->ldl = (s.vocab + 15) / 16 * 16;
  // Keys per slice of the split-KV attention: enough slices that a decode step of max_batch
  // sequences fills the SMs about four times over, and no more (every slice costs a block its
  // set-up, a partial result and a share of the merge); whole 64-key tiles.
  {
    const int want = std::max(1, std::min(64, 4 * c->n_sms / std::max(1, max_batch * s.n_kv_heads)));
    c->CH = std::max(64, ((max_seq + want - 1) / want + 63) / 64 * 64);
  }
  c->nsplit_max = (max_seq + c->CH - 1) / c->CH;
  // Rows of the workspace = rows of one prefill chunk: up to 1024.  Chunks whose attention runs over key slices take
  // less where many slices would make the slices' partial results large; never fewer than a decode pass needs.
  c->part_rows = std::max(std::max(256, max_batch * std::max(tau, kFlashMinRows)), std::min(1024, 16384 / std::max(1, c->nsplit_max)));
  c->ws_rows = std::max(1024, c->part_rows);
  CTRY(dev_alloc(c, &c->x_lo, (size_t)c->ws_rows * H));
  CTRY(dev_alloc(c, &c->x_up, (size_t)max_batch * H));
  CTRY(dev_alloc(c, &c->act, (size_t)c->ws_rows * c->lda));
  CTRY(dev_alloc(c, &c->qkv, (size_t)c->ws_rows * c->ldqkv));
  CTRY(dev_alloc(c, &c->gu, (size_t)c->ws_rows * c->ldgu));
  CTRY(dev_alloc(c, &c->logits, (size_t)max_batch * c->ldl));
  CTRY(dev_alloc(c, &c->pick_val, (size_t)max_batch * ARGMAX_SLICES));
  CTRY(dev_alloc(c, &c->pick_idx, (size_t)max_batch * ARGMAX_SLICES));
  CTRY(dev_alloc(c, &c->pick_arrived, (size_t)max_batch + 1));
  CCUDA(cudaMemsetAsync(c->pick_arrived, 0, ((size_t)max_batch + 1) * sizeof(unsigned int), c->stream));
  CTRY(dev_alloc(c, &c->part_o, (size_t)c->part_rows * s.n_q_heads * c->nsplit_max * D));
  CTRY(dev_alloc(c, &c->part_ml, (size_t)c->part_rows * s.n_q_heads * c->nsplit_max * 2));
  CTRY(dev_alloc(c, &c->rope_tab, (size_t)c->ws_rows * (D / 2)));
  c->pend_cap = std::max(1, c->part_rows / max_batch);
  CTRY(dev_alloc(c, &c->h_pend, (size_t)max_batch * c->pend_cap * H));
  CTRY(dev_alloc(c, &c->h_base, (size_t)c->ws_rows * H));
  // activation blocks: hi and lo units of every row, the rows rounded up to whole column tiles (the last of them may be
  // mostly empty)
  if (c->umma_ok) {
    const size_t rows = (size_t)c->ws_rows + 16 * (c->ws_rows / TG_SPLIT_ROWS + 1) + TG_TILE_ROWS;
    CTRY(dev_alloc(c, &c->act_blocks, rows * (c->lda / 8) * 2));
    CTRY(dev_alloc(c, &c->gated_blocks, rows * (I_pad / 8) * 2));
  }
  CTRY(configure_kernels(c));
  CTRY(setup_fused(c));
  CTRY(setup_small(c));
  c->B = max_batch; c->h.n_known = 1;        // the batch that a context of few sequences most often has
  capture_ahead(c);
  c->B = 0;
  CTRY(dmtd_reset(c));
  CCUDA(cudaStreamSynchronize(c->stream));   // repacking done: the caller may free its weights
#undef CTRY
#undef CCUDA
  *out = c;
  return DMTD_OK;
}

void dmtd_destroy(dmtd_ctx *c) {
  if (!c) return;
  if (c->stream || true) cudaStreamSynchronize(c->stream);
  drop_graphs(c);
  if (c->capture_stream) cudaStreamDestroy(c->capture_stream);
  for (void *p : c->allocs) cudaFree(p);
  if (c->h_error) cudaFreeHost(c->h_error);
  delete c;
}

dmtd_status dmtd_reset(dmtd_ctx *c) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  DevState z{};
  z.tau = c->tau;
  CUDA_TRY(c, cudaMemcpyAsync(c->dstate, &z, sizeof z, cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  c->h = dmtd_state{};
  c->h.tau = c->tau; c->h.L_d = c->L_d;
  c->prefilled = false; c->B = 0;
  c->device_failure = DMTD_OK;
  if (c->h_error) *c->h_error = 0;
  return DMTD_OK;
}

dmtd_status dmtd_prefill(dmtd_ctx *c, const int32_t *prompt, int32_t B, int32_t P, const int32_t *forced_first,
                         int32_t *out_token, float *out_logits) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!prompt || B < 1 || P < 1) return fail(c, DMTD_ERR_INVALID_ARG, "prefill: null prompt or non-positive size");
  CHECK_NOT_FAILED(c);
  if (c->prefilled) return fail(c, DMTD_ERR_STATE, "prefill: context already holds a sequence; call dmtd_reset first");
  if (B > c->max_batch || P + 1 > c->max_seq) return fail(c, DMTD_ERR_CAPACITY, "prefill: B=%d P=%d exceed max_batch=%d max_seq=%d", B, P, c->max_batch, c->max_seq);
  const int L = c->s.n_layers, lo = L - c->L_d;
  c->B = B;
  CUDA_TRY(c, cudaMemcpy2DAsync(c->tokens, (size_t)c->max_seq * 4, prompt, (size_t)P * 4, (size_t)P * 4, B,
                                cudaMemcpyDeviceToDevice, c->stream));
  // All prompt rows through all layers (Section 2.2: the prefill is pass 1 of cycle 1), in
  // causal chunks of rows that fit the workspace.
  const int Rc_max = chunk_positions(c, B);
  int last_R = 0;
  for (int p0 = 0; p0 < P; p0 += Rc_max) {
    int R = std::min(Rc_max, P - p0);
    set_int_kernel<<<1, 1, 0, c->stream>>>(&c->dstate->scratch, p0);
    LAUNCH_OK(c, "set_int_kernel");
    TRY(launch_embed(c, &c->dstate->scratch, B, R, c->x_lo, false));
    for (int l = 0; l < L; ++l) {
      if (c->literal_sum && c->L_e > 0) {
        // Eq. 4's sum with h_enc in h_emb's place: keep the encoding layers' output, add it at the boundary
        if (l == c->L_e) {
          copy_rows_kernel<<<256, 256, 0, c->stream>>>(c->x_lo, c->h_base, (size_t)B * R * c->s.hidden / 4, 0);
          LAUNCH_OK(c, "copy_rows_kernel");
        }
        if (l == lo) {
          copy_rows_kernel<<<256, 256, 0, c->stream>>>(c->h_base, c->x_lo, (size_t)B * R * c->s.hidden / 4, 1);
          LAUNCH_OK(c, "copy_rows_kernel");
        }
      } else if (l == lo && c->literal_sum && lo > 0) {
        TRY(launch_embed(c, &c->dstate->scratch, B, R, c->x_lo, true));
      }
      TRY(run_layer(c, l, c->x_lo, B, R, &c->dstate->scratch, p0 + R));
    }
    last_R = R;
  }
  CUDA_TRY(c, launch_pdl(select_last_kernel, dim3(B), dim3(256), (size_t)(0), c->stream,
                          c->x_lo, last_R, c->s.hidden, c->x_up));
  LAUNCH_OK(c, "select_last_kernel");
  // n_known must read P when the head writes the token
  set_int_kernel<<<1, 1, 0, c->stream>>>(&c->dstate->n_known, P);
  LAUNCH_OK(c, "set_int_kernel");
  TRY(run_head(c, B, forced_first == nullptr, out_token, out_logits, 0, P));
  if (forced_first)
    CUDA_TRY(c, cudaMemcpy2DAsync(c->tokens + P, (size_t)c->max_seq * 4, forced_first, 4, 4, B,
                                  cudaMemcpyDeviceToDevice, c->stream));
  c->h.n_known = P + 1; c->h.lo_len = P; c->h.up_len = P; c->h.cycle = 1;
  c->h.slot = 1 % c->tau; c->h.n_emitted = 1;
  c->prefilled = true;
  capture_ahead(c);
  return DMTD_OK;
}

dmtd_status dmtd_decode_cycle(dmtd_ctx *c, int32_t max_new, int32_t *out_tokens, int32_t *n_out) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!n_out || max_new < 0) return fail(c, DMTD_ERR_INVALID_ARG, "decode_cycle: n_out is null or max_new < 0");
  *n_out = 0;
  CHECK_NOT_FAILED(c);
  if (!c->prefilled) return fail(c, DMTD_ERR_STATE, "decode_cycle: no prefill yet");
  const int first = c->h.n_known;
  int n = 0, n_written = 0;                   // tokens; of them already in out_tokens
  dmtd_status rc = DMTD_OK;
  while (n < max_new) {
    if (c->h.n_known + 1 > c->max_seq) { rc = fail(c, DMTD_ERR_CAPACITY, "decode_cycle: position %d does not fit max_seq=%d", c->h.n_known, c->max_seq); break; }
    const int together = small_passes(c, std::min(max_new - n, c->max_seq - c->h.n_known));
    if (together > 0) {
      rc = enqueue_small(c, together, true, nullptr, nullptr, n == 0 ? out_tokens : nullptr);
      if (rc != DMTD_OK) break;
      if (n == 0) n_written = together;
      for (int i = 0; i < together; ++i) host_advance(c, c->h.slot == 0 ? 1 : 2);
      n += together;
    } else {
      rc = run_greedy_pass(c);
      if (rc != DMTD_OK) break;              // the passes that were enqueued still count
      ++n;
    }
    if (c->h.slot == 0) break;     // the cycle is complete
  }
  if (out_tokens && n > n_written) {
    gather_tokens_kernel<<<c->B, 32, 0, c->stream>>>(c->tokens, c->max_seq, first, n, c->tau, out_tokens);
    LAUNCH_OK(c, "gather_tokens_kernel");
  }
  *n_out = n;
  return rc;
}

dmtd_status dmtd_decode_forced(dmtd_ctx *c, const int32_t *forced, int32_t n, float *out_logits, int32_t *out_argmax) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!forced || n < 0) return fail(c, DMTD_ERR_INVALID_ARG, "decode_forced: null forced tokens or n < 0");
  CHECK_NOT_FAILED(c);
  if (!c->prefilled) return fail(c, DMTD_ERR_STATE, "decode_forced: no prefill yet");
  if (c->h.n_known + n > c->max_seq) return fail(c, DMTD_ERR_CAPACITY, "decode_forced: %d more positions do not fit max_seq=%d", n, c->max_seq);
  if (n == 0) return DMTD_OK;
  // the forced tokens are the sequence's next n tokens: place them, then run the schedule
  // without letting the head overwrite them
  CUDA_TRY(c, cudaMemcpy2DAsync(c->tokens + c->h.n_known, (size_t)c->max_seq * 4, forced, (size_t)n * 4, (size_t)n * 4,
                                c->B, cudaMemcpyDeviceToDevice, c->stream));
  const size_t BV = (size_t)c->B * c->s.vocab;
  for (int i = 0; i < n; ++i) {
    const int together = small_passes(c, n - i);
    if (together > 0) {
      TRY(enqueue_small(c, together, false, out_argmax ? out_argmax + (size_t)i * c->B : nullptr, out_logits ? out_logits + (size_t)i * BV : nullptr, nullptr));
      for (int k = 0; k < together; ++k) host_advance(c, c->h.slot == 0 ? 1 : 2);
      i += together - 1;
      continue;
    }
    int kind = c->h.slot == 0 ? 1 : 2;
    TRY(enqueue_pass(c, kind, c->h.n_known - c->h.lo_len, false, out_argmax ? out_argmax + (size_t)i * c->B : nullptr,
                     out_logits ? out_logits + (size_t)i * BV : nullptr));
    host_advance(c, kind);
  }
  return DMTD_OK;
}

dmtd_status dmtd_step_layers(dmtd_ctx *c, int32_t l0, int32_t l1, float *hidden, int32_t B, int32_t R, int32_t pos0) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!hidden || l0 < 0 || l1 > c->s.n_layers || l0 > l1 || B < 1 || R < 1 || pos0 < 0)
    return fail(c, DMTD_ERR_INVALID_ARG, "step_layers: bad layer range, sizes or null hidden");
  CHECK_NOT_FAILED(c);
  if (B > c->max_batch || R > c->max_seq || pos0 > c->max_seq - R || (long long)B * R > (flash_attention_ok(c, R) ? c->ws_rows : c->part_rows))
    return fail(c, DMTD_ERR_CAPACITY, "step_layers: B=%d R=%d pos0=%d exceed max_batch=%d max_seq=%d rows=%d", B, R, pos0, c->max_batch, c->max_seq,
                flash_attention_ok(c, R) ? c->ws_rows : c->part_rows);
  set_int_kernel<<<1, 1, 0, c->stream>>>(&c->dstate->scratch, pos0);
  LAUNCH_OK(c, "set_int_kernel");
  TRY(launch_rope_table(c, &c->dstate->scratch, R));
  // the kernels read rows in 16-byte loads: rows that begin elsewhere are worked on in the workspace
  float *const x = reinterpret_cast<uintptr_t>(hidden) % 16 ? c->x_lo : hidden;
  const size_t bytes = (size_t)B * R * c->s.hidden * sizeof(float);
  if (x != hidden) CUDA_TRY(c, cudaMemcpyAsync(x, hidden, bytes, cudaMemcpyDeviceToDevice, c->stream));
  for (int l = l0; l < l1; ++l) TRY(run_layer(c, l, x, B, R, &c->dstate->scratch, pos0 + R));
  if (x != hidden) CUDA_TRY(c, cudaMemcpyAsync(hidden, x, bytes, cudaMemcpyDeviceToDevice, c->stream));
  return DMTD_OK;
}

dmtd_status dmtd_masked_forward(dmtd_ctx *c, const int32_t *tokens, int32_t B, int32_t n, int32_t P, float *out_logits) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!tokens || !out_logits || B < 1 || P < 1 || n < P) return fail(c, DMTD_ERR_INVALID_ARG, "masked_forward: null pointer, or not 1 <= P <= n");
  CHECK_NOT_FAILED(c);
  if (c->prefilled) return fail(c, DMTD_ERR_STATE, "masked_forward: the context holds a sequence; call dmtd_reset first");
  if (B > c->max_batch || n > c->max_seq) return fail(c, DMTD_ERR_CAPACITY, "masked_forward: B=%d n=%d exceed max_batch=%d max_seq=%d", B, n, c->max_batch, c->max_seq);
  const int L = c->s.n_layers, lo = L - c->L_d, Le = c->L_e, H = c->s.hidden;
  c->B = B;
  CUDA_TRY(c, cudaMemcpy2DAsync(c->tokens, (size_t)c->max_seq * 4, tokens, (size_t)n * 4, (size_t)n * 4, B,
                                cudaMemcpyDeviceToDevice, c->stream));
  // Eq. 1-5 chunk by chunk: a chunk of rows goes through every layer before the next one starts
  // (each layer is causal and the earlier chunks' K and V are in the cache by then).
  const int Rc_max = chunk_positions(c, B);
  const size_t n_out = (size_t)(n - (P - 1));
  for (int p0 = 0; p0 < n; p0 += Rc_max) {
    const int R = std::min(Rc_max, n - p0);
    const size_t n4 = (size_t)B * R * H / 4;
    set_int_kernel<<<1, 1, 0, c->stream>>>(&c->dstate->scratch, p0);
    LAUNCH_OK(c, "set_int_kernel");
    TRY(launch_embed(c, &c->dstate->scratch, B, R, c->x_lo, false));                 // h_emb
    for (int l = 0; l < Le; ++l) TRY(run_layer(c, l, c->x_lo, B, R, &c->dstate->scratch, p0 + R));   // Eq. 1: h_enc
    copy_rows_kernel<<<256, 256, 0, c->stream>>>(c->x_lo, c->h_base, n4, 0);
    LAUNCH_OK(c, "copy_rows_kernel");
    for (int l = Le; l < lo; ++l) TRY(run_layer(c, l, c->x_lo, B, R, &c->dstate->scratch, p0 + R));  // Eq. 2: h_think
    masked_select_kernel<<<B * R, 256, 0, c->stream>>>(c->x_lo, c->h_base, R, H, p0, P, c->tau, c->literal_sum ? 1 : 0);   // Eq. 3-4
    LAUNCH_OK(c, "masked_select_kernel");
    for (int l = lo; l < L; ++l) TRY(run_layer(c, l, c->x_lo, B, R, &c->dstate->scratch, p0 + R));   // Eq. 5: decoding layers
    // ... and the LM head on the chunk's rows from position P - 1 on
    const int r0 = std::max(0, P - 1 - p0);
    if (r0 >= R) continue;
    const float *x0 = c->x_lo + (size_t)r0 * H;
    float *out = out_logits + (size_t)(p0 + r0 - (P - 1)) * c->s.vocab;
    const size_t V = c->s.vocab;
    if (R - r0 == (int)n_out) {
      TRY(run_head_rows(c, x0, B, R - r0, R, out, V));                               // all positions of all sequences
    } else if (R - r0 < B && n_out * V < (1ull << 31)) {
      // fewer positions than sequences: position by position, as each launch streams the head (18 positions of 64 sequences
      // in three chunks, 2 layers, 32000 tokens: a launch to a sequence 7.26 ms, to a position 2.23)
      for (int r = 0; r < R - r0; ++r) TRY(run_head_rows(c, x0 + (size_t)r * H, B, 1, R, out + r * V, (int)(n_out * V)));
    } else {
      for (int b = 0; b < B; ++b) TRY(run_head_rows(c, x0 + (size_t)b * R * H, 1, R - r0, R, out + b * n_out * V, V));
    }
  }
  // the cache now holds this forward's K and V; the schedule state is untouched (still "no sequence")
  c->B = 0;
  return DMTD_OK;
}

dmtd_status dmtd_prefill_host(dmtd_ctx *c, const int32_t *prompt_host, int32_t B, int32_t P, int32_t *out_token_host) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!prompt_host || B < 1 || P < 1) return fail(c, DMTD_ERR_INVALID_ARG, "prefill_host: null prompt or non-positive size");
  if (c->prefilled) return fail(c, DMTD_ERR_STATE, "prefill_host: context already holds a sequence; call dmtd_reset first");
  if (B > c->max_batch || P + 1 > c->max_seq) return fail(c, DMTD_ERR_CAPACITY, "prefill_host: sizes exceed capacity");
  // stage the prompt at the tail of the act workspace (unused until the first layer runs)
  int *stage = reinterpret_cast<int *>(c->gu);
  if ((size_t)B * P > (size_t)c->ws_rows * 2 * c->s.intermediate) return fail(c, DMTD_ERR_CAPACITY, "prefill_host: prompt larger than staging space");
  CUDA_TRY(c, cudaMemcpyAsync(stage, prompt_host, (size_t)B * P * 4, cudaMemcpyHostToDevice, c->stream));
  // the token buffer copy inside dmtd_prefill reads `stage` before any layer writes gu
  TRY(dmtd_prefill(c, stage, B, P, nullptr, nullptr, nullptr));
  if (out_token_host)
    CUDA_TRY(c, cudaMemcpy2DAsync(out_token_host, 4, c->tokens + P, (size_t)c->max_seq * 4, 4, B, cudaMemcpyDeviceToHost, c->stream));
  TRY(queue_error_read(c));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return device_error_status(c, *c->h_error);
}

dmtd_status dmtd_decode_cycle_host(dmtd_ctx *c, int32_t max_new, int32_t *out_tokens_host, int32_t *n_out) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!n_out) return fail(c, DMTD_ERR_INVALID_ARG, "decode_cycle_host: n_out is null");
  const int first = c->h.n_known;
  dmtd_status rc = dmtd_decode_cycle(c, max_new, nullptr, n_out);
  if (rc != DMTD_OK && rc != DMTD_ERR_CAPACITY) return rc;
  if (out_tokens_host && *n_out > 0)
    CUDA_TRY(c, cudaMemcpy2DAsync(out_tokens_host, (size_t)c->tau * 4, c->tokens + first, (size_t)c->max_seq * 4,
                                  (size_t)*n_out * 4, c->B, cudaMemcpyDeviceToHost, c->stream));
  TRY(queue_error_read(c));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  dmtd_status dev = device_error_status(c, *c->h_error);
  return dev != DMTD_OK ? dev : rc;
}

dmtd_status dmtd_get_state(const dmtd_ctx *c, dmtd_state *out) {
  if (!c || !out) return DMTD_ERR_INVALID_ARG;
  *out = c->h;
  return DMTD_OK;
}

dmtd_status dmtd_get_device_state(dmtd_ctx *c, dmtd_state *out) {
  if (!c || !out) return DMTD_ERR_INVALID_ARG;
  DevState d{};
  CUDA_TRY(c, cudaMemcpyAsync(&d, c->dstate, sizeof d, cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  TRY(device_error_status(c, d.error));
  out->n_known = d.n_known; out->lo_len = d.lo_len; out->up_len = d.up_len; out->cycle = d.cycle;
  out->slot = d.slot; out->n_emitted = d.n_emitted; out->tau = d.tau; out->L_d = c->L_d;
  return DMTD_OK;
}

dmtd_status dmtd_set_tau(dmtd_ctx *c, int32_t tau) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (tau < 1) return fail(c, DMTD_ERR_SHAPE, "set_tau: tau must be >= 1");
  if (c->prefilled && c->h.slot != 0) return fail(c, DMTD_ERR_STATE, "set_tau: only at a cycle boundary");
  if (c->max_batch * tau > c->part_rows) return fail(c, DMTD_ERR_CAPACITY, "set_tau: workspace too small for tau=%d", tau);
  c->tau = tau; c->h.tau = tau;
  CUDA_TRY(c, cudaMemcpyAsync(&c->dstate->tau, &c->tau, sizeof(int), cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return DMTD_OK;
}

dmtd_status dmtd_set_sampling(dmtd_ctx *c, float temperature, uint64_t seed) {
  if (!c) return DMTD_ERR_INVALID_ARG;
  if (!(temperature >= 0.f) || std::isinf(temperature)) return fail(c, DMTD_ERR_INVALID_ARG, "set_sampling: temperature must be finite and >= 0");
  c->temperature = temperature; c->sample_seed = seed;
  update_sampling(c);
  return DMTD_OK;
}

dmtd_status dmtd_set_option(dmtd_ctx *c, const char *name, int64_t value) {
  if (!c || !name) return DMTD_ERR_INVALID_ARG;
  if (!strcmp(name, "encoding_layers")) {
    if (c->prefilled) return fail(c, DMTD_ERR_STATE, "encoding_layers can only change before the prefill (call dmtd_reset first)");
    if (value < 0 || value + c->L_d > c->s.n_layers)
      return fail(c, DMTD_ERR_SHAPE, "encoding_layers must be in [0, n_layers - L_d]");
    c->L_e = (int)value; drop_graphs(c); return DMTD_OK;
  }
  if (!strcmp(name, "tcgen05_gemm_stages")) {
    if (value != 0 && (value < 2 || value > 6)) return fail(c, DMTD_ERR_INVALID_ARG, "tcgen05_gemm_stages takes 0 (chosen per launch) or 2..6");
    c->gemm_stages = (int)value; drop_graphs(c); return DMTD_OK;
  }
  if (value != 0 && value != 1) return fail(c, DMTD_ERR_INVALID_ARG, "option %s takes 0 or 1", name);
  if (!strcmp(name, "cuda_graph")) { c->use_graph = value != 0; return DMTD_OK; }
  if (!strcmp(name, "literal_sum")) { c->literal_sum = value != 0; drop_graphs(c); return DMTD_OK; }
  if (!strcmp(name, "fused_pass")) { c->pass_option = (int)value; return DMTD_OK; }
  if (!strcmp(name, "fused_qk_rope")) { c->fuse_qk_rope = value != 0; drop_graphs(c); return DMTD_OK; }
  if (!strcmp(name, "tcgen05_gemm")) { c->use_umma = value != 0; drop_graphs(c); return DMTD_OK; }
  if (!strcmp(name, "tc_attention")) { c->use_tc_attention = value != 0; drop_graphs(c); return DMTD_OK; }
  return fail(c, DMTD_ERR_INVALID_ARG, "unknown option %s", name);
}

dmtd_status dmtd_get_kv(dmtd_ctx *c, int32_t layer, void **k, void **v) {
  if (!c || layer < 0 || layer >= c->s.n_layers) return DMTD_ERR_INVALID_ARG;
  size_t kvb = c->s.kv_dtype == DMTD_F32 ? 4 : 2;
  if (k) *k = static_cast<unsigned char *>(c->kc) + (size_t)layer * c->kv_layer_elems * kvb;
  if (v) *v = static_cast<unsigned char *>(c->vc) + (size_t)layer * c->kv_layer_elems * kvb;
  return DMTD_OK;
}

dmtd_status dmtd_debug_set_error_word(dmtd_ctx *c, int32_t word) {
  if (!c || word < 0) return DMTD_ERR_INVALID_ARG;
  CUDA_TRY(c, cudaMemcpyAsync(&c->dstate->error, &word, sizeof(int), cudaMemcpyHostToDevice, c->stream));
  CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return DMTD_OK;
}

dmtd_status dmtd_get_memory_info(const dmtd_ctx *c, dmtd_memory_info *out) {
  if (!c || !out) return DMTD_ERR_INVALID_ARG;
  out->weight_stream_bytes = c->mem[0]; out->weight_block_bytes = c->mem[1];
  out->kv_cache_bytes = c->mem[2]; out->workspace_bytes = c->mem[3];
  return DMTD_OK;
}

dmtd_status dmtd_get_launch_count(const dmtd_ctx *c, int64_t *out) {
  if (!c || !out) return DMTD_ERR_INVALID_ARG;
  *out = c->launches;
  return DMTD_OK;
}

const char *dmtd_status_str(dmtd_status s) {
  switch (s) {
    case DMTD_OK: return "ok";
    case DMTD_ERR_INVALID_ARG: return "invalid argument";
    case DMTD_ERR_SHAPE: return "unsupported shape";
    case DMTD_ERR_STATE: return "call out of order";
    case DMTD_ERR_CAPACITY: return "capacity exceeded";
    case DMTD_ERR_CUDA: return "CUDA error";
    case DMTD_ERR_TIMEOUT: return "device wait timed out";
    case DMTD_ERR_UNSUPPORTED: return "unsupported";
  }
  return "unknown status";
}

const char *dmtd_last_error(const dmtd_ctx *c) { return c ? c->err.c_str() : g_create_error.c_str(); }

}  // extern "C"

// ---- step a4 as a context-free call ------------------------------------------------------

namespace {

struct AttnPlan { int CH, nsplit; size_t ml_off, o_off, bytes; };

// Scratch layout: [0, 256) unused, then the running (max, sum) pairs, then the unnormalised partial outputs, one set per (row, head, key slice).
AttnPlan attn_plan(int B, int R, int nq, int D, int n_keys) {
  AttnPlan p{};
  // slices enough to fill a GPU of about 150 SMs four times over (the call does not know the
  // number of kv heads: a quarter of the query heads is assumed), each of whole 64-key tiles
  const int want = std::max(1, std::min(64, 600 / std::max(1, B * std::max(1, nq / 4))));
  p.CH = std::max(64, ((n_keys + want - 1) / want + 63) / 64 * 64);
  p.nsplit = std::max(1, (n_keys + p.CH - 1) / p.CH);
  size_t slots = (size_t)B * R * nq * p.nsplit;
  p.ml_off = 256;
  p.o_off = p.ml_off + (slots * 2 * sizeof(float) + 255) / 256 * 256;
  p.bytes = p.o_off + slots * D * sizeof(float);
  return p;
}

dmtd_status attention_check(const float *q, const void *k, const void *v, int kv_dtype, int B, int R, int nq, int nkv,
                            int D, int max_seq, int pos0, const float *out) {
  if (!q || !k || !v || !out || B < 1 || R < 1 || pos0 < 0 || max_seq < 1)
    return fail(nullptr, DMTD_ERR_INVALID_ARG, "attention: null pointer or non-positive size");
  if (kv_dtype != DMTD_F32 && kv_dtype != DMTD_BF16 && kv_dtype != DMTD_F16) return fail(nullptr, DMTD_ERR_SHAPE, "attention: kv_dtype");
  if (D != 64 && D != 128) return fail(nullptr, DMTD_ERR_SHAPE, "attention: head_dim must be 64 or 128");
  if (nq < 1 || nkv < 1 || nq % nkv || nq / nkv > ATTN_QR)
    return fail(nullptr, DMTD_ERR_SHAPE, "attention: n_q_heads must be a multiple of n_kv_heads, at most 16 per kv head");
  if (R > max_seq || pos0 > max_seq - R) return fail(nullptr, DMTD_ERR_CAPACITY, "attention: pos0 = %d with R = %d rows exceeds max_seq = %d", pos0, R, max_seq);
  return DMTD_OK;
}

template <int D, typename KVT>
dmtd_status attention_launch_t(const float *q, const void *k, const void *v, int B, int R, int nq, int nkv, int max_seq,
                               int pos0, unsigned char *scratch, const AttnPlan &p, float *out, cudaStream_t stream) {
  float *part_ml = reinterpret_cast<float *>(scratch + p.ml_off);
  float *part_o = reinterpret_cast<float *>(scratch + p.o_off);
  const int G = nq / nkv, RB = std::max(1, ATTN_QR / G), n_rb = (R + RB - 1) / RB, ld = nq * D;
  int nsplit = p.nsplit;                    // slots per (row, head)
  cudaError_t e;
  int dev = 0, n_sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return fail(nullptr, DMTD_ERR_CUDA, "attention: device query failed");
  if (D == PK_D) {
    if constexpr (std::is_same<KVT, float>::value) {
      e = cudaFuncSetAttribute(attn_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ATTN_F32_SMEM);
      if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: %s", cudaGetErrorString(e));
      attn_f32_kernel<<<dim3(p.nsplit, nkv * n_rb, B), PK_THREADS, ATTN_F32_SMEM, stream>>>(
          q, ld, static_cast<const float *>(k), static_cast<const float *>(v), max_seq, nq, nkv, R, RB, p.CH, nullptr, pos0, part_o,
          part_ml, p.nsplit);
    } else {
      using Op = typename std::conditional<std::is_same<KVT, __half>::value, OpF16, OpBf16>::type;
      const int items = B * nkv * n_rb, units = (pos0 + R + AD_UNIT - 1) / AD_UNIT;
      // the clusters store whole float4; results that begin elsewhere go through the merge kernel, which stores single values
      const int ranks = reinterpret_cast<uintptr_t>(out) % 16 ? 0 : attn_cluster_ranks(dev, n_sms, items, units, units, false);
      if (ranks > 0) {
        const auto kernel = attn_decode_kernel<Op, false, true>;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AD_SMEM);
        if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: %s", cudaGetErrorString(e));
        e = launch_cluster(kernel, dim3(items * ranks), dim3(AD_THREADS), AD_SMEM, stream, ranks, q, ld, k, v, max_seq, nq, nkv, B, R, RB, nullptr, pos0,
                           out, nullptr, 1, AttnFuse{}, AttnBlocks{nullptr, ActTiles{}});
        if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: launch failed: %s", cudaGetErrorString(e));
        return DMTD_OK;
      }
      e = cudaFuncSetAttribute(attn_decode_kernel<Op>, cudaFuncAttributeMaxDynamicSharedMemorySize, AD_SMEM);
      if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: %s", cudaGetErrorString(e));
      const AttnDecodePlan dp = attn_decode_plan(n_sms, B * nkv * n_rb, (pos0 + R + AD_UNIT - 1) / AD_UNIT, p.nsplit);
      nsplit = dp.nsplit;
      e = launch_pdl(attn_decode_kernel<Op, false>, dim3(dp.n_blocks), dim3(AD_THREADS), AD_SMEM, stream, q, ld, k, v, max_seq, nq, nkv, B,
                     R, RB, nullptr, pos0, part_o, part_ml, nsplit, AttnFuse{}, AttnBlocks{nullptr, ActTiles{}});
      if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: launch failed: %s", cudaGetErrorString(e));
    }
  } else {
    const AttnPartialKernel<KVT> ap = attn_partial_for<D, KVT, false>(std::min(R, RB) * G, R, p.CH, (long long)p.nsplit * nkv * n_rb * B, n_sms);
    e = cudaFuncSetAttribute(ap.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ap.smem);
    if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: %s", cudaGetErrorString(e));
    ap.kernel<<<dim3(p.nsplit, nkv * n_rb, B), ap.threads, ap.smem, stream>>>(
        q, ld, static_cast<const KVT *>(k), static_cast<const KVT *>(v), max_seq, nq, nkv, R, RB, p.CH, nullptr, pos0, part_o,
        part_ml, p.nsplit, AttnFuse{});
  }
  int n_rh = B * R * nq;
  e = launch_pdl(attn_merge_kernel<D>, dim3((n_rh + 3) / 4), dim3(128), 0, stream, part_o, part_ml, nsplit, n_rh, nq, out, ld);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention: launch failed: %s", cudaGetErrorString(e));
  return DMTD_OK;
}

dmtd_status attention_launch(const float *q, const void *k, const void *v, int kv_dtype, int B, int R, int nq, int nkv,
                             int D, int max_seq, int pos0, unsigned char *scratch, const AttnPlan &p, float *out,
                             cudaStream_t stream) {
  if (D == 128) {
    if (kv_dtype == DMTD_BF16) return attention_launch_t<128, __nv_bfloat16>(q, k, v, B, R, nq, nkv, max_seq, pos0, scratch, p, out, stream);
    if (kv_dtype == DMTD_F16) return attention_launch_t<128, __half>(q, k, v, B, R, nq, nkv, max_seq, pos0, scratch, p, out, stream);
    return attention_launch_t<128, float>(q, k, v, B, R, nq, nkv, max_seq, pos0, scratch, p, out, stream);
  }
  if (kv_dtype == DMTD_BF16) return attention_launch_t<64, __nv_bfloat16>(q, k, v, B, R, nq, nkv, max_seq, pos0, scratch, p, out, stream);
  if (kv_dtype == DMTD_F16) return attention_launch_t<64, __half>(q, k, v, B, R, nq, nkv, max_seq, pos0, scratch, p, out, stream);
  return attention_launch_t<64, float>(q, k, v, B, R, nq, nkv, max_seq, pos0, scratch, p, out, stream);
}

}  // namespace

extern "C" {

size_t dmtd_attention_scratch_bytes(int32_t B, int32_t R, int32_t nq, int32_t D, int32_t n_keys) {
  if (B < 1 || R < 1 || nq < 1 || D < 1 || n_keys < 1) return 0;
  return attn_plan(B, R, nq, D, n_keys).bytes;
}

dmtd_status dmtd_attention_decode(const float *q, const void *k, const void *v, int32_t kv_dtype, int32_t B, int32_t R,
                                  int32_t nq, int32_t nkv, int32_t D, int32_t max_seq, int32_t pos0, void *scratch,
                                  size_t scratch_bytes, float *out, void *cuda_stream) {
  dmtd_status st = attention_check(q, k, v, kv_dtype, B, R, nq, nkv, D, max_seq, pos0, out);
  if (st != DMTD_OK) return st;
  AttnPlan p = attn_plan(B, R, nq, D, pos0 + R);
  if (!scratch) return fail(nullptr, DMTD_ERR_INVALID_ARG, "attention: null scratch");
  if (scratch_bytes < p.bytes)
    return fail(nullptr, DMTD_ERR_CAPACITY, "attention: scratch of %zu bytes is smaller than the %zu needed", scratch_bytes, p.bytes);
  return attention_launch(q, k, v, kv_dtype, B, R, nq, nkv, D, max_seq, pos0, static_cast<unsigned char *>(scratch), p, out,
                          static_cast<cudaStream_t>(cuda_stream));
}

}  // extern "C"

// ---- the same call with its scratch inside the library ------------------------------------
//
// For callers that must not allocate: the partial results go to a fixed array in the device
// image.  In host code the array's name is only a handle; the device address is looked up
// once per device (with that device current) and passed to the kernels like any pointer.

static __device__ __align__(256) unsigned char g_attention_static_scratch[DMTD_ATTENTION_STATIC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
unsigned char *g_static_scratch_addr[kMaxDevices] = {};
std::mutex g_static_scratch_mu;

// Device address of the fixed scratch on the current device.
dmtd_status static_scratch_address(unsigned char **out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(nullptr, DMTD_ERR_CUDA, "attention_static: cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return fail(nullptr, DMTD_ERR_UNSUPPORTED, "attention_static: device index %d", dev);
  std::lock_guard<std::mutex> lock(g_static_scratch_mu);
  if (!g_static_scratch_addr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_attention_static_scratch);
    if (e != cudaSuccess || !p)
      return fail(nullptr, DMTD_ERR_CUDA, "attention_static: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
    g_static_scratch_addr[dev] = static_cast<unsigned char *>(p);
  }
  *out = g_static_scratch_addr[dev];
  return DMTD_OK;
}

}  // namespace

extern "C" dmtd_status dmtd_attention_decode_static(const float *q, const void *k, const void *v, int32_t kv_dtype,
                                                    int32_t B, int32_t R, int32_t nq, int32_t nkv, int32_t D,
                                                    int32_t max_seq, int32_t pos0, float *out, void *cuda_stream) {
  dmtd_status st = attention_check(q, k, v, kv_dtype, B, R, nq, nkv, D, max_seq, pos0, out);
  if (st != DMTD_OK) return st;
  AttnPlan p = attn_plan(B, R, nq, D, pos0 + R);
  if (p.bytes > (size_t)DMTD_ATTENTION_STATIC_SCRATCH_BYTES)
    return fail(nullptr, DMTD_ERR_CAPACITY,
                "attention_static: this problem needs %zu bytes of scratch, the built-in array holds %zu; "
                "use dmtd_attention_decode with caller-owned scratch", p.bytes, (size_t)DMTD_ATTENTION_STATIC_SCRATCH_BYTES);
  unsigned char *scratch = nullptr;
  st = static_scratch_address(&scratch);
  if (st != DMTD_OK) return st;
  // nothing to clear: every (row, head, slice) entry the merge reads is written by this call
  return attention_launch(q, k, v, kv_dtype, B, R, nq, nkv, D, max_seq, pos0, scratch, p, out,
                          static_cast<cudaStream_t>(cuda_stream));
}

#ifdef DMTD_PASS_TIMING
// Profiling builds: copy out the stage time stamps of the last pass (2 x PK_TIMING_SLOTS ticks).
extern "C" int dmtd_debug_pass_timing(dmtd_ctx *c, long long *host_out) {
  if (!c || !c->pass_timing) return -1;
  cudaStreamSynchronize(c->stream);
  return (int)cudaMemcpy(host_out, c->pass_timing, sizeof(long long) * 2 * PK_TIMING_SLOTS, cudaMemcpyDeviceToHost);
}
#endif
