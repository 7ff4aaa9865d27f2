// Decode passes of a small fp32 model as one launch of one thread-block cluster.
//
// A pass of such a model is a chain of short steps (QKV, attention, O, gate+up, down; head and pick), each of which needs
// all outputs of the one before.  As launches they cost 3-5 us a step, whatever they compute; between the blocks of a full
// grid a barrier through L2 costs 1.2-2 us.  Sixteen SMs of one cluster hand the outputs over through distributed shared
// memory in a fraction of that, and stream the weights from L2 at 16 x 64 bytes a cycle: a layer of the 4-layer test shape
// (hidden 256, 3.1 MB) takes 1.7 us of streaming.  So the form is for models whose layers are small.
//
//  * Every block holds all activations.  It multiplies an equal cut of each matrix's rows and sends every output to all
//    blocks (st.async, which counts its bytes on the receiver's barrier): one trip between two steps, no fence, no
//    barrier of the cluster inside a pass.
//  * Weights do not depend on activations: every thread fetches the 16-byte parts it will multiply, in the order it will
//    need them, through a private ring in shared memory (cp.async; only the thread itself reads them, so nothing but its own
//    wait is needed), across steps, layers and passes.  (A warp of its own that fills a ring with bulk copies takes the copies'
//    instructions off the multiplying warps, but the blocks then wait 1100 instead of 400 cycles for one another's outputs:
//    8 cycles of one sequence 1.10 ms against 0.95.)
//  * The passes of a cycle are one launch: the first may be a full one (R rows per sequence through the lower layers), the
//    others are short.  The picked token never leaves the cluster between them.
//  * A buffer is overwritten at the earliest by outputs that another block could only compute from this block's outputs of
//    the step that read it, so every barrier has one phase per layer and no buffer needs a second copy.  A barrier says
//    nothing about this block's other warps (a block's own slices may be complete by one warp's outputs): what a block writes
//    for itself, the attention's merged rows, goes where no warp reads since the last __syncthreads.
//  * What a step costs is the length of a warp's chain of instructions: 8 warps (two to a scheduler), shares without
//    remainders (small_pass_fits), index arithmetic once per launch.  With 16 warps and
//    general shares a step took 4500 cycles.
//  * Measured, cycles of the SM clock in a layer of one row (16 to 100 keys): QKV 1550, norms and rotary embedding 500, keys 1900,
//    the slices together and out 600, in 700, merge 1200, O 950, gate+up 4200, down 1500, waits for outputs 2000.  A warp issues
//    one instruction in 8 to 11 cycles (a quarter of the issue slots); three gate+up batches side by side, sixteen warps,
//    products taken in pairs, or the keys requested a layer ahead did not shorten the chain.
// Arithmetic: fp32 FMAs, as the kernels of one launch per step.  Seven cycles of three tokens and three passes with given
// tokens of the 4-layer test shape, context 32 to 2000: 1.68 ms with a launch per step, 0.89 so.
#pragma once

#include <algorithm>

#include "pass_common.cuh"

namespace dmtd {

constexpr int SP_CTAS = 16, SP_WARPS = 8, SP_THREADS = SP_WARPS * 32, SP_SHARES = SP_CTAS * SP_WARPS;
constexpr int SP_D = 64;                                       // head_dim
constexpr int SP_DEPTH = 8, SP_UNITS = 4;                      // ring: groups in flight, 16-byte parts of a thread in a group
constexpr int SP_RING_BYTES = SP_DEPTH * SP_UNITS * 16 * SP_THREADS;
constexpr int SP_MAX_ROWS = 8;                                 // activation rows, and query rows of a kv head
constexpr int SP_MAX_POSITIONS = 16;                           // positions (rows of the rotary table) of a launch
constexpr int SP_MAX_LAYERS = 24;

struct SmallLayer {
  const float *qkv, *o, *gu, *down, *w_in, *w_post, *w_qn, *w_kn;
  float *kc, *vc;                                              // [sequence][kv head][max_seq][64]
};

// Shared memory of a block behind the ring, offsets in floats.
struct SmallMap {
  int xs;          // residual rows [M][H]
  int qkv;         // [M][(nq + 2 nkv) 64]
  int merged;      // the attention's merged rows [M][nq 64], where qkv was
  int wide;        // gated rows [M][I]; before that the attention's warps' outputs
  int part_o;      // partial results of the key slices [row][head][slice][64]
  int part_ml;     // ... their (max, sum) pairs
  int q;           // query rows [8][64], normalised, rotated, scaled
  int new_kv;      // K, then V rows of the pass for this block's kv head [2][8][64]
  int red;         // the attention warps' max and sum [2][8 warps][8]
  int gains;       // w_in | w_post of every layer, final norm
  int head_gains;  // w_qn | w_kn of every layer
  int rope;        // [positions][32] of (cos, sin)
  int total;
};

struct SmallParams {
  SmallLayer layers[SP_MAX_LAYERS];                            // (as a parameter: a pointer is a trip to memory less, every step)
  const float *embed, *w_final;
  const double *inv_freq;
  int n_layers, lo, B, R;                                      // R: rows per sequence of a full first pass
  int n_passes;
  int full;                                                    // the first pass is a full one (counters) ...
  int lower;                                                   // ... and there are lower layers for it to run
  int H, I, nq, nkv, vocab, max_seq;
  int ns;                                                      // key slices of a kv head
  float eps;
  int write_token;
  int *tokens;
  DevState *st;
  float *out_logits;                                           // [pass][B][vocab], or null
  int *out_argmax;                                             // [pass][B], or null
  int *out_tokens;                                             // [B][tau], a pass's token in column `pass`, or null
  int tau;
  SampleParams sample;
  SmallMap map;
  int *error;
  long long wait_limit;
};

enum { SP_BAR_QKV = 0, SP_BAR_PART, SP_BAR_O, SP_BAR_GATED, SP_BAR_DOWN, SP_BAR_PICK, SP_BARS };
enum { SP_QKV = 0, SP_O, SP_GU, SP_DOWN, SP_HEAD };

// A warp's share of a matrix, as its producer walks it: groups of four parts of a thread, one 128-value piece of four rows
// or two pieces of two rows.
struct __align__(16) SmallWalk {
  size_t first;              // bytes from the matrix to the share (a head may be larger than 4 GiB)
  uint32_t o1, o2, o3;       // from a group's first part to the others
  uint32_t step, skip;       // to the next group of a batch of rows; from the end of a batch to the next one
  int pieces, batches;       // groups of a batch; batches
};
struct SmallFixed {                                            // first bytes of the shared memory
  uint64_t bars[SP_BARS];
  const float *w[SP_MAX_LAYERS][4];                            // matrices
  SmallWalk walk[5][SP_WARPS];
  int gave_up;
  int tok[SP_MAX_ROWS];
  uint64_t pick[SP_MAX_ROWS][SP_CTAS];                         // (value, index) of every block
  float pick_val[SP_WARPS][SP_MAX_ROWS];
  int pick_idx[SP_WARPS][SP_MAX_ROWS];
};
constexpr int SP_FIXED_BYTES = (int)((sizeof(SmallFixed) + 127) / 128 * 128);

// Shapes whose matrices are cut into whole batches of rows for the 128 warps: four rows of QKV, two of O and down, two
// gate-up pairs, four rows of the head; k in whole 256-value pieces.
inline bool small_pass_fits(int H, int I, int nq, int nkv, int vocab) {
  return H % (2 * SP_SHARES) == 0 && I % (2 * SP_SHARES) == 0 && (nq + 2 * nkv) * SP_D % (4 * SP_SHARES) == 0 && nq * SP_D % 256 == 0 && vocab % 4 == 0;
}
// us that a cycle of this form gains on a launch per step (captured), for B sequences; whole: the full pass runs so, too.
// Sixteen SMs stream the weights where the other form has 148, so the form pays by the launches of small layers and
// loses by bytes and by rows of the head, the more so the more activation rows each of them is multiplied with.  The
// figures are fitted to cycles of 25 fp32 shapes (hidden 256 to 1024, layers of 3 to 50 MB, 1 to 12 of them, vocabularies of
// 1024 to 151936) at 1 to 8 rows; one launch / captured steps, us: hidden 256, 4 layers of 3.1 MB, 3 passes, vocabulary 1024 97
// / 163, 16384 145 / 182, 32768 195 / 198, 65536 306 / 241, 151936 576 / 382; two sequences 131 / 185, 206 / 202, 289 / 227, 474 /
// 271, 913 / 412; 4 layers, 1 pass, vocabulary 1024, layers of 12.6 MB (hidden 512) 69 / 85, four sequences 119 / 119; of 50 MB
// (hidden 1024) 166 / 175.  Where only the short passes run so, changing over costs a cycle some 18 us: layers of 12.6 MB, two
// sequences, 251 / 233, of 31 MB 418 / 349.
inline float small_pass_gain(int H, int I, int nq, int nkv, int vocab, int n_layers, int L_d, int B, int tau, bool whole) {
  struct Rows { float pass, layer, layer_mb, head_rows; };       // a pass's ends, a layer; less per MB of a layer, per 1000 rows of the head
  const auto rows = [](int m) { return m == 1 ? Rows{8.f, 5.4f, 0.09f, 0.6f} : m <= 4 ? Rows{5.f, 6.2f, 0.5f, 1.1f} : Rows{4.f, 8.f, 0.9f, 1.5f}; };
  const float mb = 4e-6f * H * ((2.f * nq + 2 * nkv) * SP_D + 3.f * I);
  const auto layers = [&](int n, const Rows &r) { return n * (r.layer - r.layer_mb * mb); };
  const Rows one = rows(B);
  const float top = one.pass + layers(L_d, one) - one.head_rows * 1e-3f * vocab;         // what every pass has
  return tau * top + (whole ? layers(n_layers - L_d, rows(B * tau)) : -top - 18.f);
}
// Store into a block's shared memory (cluster_address); its bytes are counted on the barrier there.
__device__ __forceinline__ void sp_send8(uint32_t dst, uint64_t v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void sp_send2(uint32_t dst, float a, float b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1,%2}, [%3];" ::"r"(dst), "r"(__float_as_uint(a)),
               "r"(__float_as_uint(b)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void sp_send4(uint32_t dst, float4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(dst),
               "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)), "r"(bar)
               : "memory");
}

// Sums over the lanes of a warp of NB sets of V values (a power of two up to 32): lane i gets, as v[..][0], the sum of value
// i >> (5 - log2 V) of each set; the sums of the N values n beside them.  Step by step side by side: each set alone is a
// chain of five exchanges.
template <int NB, int V, int N>
__device__ __forceinline__ void sp_reduce(float (&v)[NB][V], float (&n)[N], bool with_n) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int off = 16 >> step, s = V >> (step + 1), t = N >> (step + 1);
    const bool up = lane & off;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (s >= 1) {
#pragma unroll
        for (int i = 0; i < V / 2; ++i)
          if (i < s) {
            const float got = __shfl_xor_sync(0xffffffffu, up ? v[b][i] : v[b][i + s], off);
            v[b][i] = (up ? v[b][i + s] : v[b][i]) + got;
          }
      } else {
        v[b][0] += __shfl_xor_sync(0xffffffffu, v[b][0], off);
      }
    }
    if (with_n) {
      if (t >= 1) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i)
          if (i < t) {
            const float got = __shfl_xor_sync(0xffffffffu, up ? n[i] : n[i + t], off);
            n[i] = (up ? n[i + t] : n[i]) + got;
          }
      } else {
        n[0] += __shfl_xor_sync(0xffffffffu, n[0], off);
      }
    }
  }
}

extern __shared__ __align__(1024) unsigned char sp_smem[];

__device__ __forceinline__ SmallFixed &sp_fixed() { return *reinterpret_cast<SmallFixed *>(sp_smem); }
__device__ __forceinline__ float *sp_floats() { return reinterpret_cast<float *>(sp_smem + SP_FIXED_BYTES + SP_RING_BYTES); }

// Bounded wait; after one has run out the others return at once.
__device__ __forceinline__ void sp_wait_bar(const SmallParams &P, uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return;
  volatile int *const gave_up = &sp_fixed().gave_up;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*gave_up || clock64() - t0 > P.wait_limit) {
      *gave_up = 1;
      atomicMax(P.error, PK_ERR_COPY_WAIT);
      return;
    }
  }
}
// Wait for the next phase of a barrier that `bytes` of outputs complete (thread 0 announces them).
__device__ __forceinline__ void sp_wait(const SmallParams &P, int which, uint32_t &phases, uint32_t bytes) {
  const uint32_t bar = smem_u32(sp_smem) + 8 * which, parity = phases >> which & 1u;
  phases ^= 1u << which;
  if (threadIdx.x == 0) mbar_expect_tx(bar, bytes);
  sp_wait_bar(P, bar, parity);
}

// The rows of a head share, a multiple of four: all of them for a warp before the vocabulary's end.
__host__ __device__ __forceinline__ int sp_head_share(int vocab) { return ((vocab + SP_SHARES - 1) / SP_SHARES + 3) & ~3; }
__host__ __device__ __forceinline__ SmallWalk sp_walk(const SmallParams &P, int kind, int share) {
  int K = P.H, first, n;     // values of a row; first row, rows (pairs for gate+up)
  if (kind == SP_HEAD) {
    const int per = sp_head_share(P.vocab);
    first = share * per;
    n = first >= P.vocab ? 0 : P.vocab - first < per ? P.vocab - first : per;
  } else {
    n = (kind == SP_QKV ? (P.nq + 2 * P.nkv) * SP_D : kind == SP_GU ? P.I : P.H) / SP_SHARES;
    if (kind == SP_O) K = P.nq * SP_D;
    if (kind == SP_DOWN) K = P.I;
    first = share * n;
  }
  const uint32_t row = K * 4, up = (uint32_t)P.I * row;
  const size_t at = (size_t)first * row;
  if (kind == SP_O || kind == SP_DOWN) return SmallWalk{at, row, 512, row + 512, 1024, row, K / 256, n / 2};
  if (kind == SP_GU) return SmallWalk{at, up, row, up + row, 512, row, K / 128, n / 2};
  return SmallWalk{at, row, 2 * row, 3 * row, 512, 3 * row, K / 128, n / 4};
}

// The producer's position in the warp's weights of a launch.
struct SmallCursor {
  const char *p;             // part of this lane of the group's first row and piece
  SmallWalk w;               // w.batches: left, the one at hand included
  int left;                  // groups of the batch at hand
  int layer, kind, pass;     // of the matrix at hand; pass == n_passes: done
  uint32_t dst;              // shared address of this thread's slot
};
__device__ __forceinline__ void sp_cursor_matrix(const SmallParams &P, SmallCursor &cur) {
  const SmallFixed &F = sp_fixed();
  cur.w = F.walk[cur.kind][threadIdx.x >> 5];
  cur.p = reinterpret_cast<const char *>(cur.kind == SP_HEAD ? P.embed : F.w[cur.layer][cur.kind]) + cur.w.first + (threadIdx.x & 31) * 16;
  cur.left = cur.w.pieces;
}
__device__ __forceinline__ void sp_issue(const SmallParams &P, SmallCursor &cur) {
  if (cur.pass < P.n_passes) {
    auto copy = [&](int u, uint32_t off) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(cur.dst + u * SP_THREADS * 16), "l"(cur.p + off) : "memory");
    };
    copy(0, 0);
    copy(1, cur.w.o1);
    copy(2, cur.w.o2);
    copy(3, cur.w.o3);
    cur.p += cur.w.step;
    if (--cur.left == 0) {
      cur.left = cur.w.pieces;
      cur.p += cur.w.skip;
      if (--cur.w.batches == 0) {
        do {                                                              // (the last warps may have no rows of the head)
          if (cur.kind == SP_HEAD) {
            cur.layer = P.lo; cur.kind = SP_QKV;
            if (++cur.pass == P.n_passes) break;
          } else if (cur.kind == SP_DOWN) {
            cur.kind = ++cur.layer == P.n_layers ? SP_HEAD : SP_QKV;
          } else {
            ++cur.kind;
          }
          sp_cursor_matrix(P, cur);
        } while (cur.w.batches == 0);
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");                    // an empty group past the end keeps the counts uniform
}
__device__ __forceinline__ void sp_advance(SmallCursor &cur) {
  cur.dst += SP_UNITS * SP_THREADS * 16;
  if (cur.dst >= smem_u32(sp_smem) + SP_FIXED_BYTES + SP_RING_BYTES) cur.dst -= SP_RING_BYTES;
}

__device__ __forceinline__ void sp_fma4(float2 &a, const float4 &x, const float4 &y) {
  fma_f32x2(a, make_float2(x.x, x.y), make_float2(y.x, y.y));
  fma_f32x2(a, make_float2(x.z, x.w), make_float2(y.z, y.w));
}

// The activation rows of a step: row m at x + m * ld; NORM steps normalise them (RMSNorm, 1 / rms goes to the product).
struct SmallX {
  const float *x;
  int ld, rows;
  const float *gain;
};

// One batch of BATCH weight rows against MR activation rows: lane i gets the sum of (weight row v % BATCH, activation row
// v / BATCH), v = i >> (5 - log2(BATCH * MR)).  NORM: `first` says that scale, 1 / rms of the lane's activation row, is still
// to be worked out.
template <int BATCH, int MR, bool NORM>
__device__ __forceinline__ float sp_multiply(const SmallParams &P, SmallCursor &cur, int K, const SmallX &X, bool first, float &scale) {
  constexpr int PIECES = SP_UNITS / BATCH, V = BATCH * MR;
  const int lane = threadIdx.x & 31;
  const float *row[MR];
#pragma unroll
  for (int m = 0; m < MR; ++m) row[m] = X.x + min(m, X.rows - 1) * X.ld + lane * 4;
  const float *gain = X.gain + lane * 4;
  float2 acc[V], ss[MR];
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 0; m < MR; ++m) ss[m] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int k = 0; k < K; k += PIECES * 128) {
    asm volatile("cp.async.wait_group %0;" ::"n"(SP_DEPTH - 1) : "memory");
    float4 w[SP_UNITS];
#pragma unroll
    for (int u = 0; u < SP_UNITS; ++u) {
      const uint4 v = lds128(cur.dst + u * SP_THREADS * 16);              // the oldest group lies where the next one goes
      w[u] = make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
    }
#pragma unroll
    for (int p = 0; p < PIECES; ++p) {
      float4 g;
      if (NORM) g = *reinterpret_cast<const float4 *>(gain + k + p * 128);
#pragma unroll
      for (int m = 0; m < MR; ++m) {
        float4 x = *reinterpret_cast<const float4 *>(row[m] + k + p * 128);
        if (NORM) {
          sp_fma4(ss[m], x, x);
          x.x *= g.x; x.y *= g.y; x.z *= g.z; x.w *= g.w;
        }
#pragma unroll
        for (int r = 0; r < BATCH; ++r) sp_fma4(acc[m * BATCH + r], w[p * BATCH + r], x);
      }
    }
    sp_issue(P, cur);
    sp_advance(cur);
  }
  float v[1][V], n[MR];
#pragma unroll
  for (int i = 0; i < V; ++i) v[0][i] = acc[i].x + acc[i].y;
#pragma unroll
  for (int m = 0; m < MR; ++m) n[m] = ss[m].x + ss[m].y;
  if (NORM && first) {
    sp_reduce<1, V, MR>(v, n, true);
    const float s = rsqrtf(n[0] * (1.f / (float)K) + P.eps);               // lane i: activation row i * MR / 32
    scale = MR == 1 ? s : __shfl_sync(0xffffffffu, s, (lane * V / 32) / BATCH * (32 / MR));
  } else {
    sp_reduce<1, V, MR>(v, n, false);
  }
  return NORM ? v[0][0] * scale : v[0][0];
}

// The outputs of a batch to all blocks: every lane sends to block lane % 16, the two halves of the warp take the activation
// rows in turn.  at, ld: where row 0's outputs lie; rbase, rbar: the block's buffers and the barrier that counts them.
template <int KIND, int MR>
__device__ __forceinline__ void sp_batch(const SmallParams &P, SmallCursor &cur, int K, const SmallX &X, bool first, float &scale, int M,
                                         int at, int ld, uint32_t rbase, uint32_t rbar) {
  constexpr int BATCH = KIND == SP_O || KIND == SP_DOWN ? 2 : 4, COPIES = 32 / (BATCH * MR), OUT = KIND == SP_QKV ? 4 : 2;
  float v = sp_multiply<BATCH, MR, BATCH == 4>(P, cur, K, X, first, scale);
  const int half = (threadIdx.x & 31) >> 4;
  if (KIND == SP_GU) {
    // rows come in turn: gate, up.  (Both lanes of a pair work the gate out.)
    const bool up = (threadIdx.x & 31) / COPIES & 1;
    const float other = __shfl_xor_sync(0xffffffffu, v, COPIES), g = up ? other : v, u = up ? v : other;
    v = g / (1.f + expf(-g)) * u;
  }
#pragma unroll
  for (int i = 0; i < (MR + 1) / 2; ++i) {
    const int m = MR == 1 ? 0 : 2 * i + half, to = at + m * ld;
    float o[OUT];
#pragma unroll
    for (int r = 0; r < OUT; ++r) o[r] = __shfl_sync(0xffffffffu, v, (m * BATCH + r * (BATCH / OUT)) * COPIES);
    if (m >= M || (MR == 1 && half)) continue;
    if (KIND == SP_QKV) {
      sp_send4(rbase + to * 4, make_float4(o[0], o[1], o[2 % OUT], o[3 % OUT]), rbar);
    } else if (KIND == SP_GU) {
      sp_send2(rbase + to * 4, o[0], o[1], rbar);
    } else {                                                               // into the residual rows
      const float2 old = *reinterpret_cast<const float2 *>(sp_floats() + to);
      sp_send2(rbase + to * 4, old.x + o[0], old.y + o[1], rbar);
    }
  }
}

// The head: logits out, and the lane's best so far.
template <int MR>
__device__ __forceinline__ void sp_head(const SmallParams &P, SmallCursor &cur, const SmallX &X, int pass, int position, float &best, int &bi) {
  constexpr int COPIES = 32 / (4 * MR);
  const int lane = threadIdx.x & 31, idx = lane / COPIES, m = idx >> 2;
  const int per = sp_head_share(P.vocab), n0 = (blockIdx.x * SP_WARPS + (threadIdx.x >> 5)) * per, end = min(P.vocab, n0 + per);
  float scale = 1.f;
#pragma unroll 1
  for (int n = n0; n < end; n += 4) {
    const float v = sp_multiply<4, MR, true>(P, cur, P.H, X, n == n0, scale);
    const int i = n + (idx & 3);
    if (m < P.B) {
      if (P.out_logits && lane % COPIES == 0) P.out_logits[((size_t)pass * P.B + m) * P.vocab + i] = v;
      const float c = pick_value(v, i, position, m, P.sample);
      if (c > best) { best = c; bi = i; }                                  // indices rise within a lane
    }
    __syncwarp();
  }
}

// What a block's and a thread's part of the attention of R rows per sequence is: the same for every layer of a kind.
struct SmallItem {
  int R, M, pos0, rope0;     // rows per sequence, of all; position of the first, its row of the rotary table
  int j0, j1;                // cached keys of the block's slice
  int q;                     // qkv: the warp's query row (or -1), its rotary row
  int q_rope;
  int item, n_items;         // the thread's (query row, 4 dimensions) when the warps' results are put together: row * 16 + part
  int to, n_to;              // ... the blocks it sends them to: to, to + 1, ..
  int slot;                  // ... and where they lie there
};
__device__ __forceinline__ SmallItem sp_item(const SmallParams &P, int R, int pos0, int rope0, int b, int kvh, int slice) {
  const int G = P.nq / P.nkv, nQ = R * G, warp = threadIdx.x >> 5;
  SmallItem t;
  t.R = R; t.M = P.B * R; t.pos0 = pos0; t.rope0 = rope0;
  t.j0 = pos0 * slice / P.ns; t.j1 = pos0 * (slice + 1) / P.ns;
  t.q = warp < nQ ? (b * R + warp / G) * (P.nq + 2 * P.nkv) * SP_D + (kvh * G + warp % G) * SP_D : -1;
  t.q_rope = (rope0 + warp / G) * (SP_D / 2);
  // nQ * 16 threads hold a result each; as many sets of them as there is room for share the blocks
  t.n_items = nQ * (SP_D / 4);
  const int sets = nQ == 1 ? 16 : nQ == 2 ? 8 : nQ <= 4 ? 4 : 2, set = threadIdx.x / t.n_items;
  t.item = threadIdx.x - set * t.n_items;
  t.n_to = set < sets ? SP_CTAS / sets : 0;
  t.to = set * (SP_CTAS / sets);
  const int q = t.item >> 4;
  t.slot = ((b * R + q / G) * P.nq + kvh * G + q % G) * P.ns + slice;
  return t;
}

// Eight keys of the cache by a warp: four lanes to a key, dimensions 8 * (lane % 4) .. + 7 and 32 further on; of the values
// dimensions 2 lane and 2 lane + 1.
struct SmallTile {
  float4 k[4];
  float2 v[8];
};
__device__ __forceinline__ void sp_load_tile(SmallTile &t, const float *kc, const float *vc, int jb, int j1) {
  const int lane = threadIdx.x & 31;
  const float4 *k = reinterpret_cast<const float4 *>(kc + (size_t)min(jb + (lane >> 2), j1 - 1) * SP_D + (lane & 3) * 8);
  t.k[0] = __ldcg(k); t.k[1] = __ldcg(k + 1); t.k[2] = __ldcg(k + 8); t.k[3] = __ldcg(k + 9);
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) t.v[jj] = __ldcg(reinterpret_cast<const float2 *>(vc + (size_t)min(jb + jj, j1 - 1) * SP_D) + lane);
}

// Steps a3 and a4: a block takes a kv head of a sequence and a slice of its keys; the partial results of the slices go to
// every block.  Then their merge, over the projection's rows.  The last slice takes the pass's own rows.
__device__ __forceinline__ void sp_attention(const SmallParams &P, uint32_t &phases, int layer, const SmallItem &T, int b, int kvh, int slice) {
  constexpr int D = SP_D, D4 = D / 4;
  float *const f = sp_floats();
  const SmallMap &map = P.map;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ldq = (P.nq + 2 * P.nkv) * D, ns = P.ns, R = T.R, M = T.M, G = P.nq / P.nkv, nQ = T.n_items >> 4;
  const uint32_t bars = smem_u32(sp_smem), base = smem_u32(f);
  float *const q_s = f + map.q, *const new_k = f + map.new_kv, *const new_v = new_k + SP_MAX_ROWS * D;
  float *const o_s = f + map.wide, *const red_m = f + map.red, *const red_l = red_m + SP_WARPS * SP_MAX_ROWS;
  if (b < P.B) {
    const bool has_new = slice == ns - 1;
    const int j0 = T.j0, j1 = T.j1, n_cached = (j1 - j0 + 7) >> 3, n_tiles = n_cached + (has_new ? 1 : 0), n_warps = min(SP_WARPS, n_tiles);
    const size_t head = ((size_t)b * P.nkv + kvh) * P.max_seq * D;
    float *const kc = P.layers[layer].kc + head, *const vc = P.layers[layer].vc + head;
    SmallTile t;
    if (warp < n_cached) sp_load_tile(t, kc, vc, j0 + warp * 8, j1);       // older than this pass: before its projection is waited for
    // this warp's query row; the last warps: K and V of the new positions
    const float *const gains = f + map.head_gains + layer * 2 * D;
    const float2 *const rope = reinterpret_cast<const float2 *>(f + map.rope) + lane;
    const float gq0 = gains[lane], gq1 = gains[lane + 32], gk0 = gains[D + lane], gk1 = gains[D + lane + 32];
    const int r_new = SP_WARPS - 1 - warp;
    const float2 csq = rope[T.q >= 0 ? T.q_rope : 0], csk = rope[(T.rope0 + min(r_new, R - 1)) * (D / 2)];
    sp_wait(P, SP_BAR_QKV, phases, (uint32_t)(M * ldq * 4));
    auto norm_rope = [&](const float *src, float g0, float g1, float2 cs, float &lo, float &hi) {
      lo = src[lane]; hi = src[lane + 32];
      const float inv = rsqrtf(warp_sum(lo * lo + hi * hi) * (1.f / D) + P.eps);
      const float x = lo * inv * g0, y = hi * inv * g1;
      lo = x * cs.x - y * cs.y;
      hi = y * cs.x + x * cs.y;
    };
    if (T.q >= 0) {
      float lo, hi;
      norm_rope(f + map.qkv + T.q, gq0, gq1, csq, lo, hi);
      q_s[warp * D + lane] = lo * 0.125f;                         // 1 / sqrt(64)
      q_s[warp * D + lane + 32] = hi * 0.125f;
    }
    if (has_new && r_new < R) {
      const float *src = f + map.qkv + (b * R + r_new) * ldq + (P.nq + kvh) * D;
      float lo, hi;
      norm_rope(src, gk0, gk1, csk, lo, hi);
      const float v0 = src[P.nkv * D + lane], v1 = src[P.nkv * D + lane + 32];
      new_k[r_new * D + lane] = lo; new_k[r_new * D + lane + 32] = hi;
      new_v[r_new * D + lane] = v0; new_v[r_new * D + lane + 32] = v1;
      float *ck = kc + (size_t)(T.pos0 + r_new) * D, *cv = vc + (size_t)(T.pos0 + r_new) * D;
      ck[lane] = lo; ck[lane + 32] = hi;
      cv[lane] = v0; cv[lane + 32] = v1;
    }
    __syncthreads();
    if (warp < n_warps) {
      float m_run[SP_MAX_ROWS], l_run[SP_MAX_ROWS];               // l_run: of this lane's keys
      float2 o[SP_MAX_ROWS];
#pragma unroll
      for (int q = 0; q < SP_MAX_ROWS; ++q) {
        m_run[q] = -INFINITY; l_run[q] = 0.f;
        o[q] = make_float2(0.f, 0.f);
      }
#pragma unroll 1
      for (int tile = warp; tile < n_tiles; tile += SP_WARPS) {
        const bool is_new = tile == n_cached;
        const int jt = lane >> 2, n_here = is_new ? R : min(8, j1 - j0 - tile * 8);
        if (is_new) {
          const float4 *k = reinterpret_cast<const float4 *>(new_k + min(jt, R - 1) * D + (lane & 3) * 8);
          t.k[0] = k[0]; t.k[1] = k[1]; t.k[2] = k[8]; t.k[3] = k[9];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) t.v[jj] = reinterpret_cast<const float2 *>(new_v + min(jj, R - 1) * D)[lane];
        }
        const SmallTile now = t;
        if (tile + SP_WARPS < n_cached) sp_load_tile(t, kc, vc, j0 + (tile + SP_WARPS) * 8, j1);
        // two query rows side by side: each is one chain of dependent instructions.  (An odd last row has an unused partner.)
#pragma unroll
        for (int q0 = 0; q0 < SP_MAX_ROWS; q0 += 2) {
          if (q0 >= nQ) break;
          float s[2], mx[2], p[2], corr[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float4 *qr = reinterpret_cast<const float4 *>(q_s + (q0 + e) * D + (lane & 3) * 8);
            float2 c2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
            for (int c = 0; c < 4; ++c) sp_fma4(c2[c & 1], now.k[c], qr[(c >> 1) * 8 + (c & 1)]);
            s[e] = (c2[0].x + c2[1].x) + (c2[0].y + c2[1].y);
          }
#pragma unroll
          for (int x = 1; x < 4; x <<= 1)
#pragma unroll
            for (int e = 0; e < 2; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], x);
          bool ok[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            ok[e] = jt < n_here && (!is_new || jt * G <= q0 + e);          // a pass's own keys: up to the row's position
            mx[e] = ok[e] ? s[e] : -INFINITY;
          }
#pragma unroll
          for (int x = 4; x < 32; x <<= 1)
#pragma unroll
            for (int e = 0; e < 2; ++e) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], x));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int q = q0 + e;
            const float m_new = fmaxf(m_run[q], mx[e]);                    // the first key of a tile is seen by every row
            corr[e] = __expf(m_run[q] - m_new);
            p[e] = ok[e] ? __expf(s[e] - m_new) : 0.f;
            l_run[q] = l_run[q] * corr[e] + p[e];
            m_run[q] = m_new;
            o[q].x *= corr[e]; o[q].y *= corr[e];
          }
#pragma unroll
          for (int jj = 0; jj < 8; ++jj)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float pj = __shfl_sync(0xffffffffu, p[e], jj * 4);
              fma_f32x2(o[q0 + e], make_float2(pj, pj), now.v[jj]);
            }
        }
      }
#pragma unroll
      for (int x = 4; x < 32; x <<= 1)
#pragma unroll
        for (int q = 0; q < SP_MAX_ROWS; ++q)
          if (q < nQ) l_run[q] += __shfl_xor_sync(0xffffffffu, l_run[q], x);
#pragma unroll
      for (int q = 0; q < SP_MAX_ROWS; ++q) {
        if (q >= nQ) break;
        if (lane == 0) { red_m[q * SP_WARPS + warp] = m_run[q]; red_l[q * SP_WARPS + warp] = l_run[q]; }
        reinterpret_cast<float2 *>(o_s + (q * SP_WARPS + warp) * D)[lane] = o[q];
      }
    }
    __syncthreads();
    // the warps' results together, and to all blocks; a slice without keys (short contexts) sends sum 0
    if (T.n_to > 0) {
      const int q = T.item >> 4, d4 = T.item & 15;
      const float *rm = red_m + q * SP_WARPS, *rl = red_l + q * SP_WARPS;
      const float4 *os = reinterpret_cast<const float4 *>(o_s + q * SP_WARPS * D) + d4;
      float m = -INFINITY, l = 0.f;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      if (n_warps == 1) {
        m = rm[0]; l = rl[0]; o = os[0];
      } else {
        float mw[SP_WARPS];
#pragma unroll
        for (int w = 0; w < SP_WARPS; ++w) {
          mw[w] = w < n_warps ? rm[w] : -INFINITY;
          m = fmaxf(m, mw[w]);
        }
#pragma unroll
        for (int w = 0; w < SP_WARPS; ++w)
          if (w < n_warps) {
            const float fw = __expf(mw[w] - m);
            const float4 v = os[w * D4];
            l += fw * rl[w];
            o.x += fw * v.x; o.y += fw * v.y; o.z += fw * v.z; o.w += fw * v.w;
          }
      }
      const uint32_t dst = base + (map.part_o + T.slot * D + d4 * 4) * 4, dst_ml = base + (map.part_ml + T.slot * 2) * 4;
#pragma unroll 2
      for (int c = T.to; c < T.to + T.n_to; ++c) {
        const uint32_t bar = cluster_address(bars + 8 * SP_BAR_PART, c);
        sp_send4(cluster_address(dst, c), o, bar);
        if (d4 == c) sp_send2(cluster_address(dst_ml, c), m, l, bar);              // (every block's pair from another thread)
      }
    }
  } else {
    sp_wait(P, SP_BAR_QKV, phases, (uint32_t)(M * ldq * 4));
  }
  // the merge
  sp_wait(P, SP_BAR_PART, phases, (uint32_t)(M * P.nq * ns * (D + 2) * 4));
  float4 *const att = reinterpret_cast<float4 *>(f + map.merged);         // (not over the warps' outputs: other warps may still read them)
  for (int i = threadIdx.x; i < M * P.nq * D4; i += SP_THREADS) {
    const int rh = i / D4, d4 = i % D4;
    const float2 *ml = reinterpret_cast<const float2 *>(f + map.part_ml) + rh * ns;
    const float4 *po = reinterpret_cast<const float4 *>(f + map.part_o) + rh * ns * D4 + d4;
    float m = -INFINITY, l = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int s = 0; s < ns; ++s) m = fmaxf(m, ml[s].y > 0.f ? ml[s].x : -INFINITY);
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
      const float2 u = ml[s];
      const float w = u.y > 0.f ? __expf(u.x - m) : 0.f;
      const float4 v = po[s * D4];
      l += w * u.y;
      o.x += w * v.x; o.y += w * v.y; o.z += w * v.z; o.w += w * v.w;
    }
    const float inv = 1.f / l;
    att[i] = make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
  }
  __syncthreads();
}

// Steps a2 to a7 of one layer.  x_off, x_ld: the residual rows (a8: behind the lower layers of a full pass they are the
// newest row of each sequence).  rbase, rbars: buffers and barriers of the block this lane sends to.
template <int MR>
__device__ __forceinline__ void sp_layer(const SmallParams &P, SmallCursor &cur, uint32_t &phases, int layer, const SmallItem &T, int x_off,
                                         int x_ld, int b, int kvh, int slice, uint32_t rbase, uint32_t rbars) {
  const SmallMap &map = P.map;
  float *const f = sp_floats();
  const int warp = threadIdx.x >> 5, share = blockIdx.x * SP_WARPS + warp, H = P.H, I = P.I, M = T.M, QD = P.nq * SP_D, ldq = QD + 2 * P.nkv * SP_D;
  const int n_qkv = ldq / SP_SHARES, n_h = H / SP_SHARES, n_i = I / SP_SHARES;
  float scale = 1.f;
  SmallX X{f + map.xs + x_off, x_ld, M, f + map.gains + 2 * layer * H};
#pragma unroll 1
  for (int n = 0; n < n_qkv; n += 4)
    sp_batch<SP_QKV, MR>(P, cur, H, X, n == 0, scale, M, map.qkv + share * n_qkv + n, ldq, rbase, rbars + 8 * SP_BAR_QKV);
  sp_attention(P, phases, layer, T, b, kvh, slice);
  const SmallX A{f + map.merged, QD, M, nullptr};
  const int at_h = map.xs + x_off + share * n_h;
#pragma unroll 1
  for (int n = 0; n < n_h; n += 2) sp_batch<SP_O, MR>(P, cur, QD, A, false, scale, M, at_h + n, x_ld, rbase, rbars + 8 * SP_BAR_O);
  sp_wait(P, SP_BAR_O, phases, (uint32_t)(M * H * 4));
  X.gain += H;
#pragma unroll 1
  for (int n = 0; n < n_i; n += 2)
    sp_batch<SP_GU, MR>(P, cur, H, X, n == 0, scale, M, map.wide + share * n_i + n, I, rbase, rbars + 8 * SP_BAR_GATED);
  sp_wait(P, SP_BAR_GATED, phases, (uint32_t)(M * I * 4));
  const SmallX W{f + map.wide, I, M, nullptr};
#pragma unroll 1
  for (int n = 0; n < n_h; n += 2) sp_batch<SP_DOWN, MR>(P, cur, I, W, false, scale, M, at_h + n, x_ld, rbase, rbars + 8 * SP_BAR_DOWN);
  sp_wait(P, SP_BAR_DOWN, phases, (uint32_t)(M * H * 4));
}

// x[m][:] = E[token of row m], rows of sequence b at positions pos0 .. pos0 + R - 1; the position of a short pass behind
// another one has its token in F.tok.
__device__ __forceinline__ void sp_embed(const SmallParams &P, int R, int pos0, bool picked) {
  float4 *const xs = reinterpret_cast<float4 *>(sp_floats() + P.map.xs);
  const int h4 = P.H / 4, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int m = warp; m < P.B * R; m += SP_WARPS) {
    int tok = picked ? sp_fixed().tok[m] : __ldcg(P.tokens + (size_t)(m / R) * P.max_seq + pos0 + m % R);
    if (tok < 0 || tok >= P.vocab) {
      atomicMax(P.error, PK_ERR_TOKEN);
      tok = min(max(tok, 0), P.vocab - 1);
    }
    const float4 *e = reinterpret_cast<const float4 *>(P.embed + (size_t)tok * P.H);
#pragma unroll 4
    for (int k4 = lane; k4 < h4; k4 += 32) xs[m * h4 + k4] = __ldg(e + k4);
  }
  __syncthreads();
}

__device__ __forceinline__ void sp_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __launch_bounds__(SP_THREADS, 1) small_pass_kernel(const __grid_constant__ SmallParams P) {
  float *const f = sp_floats();
  const SmallMap &map = P.map;
  SmallFixed &F = sp_fixed();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = blockIdx.x;
  const int H = P.H, B = P.B;
  const uint32_t bars = smem_u32(sp_smem);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) {
    for (int i = 0; i < SP_BARS; ++i) mbar_init(bars + 8 * i, 1);
    F.gave_up = 0;
    fence_mbar_init();
  }
  if (threadIdx.x < 5 * SP_WARPS) F.walk[threadIdx.x / SP_WARPS][threadIdx.x % SP_WARPS] = sp_walk(P, threadIdx.x / SP_WARPS, blockIdx.x * SP_WARPS + threadIdx.x % SP_WARPS);
  if ((int)threadIdx.x < P.n_layers) {
    const SmallLayer &L = P.layers[threadIdx.x];
    F.w[threadIdx.x][SP_QKV] = L.qkv; F.w[threadIdx.x][SP_O] = L.o; F.w[threadIdx.x][SP_GU] = L.gu; F.w[threadIdx.x][SP_DOWN] = L.down;
  }
  __syncthreads();
  // every block's barriers are ready before the first output is sent
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  // weights and gains are as old as the context: requested before the kernel in front is waited for
  SmallCursor cur;
  cur.layer = P.lower ? 0 : P.lo; cur.kind = SP_QKV; cur.pass = 0;
  cur.dst = bars + SP_FIXED_BYTES + threadIdx.x * 16;
  sp_cursor_matrix(P, cur);
#pragma unroll 1
  for (int i = 0; i < SP_DEPTH; ++i) {
    sp_issue(P, cur);
    sp_advance(cur);
  }
  {
    // gains: two floats of every layer's four vectors are on their way before the first is stored
    const int n_vec = 2 * P.n_layers + 1, h4 = H / 4;
#pragma unroll 4
    for (int i = threadIdx.x; i < n_vec * h4; i += SP_THREADS) {
      const int v = i / h4, k = i - v * h4;
      const float *src = v == 2 * P.n_layers ? P.w_final : v & 1 ? P.layers[v >> 1].w_post : P.layers[v >> 1].w_in;
      reinterpret_cast<float4 *>(f + map.gains)[i] = __ldg(reinterpret_cast<const float4 *>(src) + k);
    }
#pragma unroll 4
    for (int i = threadIdx.x; i < P.n_layers * 2 * (SP_D / 4); i += SP_THREADS) {
      const int v = i / (SP_D / 4), k = i % (SP_D / 4);
      reinterpret_cast<float4 *>(f + map.head_gains)[i] = __ldg(reinterpret_cast<const float4 *>(v & 1 ? P.layers[v >> 1].w_kn : P.layers[v >> 1].w_qn) + k);
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lo_len = __ldcg(&P.st->lo_len), n_known = __ldcg(&P.st->n_known);
  const int first_pos = P.lower ? lo_len : n_known - 1;               // rows of the rotary table: first_pos ..
  for (int i = threadIdx.x; i < (n_known - first_pos + P.n_passes - 1) * (SP_D / 2); i += SP_THREADS) {
    double s, c;
    sincos((double)(first_pos + i / (SP_D / 2)) * P.inv_freq[i % (SP_D / 2)], &s, &c);
    reinterpret_cast<float2 *>(f + map.rope)[i] = make_float2((float)c, (float)s);
  }
  // the block's kv head and key slice, and where this lane sends its outputs
  const int item = cta / P.ns, slice = cta - item * P.ns, item_b = item / P.nkv, item_h = item - item_b * P.nkv;
  const uint32_t rbars = cluster_address(bars, lane & 15), rbase = rbars + (uint32_t)(SP_FIXED_BYTES + SP_RING_BYTES);
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");

  uint32_t phases = 0;
#pragma unroll 1
  for (int pass = 0; pass < P.n_passes; ++pass) {
    const bool full = P.lower && pass == 0;
    const int newest = n_known - 1 + pass;
    sp_embed(P, full ? P.R : 1, full ? lo_len : newest, pass > 0 && P.write_token);
    float best = -INFINITY;
    int bi = 0x7fffffff;
    const int l0 = full ? 0 : P.lo;
    SmallItem T = sp_item(P, full ? P.R : 1, full ? lo_len : newest, full ? 0 : newest - first_pos, item_b, item_h, slice);
    int x_off = 0, x_ld = H;
#pragma unroll 1
    for (int l = l0;; ++l) {
      if (l == P.lo && full) {
        // a8: the newest row of each sequence goes on
        T = sp_item(P, 1, newest, newest - first_pos, item_b, item_h, slice);
        x_off = (P.R - 1) * H; x_ld = P.R * H;
      }
      if (l == P.n_layers) break;
      if (T.M == 1) sp_layer<1>(P, cur, phases, l, T, x_off, x_ld, item_b, item_h, slice, rbase, rbars);
      else if (T.M <= 4) sp_layer<4>(P, cur, phases, l, T, x_off, x_ld, item_b, item_h, slice, rbase, rbars);
      else sp_layer<8>(P, cur, phases, l, T, x_off, x_ld, item_b, item_h, slice, rbase, rbars);
    }
    const SmallX X{f + map.xs + x_off, x_ld, B, f + map.gains + 2 * P.n_layers * H};
    if (B == 1) sp_head<1>(P, cur, X, pass, newest + 1, best, bi);
    else if (B <= 4) sp_head<4>(P, cur, X, pass, newest + 1, best, bi);
    else sp_head<8>(P, cur, X, pass, newest + 1, best, bi);
    // a9, a10: the pick.  A lane's best is of one sequence (its quarter, eighth, ... of the warp): over those lanes, over the
    // block's warps, over the blocks, all of which learn the token
    const int lanes = B == 1 ? 32 : B <= 4 ? 8 : 4;                          // lanes of a sequence
    for (int o = lanes / 2; o > 0; o >>= 1) {
      const float v2 = __shfl_xor_sync(0xffffffffu, best, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
      if (v2 > best || (v2 == best && i2 < bi)) { best = v2; bi = i2; }
    }
    if (lane % lanes == 0) { F.pick_val[warp][lane / lanes] = best; F.pick_idx[warp][lane / lanes] = bi; }
    __syncthreads();
    if ((int)threadIdx.x < B * SP_CTAS) {
      const int b = threadIdx.x / SP_CTAS, t = threadIdx.x % SP_CTAS;
      float v = -INFINITY;
      int i = 0x7fffffff;
      for (int w = 0; w < SP_WARPS; ++w) {
        const float v2 = F.pick_val[w][b];
        const int i2 = F.pick_idx[w][b];
        if (v2 > v || (v2 == v && i2 < i)) { v = v2; i = i2; }
      }
      sp_send8(cluster_address(smem_u32(&F.pick[b][cta]), t), (uint64_t)__float_as_uint(v) | (uint64_t)(unsigned)i << 32, cluster_address(bars + 8 * SP_BAR_PICK, t));
    }
    __syncwarp();
    sp_wait(P, SP_BAR_PICK, phases, (uint32_t)(B * SP_CTAS * 8));
    if ((int)threadIdx.x < B) {
      const int b = threadIdx.x;
      float v = -INFINITY;
      int i = 0x7fffffff;
      for (int t = 0; t < SP_CTAS; ++t) {
        const uint64_t p = F.pick[b][t];
        const float v2 = __uint_as_float((unsigned)p);
        const int i2 = (int)(p >> 32);
        if (v2 > v || (v2 == v && i2 < i)) { v = v2; i = i2; }
      }
      if (i == 0x7fffffff) i = 0;
      F.tok[b] = i;
      if (cta == 0) {
        if (P.write_token) P.tokens[(size_t)b * P.max_seq + newest + 1] = i;
        if (P.out_argmax) P.out_argmax[(size_t)pass * B + b] = i;
        if (P.out_tokens) P.out_tokens[(size_t)b * P.tau + pass] = i;
      }
    }
    // this pass's cache rows are there for all blocks before the next pass reads them; at the end no block leaves while
    // another may still write to it
    sp_cluster_sync();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (cta == 0 && threadIdx.x == 0) {
    DevState *st = P.st;
    const int n = n_known + P.n_passes;
    if (P.full) { st->lo_len = n_known; st->cycle += 1; }
    st->up_len = n - 1;
    st->n_known = n;
    st->slot = (st->slot + P.n_passes) % st->tau;
    st->n_emitted += P.n_passes;
    st->newest = n - 1;
  }
}

// The shared memory of a launch of B sequences, R rows each in a full pass.
inline SmallMap small_pass_map(int H, int I, int nq, int nkv, int n_layers, int B, int R) {
  const int M = B * R, ns = std::max(1, SP_CTAS / (B * nkv));
  SmallMap m{};
  int at = 0;
  auto take = [&](int n) { const int r = at; at += (n + 31) / 32 * 32; return r; };
  m.xs = take(M * H);
  m.qkv = m.merged = take(M * (nq + 2 * nkv) * SP_D);
  m.wide = take(std::max(M * I, SP_WARPS * SP_MAX_ROWS * SP_D));
  m.part_o = take(M * nq * ns * SP_D);
  m.part_ml = take(M * nq * ns * 2);
  m.q = take(SP_MAX_ROWS * SP_D);
  m.new_kv = take(2 * SP_MAX_ROWS * SP_D);
  m.red = take(2 * SP_WARPS * SP_MAX_ROWS);
  m.gains = take((2 * n_layers + 1) * H);
  m.head_gains = take(2 * n_layers * SP_D);
  m.rope = take(SP_MAX_POSITIONS * SP_D);
  m.total = at;
  return m;
}
constexpr int SP_SMEM = 227 * 1024;
inline int small_pass_smem(const SmallMap &m) { return SP_FIXED_BYTES + SP_RING_BYTES + m.total * 4; }

}  // namespace dmtd
