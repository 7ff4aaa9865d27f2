// GEMM on the 5th-generation tensor cores (tcgen05, sm_100a) for every projection outside the pass kernel:
// out[m][n] += sum_k W[n][k] act[m][k], one row m up to the rows of a prefill chunk.
//
// Operands are swapped against the usual orientation: weight rows are the M axis of the MMA, activation rows its N
// axis, so that every weight byte is read from HBM once whatever the batch is.  The fp32 activations enter as two
// bf16 parts, hi + lo (error 2^-17 relative), one MMA each.  Two SMs work as a pair (cta_group::2): M = 256 weight
// rows, 128 from each SM's shared memory, and each SM holds one half of the columns, which halves the activation
// traffic per weight byte.
//
// Two forms of a column tile:
//   up to 128 rows (decode):  hi and lo parts are columns of their own (N = 2 x rows): SM 0 of the pair holds the hi
//     columns, SM 1 the lo columns, the epilogue adds them.  Four MMAs per 64-deep k block: one thread issues an MMA
//     every 80 cycles or more whatever N is.
//   more rows (prefill):      hi and lo MMAs add into the same columns (N = rows, up to 256 per tile): a weight block
//     is multiplied with 256 rows x 2 parts for one copy into shared memory, 47 bytes per cycle and SM at full rate.
//
// Both operands are K-major in shared memory in the interleaved (no swizzle) canonical form: 8 rows x 16 bytes per
// core matrix.  The weights are stored in global memory in exactly that order (16 KiB blocks, one per 128-row tile and
// k block), the activations are written that way by the kernels below, so a pipeline stage is a few bulk copies.
//
// Persistent: one pair of blocks per two SMs.  The units of a launch (row-tile pairs x column tiles x k blocks) are cut
// into equal shares whatever the shape is: the row-tile pairs that are not a multiple of the block pairs (all of them,
// where there are fewer) form one line of units cut into equal parts, and a part that ends inside a tile adds its
// partial sums with fp32 reductions (measured at 3.9 TB/s into L2; plain stores 4.8).  The other row-tile pairs are
// dealt out whole: their outputs can be stored (nothing to clear, nothing to add), or, for gate+up, gated and written
// as the down projection's activation blocks by the epilogue.  The accumulators of a tile are read back while the next
// tile is multiplied where tensor memory holds two.
//
// Measured (Qwen3-4B shapes, launches back to back, against the kernel before this one: 128-row sweeps, one MMA-issuing
// block per tile, hi and lo columns always apart): gate+up at 512 rows 139 -> 75 us (1350 TFLOP/s counting both
// parts, at the clock the power cap leaves), QKV 50 -> 29 us; head at 512 rows 541 us (1470 TFLOP/s); decode is bound by
// HBM and by what a launch costs: head at 32 rows 127 us (6.1 TB/s), gate+up at 96 rows 44 -> 27 us, at 8 rows 24 us.
// Gating in gate+up's epilogue instead of clearing, adding and reading 40 MB per 512 rows: prefill of 512 tokens
// 8.8 -> 8.1 ms, of 32 x 1024 tokens 539 -> 469 ms.
//
// Warp roles: warp 0 issues the bulk copies, warp 1 issues the MMAs (first SM of the pair) or passes on to the first
// SM that a stage has landed (second SM), warps 2-9 run the epilogue (each the 32 lanes of its quarter, every second 16 columns).  Every barrier wait is
// bounded and reports through an error word; tensor memory is freed on every path.  Its allocation waits without a limit,
// so it is taken in the order of the stream: a block lets the grids behind it in only once it holds its own.
#pragma once

#include "pass_stream.cuh"

namespace dmtd {

constexpr int TG_EPI_WARPS = 8;              // epilogue warps: two per quarter of the tensor-memory lanes
constexpr int TG_THREADS = 64 + 32 * TG_EPI_WARPS;
constexpr int TG_MAX_STAGES = 8;             // most pipeline stages of a block
constexpr int TG_ROWS = 128;                 // weight rows per tile; a pair of blocks takes two tiles (MMA M = 256)
constexpr int TG_KB = 64;                    // k per unit: four MMAs of K = 16 (per part)
constexpr int TG_WBLOCK = TG_ROWS * TG_KB * 2;      // 16384 bytes
constexpr int TG_SPLIT_ROWS = 128;           // most rows of a column tile with hi and lo in columns of their own
constexpr int TG_TILE_ROWS = 256;            // most rows of a column tile
// k blocks of a pipeline stage.  Up to 128 rows: two; a stage costs its waits, its commit and its copies' issue whatever it
// holds (4 cycles of 32 sequences of the Qwen3-4B shape: 20.26 ms with one, 20.12 with two).  More rows: one, the
// activations of a stage are 32 KiB there.
__host__ __device__ constexpr int tg_stage_units(bool split) { return split ? 2 : 1; }
// Decode launches: the ring's first round, requested before the activations are there, is asked for about as fast as HBM delivers
// it and not at once: two stages (64 KiB an SM, HBM's bandwidth times its latency and a little more), then one every TG_PACE
// cycles.  (32 KiB for 148 SMs take HBM 0.74 us at its copy rate; 1200 cycles are 0.61 us at 1965 MHz and 0.75 us at 1600 MHz.)  With
// 192 KiB an SM outstanding, the few reads between two projections (the norms' and gates' kernels, the keys) waited some 4 us in
// the L2's queues: a projection had its activations 8 us after the end of the one in front.  A cycle of three passes, 4 layers and
// the head, context 512 to 1400, 1965 MHz, 1 / 3 / 16 sequences, us, a stage every 600 cycles 823 / 830 / 895, 1000 805 / 815 / 881, 1200
// 802 / 814 / 882, 1400 805 / 819 / 888, 2000 832 / 847 / 915; all at once 3 to 5 % longer than 1000.  (Asking L2 for the next projection's
// first weights at the end of a launch: 2 % without pacing, nothing beside it.  Activations converted by warps of the GEMM
// instead of kernels in front: as fast at 1 to 3 rows, slower above.)
constexpr int TG_PACE_FREE = 2, TG_PACE = 1200;
constexpr int TG_TAIL_BYTES = 16 * TG_MAX_STAGES + 48;     // barriers, tensor-memory address, flag
// Dynamic shared memory of a block: it has its SM to itself, beside a block of the prefill attention (96 KiB) or another
// GEMM's, which take tensor memory as well.  Two stages of narrow column tiles need less than the lower bound.
constexpr int TG_MAX_SMEM = 226 * 1024, TG_MIN_SMEM = 136 * 1024;
enum { TG_ERR_WAIT = 4 };
enum { TG_ADD = 0, TG_STORE = 1, TG_SWIGLU = 2 };           // tiles dealt out whole: none; stored; gated

// A weight matrix [N][K] as 16 KiB blocks [row tile][k block][k chunk 8][row group 16][row 8][8 values].
struct UmmaMat {
  const uint4 *w;
  int N, K;
  int n_tiles;       // ceil(N / 128), rounded up to even (the last tile may be all zero)
  int n_kb;          // K / 64
};

// How a launch's activation rows are cut into column tiles, and where their 16-byte units (8 values of k of one row,
// hi or lo part) lie: per column tile and k block the two SMs' shares one after the other, each in the canonical
// K-major order [part][k chunk 8][column].
struct ActTiles {
  int n_kb;
  int n_ctiles;      // column tiles
  int tile_rows;     // activation rows per column tile: a multiple of 8 (split parts) or 16
  int split;         // 1: SM 0 holds the hi columns of all rows, SM 1 the lo columns; 0: each SM holds half of the rows, both parts
  __host__ __device__ __forceinline__ size_t units_per_sm() const { return (size_t)tile_rows * 8; }      // of one k block
  // unit of (row m, k block kb, k chunk c): hi part; the lo part lies lo_offset() further
  __device__ __forceinline__ size_t unit(int m, int kb, int c) const {
    const int ct = m / tile_rows, col = m - ct * tile_rows;
    const size_t base = ((size_t)ct * n_kb + kb) * 2 * units_per_sm();
    if (split) return base + c * tile_rows + col;
    const int half = tile_rows / 2, sm = col >= half ? 1 : 0;
    return base + sm * units_per_sm() + c * half + (col - sm * half);
  }
  __device__ __forceinline__ size_t lo_offset() const { return split ? units_per_sm() : units_per_sm() / 2; }
};

inline ActTiles act_tiles_for(int rows, int n_kb) {
  ActTiles t;
  t.n_kb = n_kb;
  t.split = rows <= TG_SPLIT_ROWS;
  t.n_ctiles = t.split ? 1 : (rows + TG_TILE_ROWS - 1) / TG_TILE_ROWS;
  const int per = (rows + t.n_ctiles - 1) / t.n_ctiles, unit = t.split ? 8 : 16;
  t.tile_rows = (per + unit - 1) / unit * unit;
  return t;
}

// A line of units in equal parts: the first `pairs` block pairs take q units each, the first r of them one more.
struct TgLine {
  int q, r, pairs;
  __host__ __device__ __forceinline__ int begin(int pair) const { return pair * q + (pair < r ? pair : r); }
  __host__ __device__ __forceinline__ int size(int pair) const { return pair < pairs ? q + (pair < r ? 1 : 0) : 0; }
  // the pair that holds unit u
  __host__ __device__ __forceinline__ int holder(int u) const { return u < r * (q + 1) ? u / (q + 1) : r + (u - r * (q + 1)) / q; }
};

struct GemmTcParams {
  UmmaMat W;
  const uint4 *act_blocks;
  ActTiles T;
  int rows;                  // activation rows of this launch
  float *out;                // [rows][ldo], added into
  int ldo;
  int rt_whole;              // row-tile pairs dealt out whole, a multiple of the block pairs: the first ones
  int whole_units;           // units of a block pair's whole tiles
  TgLine line;               // the block pairs' parts of the units of the others
  int out_n0;                // first weight row of out's columns (TG_SWIGLU: out holds the remaining row-tile pairs only)
  uint4 *gated;              // TG_SWIGLU: units of the next projection (k = half of the interleaved weight row)
  ActTiles gated_T;          // ... and their tiles
  size_t part_stride;        // TG_SWIGLU: part i of a cut tile (counted along the line) is stored i * part_stride further; 0: added
  int stages;                // pipeline stages of a block, 2 .. TG_MAX_STAGES
  int n_acc, tmem_cols;      // accumulators in tensor memory (1 or 2), tmem_cols / n_acc columns apart
  int *error;
  long long wait_limit;
};

__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  // start address, leading (between the two k chunks of an MMA) and stride (between 8-row groups)
  // byte offsets, all without their 4 low bits; descriptor version 1; no swizzle
  return (uint64_t)((smem_addr & 0x3ffff) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
         (1ull << 46);
}

// kind::f16 instruction descriptor: fp32 accumulate, bf16 A and B, both K-major, M x N
__device__ __forceinline__ uint32_t umma_instr_desc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Bounded wait.  The error word (another block gave up) is looked at only after the wait has lasted half a
// millisecond: a read of global memory inside the spin takes a microsecond under load, which made every wait that
// long (head at 8 rows 2.2 TB/s instead of 6).
__device__ __noinline__ bool tg_wait_slow(uint32_t bar, uint32_t parity, int *error, long long limit) {
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    const long long dt = clock64() - t0;
    if (dt > (1 << 20) && (dt > limit || *reinterpret_cast<volatile int *>(error) >= TG_ERR_WAIT)) {
      atomicMax(error, TG_ERR_WAIT);
      return false;
    }
  }
}
template <class Params>
__device__ __forceinline__ bool tg_wait(uint32_t bar, uint32_t parity, const Params &P) {
  return mbar_try_wait(bar, parity) || tg_wait_slow(bar, parity, P.error, P.wait_limit);
}
// Arrive on the barrier at the same place in the first SM of the pair.  Without a scope: what is handed over is the
// completion of bulk copies and of tensor-memory loads, not this thread's stores, and an arrive that releases at
// cluster scope waits for a fence of about 2000 cycles under load, once per stage.
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
  asm volatile(
      "{\n .reg .b32 a;\n mapa.shared::cluster.u32 a, %0, 0;\n"
      " mbarrier.arrive.shared::cluster.b64 _, [a];\n}\n" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  // arrives on the barrier at this place in both SMs once the MMAs issued so far are complete
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
}
__device__ __forceinline__ void red_add(float *p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
// `tiles` tiles of n_kb units each, cut into equal parts for n_pairs block pairs.
inline TgLine tg_line(int tiles, int n_kb, int n_pairs) { return TgLine{tiles * n_kb / n_pairs, tiles * n_kb % n_pairs, n_pairs}; }
// ... no tile in more than two parts: a sum onto zeroed outputs is then the same in either order.  Leaves block pairs idle
// where there are fewer tiles than pairs.
inline TgLine tg_line_two(int tiles, int n_kb, int n_pairs) {
  return tg_line(tiles, n_kb, tiles >= n_pairs ? n_pairs : std::max(1, n_kb % 2 == 0 && 2 * tiles <= n_pairs ? 2 * tiles : tiles));
}
// Column tiles so narrow that every block pair takes one whole tile of n_rt row-tile pairs (or none): nothing is cut, every
// output has one sum.
inline ActTiles act_tiles_uncut(int rows, int n_kb, int n_rt, int n_pairs) {
  ActTiles t = act_tiles_for(rows, n_kb);
  const int most = std::max(1, n_pairs / n_rt);
  t.tile_rows = ((rows + most - 1) / most + 15) / 16 * 16;
  t.n_ctiles = (rows + t.tile_rows - 1) / t.tile_rows;
  return t;
}
// Row-tile pairs dealt out whole: the largest multiple of the block pairs.
inline int tg_whole_pairs(const UmmaMat &W, int whole, int n_pairs) {
  return whole == TG_ADD ? 0 : W.n_tiles / 2 / n_pairs * n_pairs;
}

// The units of a block pair in order: its part of the line of units of the remaining row-tile pairs, then its whole
// tiles; k fastest, then the column tile.
struct TgCursor {
  int kb, ct, rt;            // k block, column tile, row-tile pair
  int left;                  // units left of the line; then 0
  int step;                  // row-tile pairs from one tile row to the next
  // units of the next stage: whole tiles and the line's parts end where a stage ends
  __device__ __forceinline__ int units(int n_kb, int most) const { return min(min(most, n_kb - kb), left > 0 ? left : most); }
  __device__ __forceinline__ void next(int n, int n_kb, int n_ct, int pair, int n_pairs) {
    if (left > 0 && (left -= n) == 0) {
      kb = 0; ct = 0; rt = pair; step = n_pairs;
      return;
    }
    if ((kb += n) == n_kb) {
      kb = 0;
      if (++ct == n_ct) { ct = 0; rt += step; }
    }
  }
};

// TG_SWIGLU epilogue: the lane's weight row is 2 i (gate) or 2 i + 1 (up) of intermediate index i, r its values for 16
// activation rows.  Even lanes gate the even columns, odd lanes the odd ones; the 8 x 8 transposes between the lanes of
// eight indices then leave every lane with one 16-byte unit (8 indices of one activation row), hi and lo part.
// On return hi / lo are the unit of column 2 * ((lane >> 1) & 7) + (lane & 1) and of the indices 8 * (lane >> 4) .. + 7 of
// the warp's 16.
__device__ __forceinline__ void swiglu_units(const uint32_t (&r)[16], uint4 &hi, uint4 &lo) {
  const int lane = threadIdx.x & 31, odd = lane & 1, p = lane >> 1;
  uint32_t w[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float send = __uint_as_float(odd ? r[2 * q] : r[2 * q + 1]);
    const float recv = __shfl_xor_sync(0xffffffffu, send, 1);
    const float g = odd ? recv : __uint_as_float(r[2 * q]), u = odd ? __uint_as_float(r[2 * q + 1]) : recv;
    const float a = g / (1.f + expf(-g)) * u;
    const __nv_bfloat16 h = __float2bfloat16_rn(a), l = __float2bfloat16_rn(a - __bfloat162float(h));
    w[q] = (uint32_t)__bfloat16_as_ushort(h) | ((uint32_t)__bfloat16_as_ushort(l) << 16);
  }
#pragma unroll
  for (int b = 1; b < 8; b <<= 1) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (q & b) continue;
      const bool up = (p & b) != 0;
      const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? w[q] : w[q | b], b << 1);
      if (up) w[q] = got; else w[q | b] = got;
    }
  }
  uint32_t h4[4], l4[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    h4[j] = __byte_perm(w[2 * j], w[2 * j + 1], 0x5410);
    l4[j] = __byte_perm(w[2 * j], w[2 * j + 1], 0x7632);
  }
  hi = make_uint4(h4[0], h4[1], h4[2], h4[3]);
  lo = make_uint4(l4[0], l4[1], l4[2], l4[3]);
}

// SPLIT: the form of the column tiles (one tile of up to 128 rows); WHOLE: what becomes of the tiles dealt out whole.  (Forms
// of their own: the code that a decode launch does not run cost it 2 us per layer, a launch fetches its instructions anew.)
template <bool SPLIT, int WHOLE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TG_THREADS, 1) gemm_tc05_kernel(const __grid_constant__ GemmTcParams P) {
  extern __shared__ __align__(1024) unsigned char tg_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int S = P.stages, n_kb = P.W.n_kb, tile_rows = P.T.tile_rows;
  constexpr int KPS = tg_stage_units(SPLIT);
  const uint32_t act_bytes = (uint32_t)tile_rows * 128, act_off = KPS * TG_WBLOCK, stage_bytes = act_off + KPS * act_bytes;
  unsigned char *const tail = tg_smem + (size_t)S * stage_bytes;
  const uint32_t full0 = smem_u32(tail), empty0 = full0 + 8 * TG_MAX_STAGES, acc_full0 = empty0 + 8 * TG_MAX_STAGES,
                 acc_empty0 = acc_full0 + 16;
  uint32_t *const tmem_slot = reinterpret_cast<uint32_t *>(tail + 16 * TG_MAX_STAGES + 32);
  volatile int *const gave_up = reinterpret_cast<volatile int *>(tmem_slot + 1);   // a wait of this block ran out: no more output

  // this pair's share of the units
  const int n_ct = SPLIT ? 1 : P.T.n_ctiles;
  const int u0 = P.line.begin(pair), n_part = P.line.size(pair);
  const int n_it = n_part + (WHOLE == TG_ADD ? 0 : P.whole_units);
  TgCursor start;
  if (n_part > 0) {
    const int tile = u0 / n_kb, row = n_ct == 1 ? tile : tile / n_ct;
    start = TgCursor{u0 - tile * n_kb, tile - row * n_ct, P.rt_whole + row, n_part, 1};
  } else {
    start = TgCursor{0, 0, pair, 0, n_pairs};
  }

  TgCursor cur_w = start, cur_a = start;               // producer's positions (thread 0)
  auto copy_w = [&](int st, int n) {                   // the k blocks of a row tile follow one another
    bulk_g2s(smem_u32(tg_smem) + st * stage_bytes, P.W.w + ((size_t)(2 * cur_w.rt + rank) * n_kb + cur_w.kb) * (TG_WBLOCK / 16),
             n * TG_WBLOCK, full0 + st * 8);
    cur_w.next(n, n_kb, n_ct, pair, n_pairs);
  };
  auto copy_act = [&](int st, int n) {
    for (int u = 0; u < n; ++u)
      bulk_g2s(smem_u32(tg_smem) + st * stage_bytes + act_off + u * act_bytes,
               P.act_blocks + (((size_t)cur_a.ct * n_kb + cur_a.kb + u) * 2 + rank) * P.T.units_per_sm(), act_bytes, full0 + st * 8);
    cur_a.next(n, n_kb, n_ct, pair, n_pairs);
  };
  int n_first = 0, issued_units = 0;                   // (thread 0) the stages requested before the activations are there
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full0 + s * 8, rank == 0 ? 2 : 1);       // this block's copies; on the first SM also the other's
      mbar_init(empty0 + s * 8, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(acc_full0 + a * 8, 1);
      mbar_init(acc_empty0 + a * 8, 2 * TG_EPI_WARPS);   // the epilogue warps of both blocks
    }
    *gave_up = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(P.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // The kernel after this one (the next projection's activation-block kernel, launched the same way) may become
  // resident now; it waits for this grid's completion before it reads or writes anything, and the GEMM behind it
  // can then request its first weight blocks while this grid's last blocks finish.  Not before this block holds its
  // tensor memory: a later grid that took the columns first would wait for this one, and an allocation has no limit.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  if (threadIdx.x == 0) {
    // the weight blocks of the first stages are requested before the other block is waited for: they touch this
    // block's barriers only, and eight copies take the issuing thread some thousand cycles
    for (; n_first < (SPLIT ? min(S, TG_PACE_FREE) : S) && issued_units < n_it; ++n_first) {
      const int n = cur_w.units(n_kb, KPS);
      mbar_expect_tx(full0 + n_first * 8, n * (TG_WBLOCK + act_bytes));
      copy_w(n_first, n);
      issued_units += n;
    }
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const int acc_cols = P.tmem_cols / P.n_acc;

  if (warp == 0) {
    if (lane == 0) {
      // ---- producer: a bulk copy for a stage's weights and one for each unit's activations; the activation blocks only after the kernel that writes them has
      // completed and its writes are visible
      if (SPLIT) {
        // the rest of the ring's first round at the pace of HBM; the activations of this round are copied by an epilogue warp
        long long t = clock64();
        for (; n_first < S && issued_units < n_it; ++n_first) {
          while (clock64() - t < TG_PACE) {}
          t = clock64();
          const int n = cur_w.units(n_kb, KPS);
          mbar_expect_tx(full0 + n_first * 8, n * (TG_WBLOCK + act_bytes));
          copy_w(n_first, n);
          issued_units += n;
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int i = 0; i < n_first; ++i) cur_a.next(cur_a.units(n_kb, KPS), n_kb, n_ct, pair, n_pairs);
      } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int i = 0; i < n_first; ++i) copy_act(i, cur_a.units(n_kb, KPS));
      }
      int st = 0, issued = n_first;
      uint32_t ph = 0;
      bool ok = true;
      while (issued_units < n_it) {
        ok = tg_wait(empty0 + st * 8, ph, P);
        if (!ok) break;
        const int n = cur_w.units(n_kb, KPS);
        mbar_expect_tx(full0 + st * 8, n * (TG_WBLOCK + act_bytes));
        copy_w(st, n);
        copy_act(st, n);
        issued_units += n;
        ++issued;
        if (++st == S) { st = 0; ph ^= 1; }
      }
      if (!ok) {
        // leave no copy in flight: each stage's last copies get a bounded wait
        for (int i = max(0, issued - S); i < issued; ++i) {
          const long long t0 = clock64();
          while (!mbar_try_wait(full0 + (i % S) * 8, (i / S) & 1))
            if (clock64() - t0 > P.wait_limit) break;
        }
      }
    }
  } else if (warp == 1 && rank == 0) {
    // ---- MMA issuer
    const int n_cols = SPLIT ? 2 * tile_rows : tile_rows;         // MMA N
    const uint32_t idesc = umma_instr_desc(2 * TG_ROWS, n_cols);
    const uint32_t b_lbo = (uint32_t)(n_cols / 2) * 16;
    // what a unit costs is instructions in a row, so the descriptors and barriers of the stage are carried along
    const uint64_t da0 = umma_smem_desc(smem_u32(tg_smem), (TG_ROWS / 8) * 128, 128),
                   db0 = umma_smem_desc(smem_u32(tg_smem) + act_off, b_lbo, 128);
    const uint64_t da_step = 2 * (TG_ROWS / 8) * 128 / 16, db_step = 2 * b_lbo / 16, part_step = b_lbo * 8 / 16;
    const uint32_t st_step = stage_bytes / 16, full_end = full0 + 8 * S;
    uint64_t da_st = da0, db_st = db0;
    uint32_t full = full0, ph = 0, acc_ph = 1, d = tmem;              // the accumulators start free
    int kb = start.kb, acc = 0;
    bool first = true, ok = true;
    for (int i = 0; i < n_it;) {
      if (first) {
        ok = __all_sync(0xffffffffu, tg_wait(acc_empty0 + acc * 8, acc_ph, P));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      }
      ok = __all_sync(0xffffffffu, mbar_try_wait(full, ph)) || __all_sync(0xffffffffu, tg_wait_slow(full, ph, P.error, P.wait_limit));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int n = min(min(KPS, n_kb - kb), i < n_part ? n_part - i : KPS);
      kb += n;
      i += n;
      const bool last = kb == n_kb || i == n_part;
      if (elect_one()) {
        const uint32_t accumulate = first ? 0u : 1u;
#pragma unroll
        for (int u = 0; u < KPS; ++u) {
          if (u && n == 1) break;
          const uint64_t da = da_st + u * (TG_WBLOCK / 16), db = db_st + u * (act_bytes / 16);
#pragma unroll
          for (int kk = 0; kk < TG_KB / 16; ++kk) {
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(da + kk * da_step), "l"(db + kk * db_step), "r"(idesc), "r"(u || kk ? 1u : accumulate)
                : "memory");
            if (!SPLIT)                                           // the lo part into the same columns
              asm volatile(
                  "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                  " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                  "l"(da + kk * da_step), "l"(db + kk * db_step + part_step), "r"(idesc), "r"(1u)
                  : "memory");
          }
        }
        umma_commit_pair(full + 8 * TG_MAX_STAGES);               // the stage's empty barrier
        if (last) umma_commit_pair(acc_full0 + acc * 8);
      }
      __syncwarp();
      first = last;
      if (last) {
        kb = 0;
        if (++acc == P.n_acc) { acc = 0; acc_ph ^= 1; }
        d = tmem + acc * acc_cols;
      }
      full += 8; da_st += st_step; db_st += st_step;
      if (full == full_end) { full = full0; ph ^= 1; da_st = da0; db_st = db0; }
    }
    if (!ok && lane == 0) { *gave_up = 1; __threadfence_block(); }
  } else if (warp == 1) {
    // ---- second SM: pass every landed stage on to the issuer
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 0;
      TgCursor cur = start;
      for (int i = 0; i < n_it;) {
        const int n = cur.units(n_kb, KPS);
        if (!tg_wait(full0 + st * 8, ph, P)) break;
        mbar_arrive_leader(full0 + st * 8);
        cur.next(n, n_kb, n_ct, pair, n_pairs);
        i += n;
        if (++st == S) { st = 0; ph ^= 1; }
      }
    }
  } else {
    // ---- epilogue: thread = weight row (lane of tensor memory), registers = columns
    if (SPLIT && warp == 2) {
      // the activations of the ring's first round, while the producer is still asking for its weights
      if (lane == 0) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int i = 0, units = 0; i < S && units < n_it; ++i) {
          const int n = cur_a.units(n_kb, KPS);
          copy_act(i, n);
          units += n;
        }
      }
      __syncwarp();
    }
    const int quarter = warp & 3;
    int acc = 0, kb = start.kb, ct = start.ct, rt = start.rt, left = n_part;
    uint32_t ph = 0;
    for (int i = 0; i < n_it;) {
      // the next tile of the share, or part of one
      const bool whole = WHOLE != TG_ADD && left == 0;
      const int units = whole ? n_kb : min(n_kb - kb, left), this_ct = ct, this_rt = rt;
      i += units;
      kb = 0;
      if (!whole && (left -= units) == 0) { ct = 0; rt = pair; }
      else if (++ct == n_ct) { ct = 0; rt += whole ? n_pairs : 1; }
      const bool ok = __all_sync(0xffffffffu, tg_wait(acc_full0 + acc * 8, ph, P)) && !*gave_up;
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int n = (2 * this_rt + rank) * TG_ROWS + quarter * 32 + lane;
      const int m0 = this_ct * tile_rows, n_rows = min(tile_rows, P.rows - m0);
      const uint32_t t_base = tmem + ((uint32_t)(quarter * 32) << 16) + acc * acc_cols;
      const int c_first = warp < 6 ? 0 : 16;
      float *dst = P.out + (size_t)(m0 + c_first) * P.ldo + (n - (WHOLE == TG_SWIGLU ? P.out_n0 : 0));
      const bool in_parts = WHOLE == TG_SWIGLU && !whole && P.part_stride;
      if (in_parts) dst += (pair - P.line.holder(((this_rt - P.rt_whole) * n_ct + this_ct) * n_kb)) * P.part_stride;
#pragma unroll 1
      for (int c0 = c_first; c0 < n_rows; c0 += 32) {
        uint32_t r[16];
        tmem_ld16(t_base + c0, r);
        if (SPLIT) {                                              // the lo columns
          uint32_t q[16];
          tmem_ld16(t_base + tile_rows + c0, q);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(q[j]));
        } else {
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        }
        // straight-line code for whole groups of 16 rows: a warp has its scheduler to itself, every instruction counts
        if (n >= P.W.N) {                                             // rows that pad the last tile (gate+up: whole tiles of them)
        } else if (WHOLE == TG_SWIGLU && whole) {
          uint4 hi, lo;
          swiglu_units(r, hi, lo);
          const int col = c0 + 2 * ((lane >> 1) & 7) + (lane & 1);
          if (col < n_rows) {
            const int kb = 2 * this_rt + rank, c = 2 * quarter + (lane >> 4), half = tile_rows / 2, sm = col >= half ? 1 : 0;
            uint4 *u = P.gated + (P.gated_T.tile_rows != tile_rows
                                      ? P.gated_T.unit(m0 + col, kb, c)
                                      : (((size_t)this_ct * P.gated_T.n_kb + kb) * 2 + sm) * P.T.units_per_sm() + c * half + (col - sm * half));
            u[0] = hi;
            u[P.gated_T.lo_offset()] = lo;
          }
        } else {
          if (whole || in_parts) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j < n_rows) dst[(size_t)j * P.ldo] = __uint_as_float(r[j]);
          } else if (c0 + 16 <= n_rows) {
            float *d = dst;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              red_add(d, __uint_as_float(r[j]));
              d += P.ldo;
            }
          } else {
#pragma unroll
            for (int j = 0; j < 15; ++j)
              if (c0 + j < n_rows) red_add(dst + (size_t)j * P.ldo, __uint_as_float(r[j]));
          }
        }
        dst += (size_t)32 * P.ldo;
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_leader(acc_empty0 + acc * 8);
      if (++acc == P.n_acc) { acc = 0; ph ^= 1; }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // the other block is done with this one's shared and tensor memory (no release: it would wait for the reductions)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(P.tmem_cols) : "memory");
  }
}

// 8 values of k of an activation row as its hi and lo units.
__device__ __forceinline__ void store_hi_lo(const float (&f)[8], uint4 *dst, size_t lo_offset) {
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    hi[j] = pack_bf16x2(f[2 * j], f[2 * j + 1]);
    lo[j] = pack_bf16x2(f[2 * j] - __uint_as_float(hi[j] << 16), f[2 * j + 1] - __uint_as_float(hi[j] & 0xffff0000u));
  }
  dst[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  dst[lo_offset] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

// Activations [rows][lda] fp32 -> bf16 hi/lo units (8 values of k of a row, 16 bytes a part) in the order of ActTiles.
// With GATED the source rows hold gate and up values in turn and the activation is the SwiGLU gate silu(gate) * up
// (step a6, second half), computed on the way; the source's first column then belongs to k block kb0.
// A warp takes a k block of four rows at a time: it reads whole rows of it (512 bytes in a row; every load in flight
// before the first is used), and the lanes exchange their parts so that each stores a unit beside its neighbour row's.
// No shared memory, so that the blocks become resident beside the GEMM in front.
// Bound by the time of one trip to memory behind the next projection's first weights, which its blocks
// request meanwhile: with a thread to a unit (its lanes' loads 32 rows apart, 16 bytes each) a block took 13.6 us at
// 96 rows of the Qwen3-4B shape and 6 us at 32 (4 cycles of 32 sequences 21.3 ms, 20.3 so).
constexpr int AB_ROWS = 4, AB_THREADS = 256;
// The parts that the cut tiles of gate+up were stored in (stride 0: one buffer that they were added into).  A form of its own:
// with the registers of its loads in flight fewer blocks become resident beside the GEMM in front (4 cycles of 32 sequences:
// 20.7 ms with one form for both, 20.45 with two).
struct GateUpParts {
  TgLine line;
  int n_ct, n_kb, tile_rows;
  size_t stride;
  // parts of the tile of k block kb (of the intermediate values: two of them to a row-tile pair) and row m
  __device__ __forceinline__ int count(int kb, int m) const {
    const int u = (kb / (TG_ROWS / TG_KB) * n_ct + m / tile_rows) * n_kb;
    return line.holder(u + n_kb - 1) - line.holder(u) + 1;
  }
};
template <bool GATED, bool PARTS = false>
__global__ void __launch_bounds__(AB_THREADS) act_blocks_kernel(const float *act, int lda, int rows, ActTiles T,
                                                                uint4 *blocks, int kb0, GateUpParts parts) {
  // lanes of a row, 16-byte loads of a lane, and 32-bit registers of a part that a load becomes
  constexpr int LANES = GATED ? 32 : 16, LOADS = AB_ROWS * LANES / 32, REGS = GATED ? 1 : 2;
  // the GEMM that follows may be scheduled already: it waits for this grid before it reads the blocks
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ... and this grid may itself have started before the kernel before it has finished (the GEMM of the previous
  // projection lets its dependents in at once): nothing is read or written before that kernel is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31, col = lane % LANES, half = lane / LANES;
  const int row_tiles = (rows + AB_ROWS - 1) / AB_ROWS, n_tiles = (T.n_kb - kb0) * row_tiles;
  for (int tile = blockIdx.x * (AB_THREADS / 32) + (threadIdx.x >> 5); tile < n_tiles; tile += gridDim.x * (AB_THREADS / 32)) {
    const int kb = tile / row_tiles, m0 = (tile % row_tiles) * AB_ROWS;
    float4 v[LOADS];                                                 // load i: row m0 + i (32 / LANES) + half
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
      const int m = m0 + i * (32 / LANES) + half;
      v[i] = m < rows ? *reinterpret_cast<const float4 *>(act + (size_t)m * lda + (size_t)kb * LANES * 4 + col * 4)
                      : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (PARTS) {
      const int n = parts.count(kb, m0);                             // four rows lie in one tile
      constexpr int AHEAD = 5;
#pragma unroll 1
      for (int p0 = 1; p0 < n; p0 += AHEAD) {
        float4 u[AHEAD][LOADS];
#pragma unroll
        for (int p = 0; p < AHEAD; ++p)
#pragma unroll
          for (int i = 0; i < LOADS; ++i) {
            const int m = min(m0 + i * (32 / LANES) + half, rows - 1);
            u[p][i] = *reinterpret_cast<const float4 *>(act + min(p0 + p, n - 1) * parts.stride + (size_t)m * lda + (size_t)kb * LANES * 4 + col * 4);
          }
#pragma unroll
        for (int p = 0; p < AHEAD; ++p)
#pragma unroll
          for (int i = 0; i < LOADS; ++i)
            if (p0 + p < n) { v[i].x += u[p][i].x; v[i].y += u[p][i].y; v[i].z += u[p][i].z; v[i].w += u[p][i].w; }
      }
    }
    uint32_t hi[LOADS][REGS], lo[LOADS][REGS];
    auto split = [](float a, float b, uint32_t &h, uint32_t &l) {
      h = pack_bf16x2(a, b);
      l = pack_bf16x2(a - __uint_as_float(h << 16), b - __uint_as_float(h & 0xffff0000u));
    };
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
      if (GATED) {
        split(v[i].x / (1.f + expf(-v[i].x)) * v[i].y, v[i].z / (1.f + expf(-v[i].z)) * v[i].w, hi[i][0], lo[i][0]);
      } else {
        split(v[i].x, v[i].y, hi[i][0], lo[i][0]);
        split(v[i].z, v[i].w, hi[i][REGS - 1], lo[i][REGS - 1]);
      }
    }
    // the LOADS lanes of a unit hold a LOADS-th of it for each of LOADS rows: transposed, lane q of them holds row q's unit
    auto transpose = [&](uint32_t (&x)[LOADS][REGS]) {
#pragma unroll
      for (int step = 1; step < LOADS; step <<= 1) {
        const bool up = lane & step;
#pragma unroll
        for (int i = 0; i < LOADS; ++i)
          if (!(i & step)) {
#pragma unroll
            for (int r = 0; r < REGS; ++r) {
              const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? x[i][r] : x[i + step][r], step);
              if (up) x[i][r] = got;
              else x[i + step][r] = got;
            }
          }
      }
    };
    transpose(hi);
    transpose(lo);
    const int q = col & (LOADS - 1), m = m0 + q * (32 / LANES) + half;
    if (m < rows) {
      uint4 *dst = blocks + T.unit(m, kb0 + kb, col / LOADS);
      if (GATED) {
        dst[0] = make_uint4(hi[0][0], hi[1 % LOADS][0], hi[2 % LOADS][0], hi[3 % LOADS][0]);
        dst[T.lo_offset()] = make_uint4(lo[0][0], lo[1 % LOADS][0], lo[2 % LOADS][0], lo[3 % LOADS][0]);
      } else {
        dst[0] = make_uint4(hi[0][0], hi[0][REGS - 1], hi[1][0], hi[1][REGS - 1]);
        dst[T.lo_offset()] = make_uint4(lo[0][0], lo[0][REGS - 1], lo[1][0], lo[1][REGS - 1]);
      }
    }
  }
}

// RMSNorm and the activation blocks in one kernel (steps a2 / a6 / a9, first half, on the tcgen05
// path): block g < n_groups takes 4 rows, sums their squares, and writes their hi and lo parts of
// every k block; the blocks behind them clear the buffer the GEMM accumulates into.  x [rows][ldx]
// fp32; K values per row.
// The rows come in segments of seg_rows every seg_stride rows of x (the rows of a chunk that the LM head
// reads when logits of many positions are asked for); seg_rows = 0: one segment.
constexpr int NAB_ROWS = 4;
// `cols` columns of `rows` rows that lie ld floats apart
struct ZeroArea {
  float *p;
  int rows, cols;
  size_t ld;
};
struct RowSegments {
  int seg_rows, seg_stride;
  __host__ __device__ __forceinline__ size_t row(int m) const {
    return seg_rows > 0 ? (size_t)(m / seg_rows) * seg_stride + m % seg_rows : (size_t)m;
  }
};
// Rows m0 .. m0 + 3 by 256 threads (tid), k blocks [kb_lo, kb_hi): a share of the k blocks needs the whole rows' sums of
// squares.  What a thread's first unit needs is requested beside the rows, so that the whole costs one trip to memory
// (as two, and with the rows' loads in small batches, 5.5 us a launch instead of 4.5).  part: 8 floats of shared memory.
__device__ __forceinline__ void norm_group(const float *x, int ldx, RowSegments seg, const float *__restrict__ w, float eps, int rows_all,
                                           int K, const ActTiles &T, uint4 *blocks, int m0, int kb_lo, int kb_hi, float *part,
                                           int tid) {
  const int warp = tid >> 5, lane = tid & 31;
  // unit = (k block, k chunk of 8, row of the group): this thread writes the row's hi and lo parts
  const int r = tid % NAB_ROWS, c = (tid / NAB_ROWS) % 8, total = (kb_hi - kb_lo) * 8 * NAB_ROWS;
  const bool row_ok = m0 + r < rows_all;
  const float *xu = x + seg.row(row_ok ? m0 + r : 0) * ldx + c * 8;
  float4 ua = make_float4(0.f, 0.f, 0.f, 0.f), ub = ua, wa = ua, wb = ua;
  auto load_unit = [&](int u) {
    const int k0 = (kb_lo + u / (NAB_ROWS * 8)) * TG_KB;
    ua = __ldcg(reinterpret_cast<const float4 *>(xu + k0));
    ub = __ldcg(reinterpret_cast<const float4 *>(xu + k0 + 4));
    wa = __ldg(reinterpret_cast<const float4 *>(w + k0 + c * 8));
    wb = __ldg(reinterpret_cast<const float4 *>(w + k0 + c * 8 + 4));
  };
  if (tid < total && row_ok) load_unit(tid);
  {
    // two warps per row
    const int m = m0 + (warp >> 1);
    float ss = 0.f;
    if (m < rows_all) {
      const float4 *xr = reinterpret_cast<const float4 *>(x + seg.row(m) * ldx);
      const int n4 = K / 4;
#pragma unroll 1
      for (int k4 = (warp & 1) * 32 + lane; k4 < n4; k4 += 64 * 10) {
        float4 v[10];
#pragma unroll
        for (int j = 0; j < 10; ++j) v[j] = k4 + 64 * j < n4 ? __ldcg(xr + k4 + 64 * j) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 10; ++j) ss += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
      }
    }
    ss = warp_sum(ss);
    if (lane == 0) part[warp] = ss;
  }
  __syncthreads();
  const float s = rsqrtf((part[2 * r] + part[2 * r + 1]) / (float)K + eps);
  if (!row_ok) return;
#pragma unroll 1
  for (int u = tid; u < total; u += 256) {
    if (u != tid) load_unit(u);
    const float f[8] = {ua.x * s * wa.x, ua.y * s * wa.y, ua.z * s * wa.z, ua.w * s * wa.w,
                        ub.x * s * wb.x, ub.y * s * wb.y, ub.z * s * wb.z, ub.w * s * wb.w};
    store_hi_lo(f, blocks + T.unit(m0 + r, kb_lo + u / (NAB_ROWS * 8), c), T.lo_offset());
  }
}

__global__ void __launch_bounds__(256) norm_act_blocks_kernel(const float *x, int ldx, RowSegments seg,
                                                              const float *__restrict__ w, float eps, int rows_all, int K,
                                                              ActTiles T, uint4 *blocks, int n_groups,
                                                              ZeroArea zero_area) {
  // the GEMM that follows may be scheduled already: it waits for this grid before it reads the blocks
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ... and this grid may itself have started before the kernel before it has finished (the GEMM of the previous
  // projection lets its dependents in at once): nothing is read or written before that kernel is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if ((int)blockIdx.x >= n_groups) {
    const size_t n_z = (size_t)(gridDim.x - n_groups) * gridDim.y;
    const size_t zero_n = (size_t)zero_area.rows * zero_area.cols;
    float *zero = zero_area.p;
    const size_t i0 = ((size_t)(blockIdx.x - n_groups) * gridDim.y + blockIdx.y) * blockDim.x + threadIdx.x;
    if (zero_area.cols < zero_area.ld) {               // columns of longer rows
      for (size_t i = i0; i < zero_n; i += n_z * blockDim.x) zero[i / zero_area.cols * zero_area.ld + i % zero_area.cols] = 0.f;
      return;
    }
    const size_t head = min(zero_n, (size_t)((16 - (reinterpret_cast<uintptr_t>(zero) & 15)) & 15) / 4);   // up to the first 16-byte boundary
    float4 *z4 = reinterpret_cast<float4 *>(zero + head);
    const size_t n4 = (zero_n - head) / 4;
    for (size_t i = i0; i < n4; i += n_z * blockDim.x) z4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 < head) zero[i0] = 0.f;
    if (i0 < zero_n - head - n4 * 4) zero[head + n4 * 4 + i0] = 0.f;
    return;
  }
  __shared__ float part[8];
  norm_group(x, ldx, seg, w, eps, rows_all, K, T, blocks, blockIdx.x * NAB_ROWS, T.n_kb * blockIdx.y / gridDim.y,
             T.n_kb * (blockIdx.y + 1) / gridDim.y, part, threadIdx.x);
}

// The merge of the attention's key slices (step a4, second half) and the activation blocks of the O
// projection in one kernel: block g takes 4 rows, works out the weight of every (row, head, slice)
// from the slices' running max and sum, and writes the merged head outputs as hi and lo columns.
// part_o [(row * nq + head) * nsplit + slice][D], part_ml the same with (max, sum); K = nq * D.
constexpr int MAB_MAX_SLOTS = 2048;            // (rows of a group) x heads x slices the weights of a group may take
// Rows m0 .. m0 + 3, k blocks [kb_lo, kb_hi), by 256 threads: the weight of every (row, head, slice) from the slices' max and
// sum (one thread per row and head, into wgt), then the merged values.  A thread's first unit has its first slices
// requested beside the weights' inputs: one trip to memory for up to eight slices, and as many at a time behind them.
// (The slices behind the first four one by one were a trip each: 3 sequences at context 700 to 1000, 6 cycles 21.2 -> 20.0 ms;
// one sequence at 1500 keys 863 -> 828 us for 4 layers' three passes.)
constexpr int MERGE_AHEAD = 8;
__device__ __forceinline__ void merge_group(const float *part_o, const float *part_ml, int nsplit, int nq, int D,
                                            int rows_all, const ActTiles &T, uint4 *blocks, int m0, int kb_lo, int kb_hi,
                                            float *wgt, int tid) {
  const int r = tid % NAB_ROWS, c = (tid / NAB_ROWS) % 8, m = m0 + r, total = (kb_hi - kb_lo) * 8 * NAB_ROWS;
  const bool row_ok = m < rows_all;
  float4 va[MERGE_AHEAD], vb[MERGE_AHEAD];
  const float *po = nullptr;
  int h = 0;
  auto load_unit = [&](int u) {
    const int k = (kb_lo + u / (NAB_ROWS * 8)) * TG_KB + c * 8;
    h = k / D;
    po = part_o + ((size_t)m * nq + h) * nsplit * D + (k - h * D);
    // (slots that no slice was written to are loaded too, but not used)
#pragma unroll
    for (int s = 0; s < MERGE_AHEAD; ++s)
      if (s < nsplit) {
        va[s] = *reinterpret_cast<const float4 *>(po + (size_t)s * D);
        vb[s] = *reinterpret_cast<const float4 *>(po + (size_t)s * D + 4);
      }
  };
  if (tid < total && row_ok) load_unit(tid);
#pragma unroll 1
  for (int i = tid; i < NAB_ROWS * nq; i += 256) {
    const int wr_row = i / nq, wr_h = i - wr_row * nq, wm = m0 + wr_row;
    if (wm >= rows_all) continue;
    float *wr = wgt + (size_t)i * nsplit;
    const float2 *ml = reinterpret_cast<const float2 *>(part_ml) + ((size_t)wm * nq + wr_h) * nsplit;
    float2 v[MERGE_AHEAD];
    float mx = -INFINITY;
    for (int s0 = 0; s0 < nsplit; s0 += MERGE_AHEAD) {
#pragma unroll
      for (int s = 0; s < MERGE_AHEAD; ++s) v[s] = s0 + s < nsplit ? ml[s0 + s] : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int s = 0; s < MERGE_AHEAD; ++s)
        if (v[s].y > 0.f) mx = fmaxf(mx, v[s].x);
    }
    float l = 0.f;
    for (int s0 = 0; s0 < nsplit; s0 += MERGE_AHEAD) {
      if (nsplit > MERGE_AHEAD) {
#pragma unroll
        for (int s = 0; s < MERGE_AHEAD; ++s) v[s] = s0 + s < nsplit ? ml[s0 + s] : make_float2(-INFINITY, 0.f);
      }
#pragma unroll
      for (int s = 0; s < MERGE_AHEAD; ++s) {
        const float f = v[s].y > 0.f ? __expf(v[s].x - mx) : 0.f;
        if (s0 + s < nsplit) wr[s0 + s] = f;
        l += v[s].y * f;
      }
    }
    const float inv = 1.f / l;
    for (int s = 0; s < nsplit; ++s) wr[s] *= inv;
  }
  __syncthreads();
  if (!row_ok) return;
#pragma unroll 1
  for (int u = tid; u < total; u += 256) {
    if (u != tid) load_unit(u);
    const float *wr = wgt + (size_t)(r * nq + h) * nsplit;
    float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    auto add = [&](float ws, const float4 &a, const float4 &b) {
      if (ws != 0.f) {                                     // empty slices hold nothing that may be used
        f[0] += ws * a.x; f[1] += ws * a.y; f[2] += ws * a.z; f[3] += ws * a.w;
        f[4] += ws * b.x; f[5] += ws * b.y; f[6] += ws * b.z; f[7] += ws * b.w;
      }
    };
#pragma unroll
    for (int s = 0; s < MERGE_AHEAD; ++s)
      if (s < nsplit) add(wr[s], va[s], vb[s]);
    for (int s0 = MERGE_AHEAD; s0 < nsplit; s0 += MERGE_AHEAD) {
#pragma unroll
      for (int s = 0; s < MERGE_AHEAD; ++s)
        if (s0 + s < nsplit) {
          va[s] = *reinterpret_cast<const float4 *>(po + (size_t)(s0 + s) * D);
          vb[s] = *reinterpret_cast<const float4 *>(po + (size_t)(s0 + s) * D + 4);
        }
#pragma unroll
      for (int s = 0; s < MERGE_AHEAD; ++s)
        if (s0 + s < nsplit) add(wr[s0 + s], va[s], vb[s]);
    }
    store_hi_lo(f, blocks + T.unit(m, kb_lo + u / (NAB_ROWS * 8), c), T.lo_offset());
  }
}
__global__ void __launch_bounds__(256) merge_act_blocks_kernel(const float *part_o, const float *part_ml,
                                                               int nsplit, int nq, int D, int rows_all, ActTiles T,
                                                               uint4 *blocks) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ... and this grid may itself have started before the kernel before it has finished (the GEMM of the previous
  // projection lets its dependents in at once): nothing is read or written before that kernel is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ float wgt[MAB_MAX_SLOTS];
  merge_group(part_o, part_ml, nsplit, nq, D, rows_all, T, blocks, blockIdx.x * NAB_ROWS, T.n_kb * blockIdx.y / gridDim.y,
              T.n_kb * (blockIdx.y + 1) / gridDim.y, wgt, threadIdx.x);
}

// Weights [N][K] bf16 row-major (rows [row0, row0 + N_src) of the fused matrix) -> 16 KiB blocks.
// Source row r becomes row row0 + r * row_step (gate and up rows in turn: step 2).
__global__ void pack_umma_kernel(const __nv_bfloat16 *__restrict__ src, int N_src, int K, int row0, int row_step, int n_kb,
                                 uint4 *__restrict__ dst) {
  const long long total = (long long)N_src * (K / 8);              // 16-byte units of the source
  for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < total; u += (long long)gridDim.x * blockDim.x) {
    const int kc = (int)(u % (K / 8)), src_row = (int)(u / (K / 8)), row = row0 + src_row * row_step;
    const int tile = row / TG_ROWS, rg = (row % TG_ROWS) / 8, j = row % 8, kb = kc / 8, c = kc % 8;
    dst[(((size_t)tile * n_kb + kb) * 8 + c) * TG_ROWS + rg * 8 + j] =
        *reinterpret_cast<const uint4 *>(src + (size_t)src_row * K + kc * 8);
  }
}

}  // namespace dmtd
