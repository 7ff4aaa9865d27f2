// Step a4 as kernels of their own, for the per-step path and for dmtd_attention_decode: split-KV attention of a few new
// rows per sequence on the tensor cores (16-bit cache) or in FMAs (fp32 cache).  The G query heads of a kv head for up
// to 16 / G new positions form one set of query rows that share every key and value a block stages; the partial
// results of the key slices are merged by attn_merge_kernel or by the O projection's activation-block kernel.
#pragma once

#include "gemm_tc05.cuh"
#include "kernels.cuh"
#include "pass_attention_f32.cuh"

namespace dmtd {

// ---- 16-bit cache, head_dim 128: attn_decode_kernel
//
// KV-bound: a block has to keep as many bytes in flight as HBM's latency asks for and to lose no time between tiles.
//  * Every warp walks key tiles of its own (16 keys, K and V 4 KiB each) through a private ring filled by its own
//    asynchronous copies: no barrier of the block inside the key loop, so the warps' chains (scores, softmax, values:
//    about 1000 cycles per tile, latency of dependent instructions, not issue) run under each other and under the
//    copies.  mma.sync takes 8 cycles per SM sub-partition: the products of a tile are a fifth of HBM's time for it.
//  * The key tiles of all (sequence, kv head, row block) items are one line of 64-key units, cut into equal shares:
//    one wave of blocks (two per SM) whatever the batch and the context.  A share that crosses an item boundary writes
//    one partial result per item.
//  * Rows are 256 dense bytes; 16-byte part c of row r lies at part c ^ f(r) of its half row, f(r) = (r & 1) * 4 +
//    (r >> 1 & 3): free of bank conflicts for the copies, for the 16-byte operand loads of K and for ldmatrix on V.
// Measured, attention with its merge, against the kernel before it (64-key tiles of the whole block, two barriers per
// tile, slices of fixed length): 8 sequences x 16387 keys, 12 query rows per kv head, 159.8 -> 87.9 us, as clusters 81.3 (537 MB of K
// and V: 6.6 TB/s); a layer step of 64 sequences x 8192 keys, 4 query rows, 507 -> 381 us.
constexpr int AD_WARPS = 4;
constexpr int AD_THREADS = AD_WARPS * 32;
constexpr int AD_KEYS = 16;                                   // keys per warp tile
constexpr int AD_UNIT = AD_WARPS * AD_KEYS;                   // keys per unit of work
#ifndef DMTD_AD_STAGES
#define DMTD_AD_STAGES 2
#endif
constexpr int AD_STAGES = DMTD_AD_STAGES;                     // ring slots per warp: one tile multiplied, the others in flight
constexpr int AD_SLOT = 2 * AD_KEYS * 256;                    // K rows, then V rows
constexpr int AD_MAX_NEW = 15;                                // new positions per sequence the fused form takes (more: the prefill kernel)
constexpr int AD_RING = 0;
constexpr int AD_Q = AD_RING + AD_WARPS * AD_STAGES * AD_SLOT;        // query rows [16][PK_QROW]
constexpr int AD_NEW = AD_Q + PK_QR * PK_QROW;                // fused form: K rows of the pass [AD_MAX_NEW][128] (cache type), then V rows
constexpr int AD_OS = AD_NEW + 2 * AD_MAX_NEW * 256;          // the warps' outputs [AD_WARPS][16][PK_OROW] floats
constexpr int AD_RED = AD_OS + AD_WARPS * PK_QR * PK_OROW * 4;        // running max [AD_WARPS][16], then sum / merge factor
constexpr int AD_SMEM = AD_RED + 2 * AD_WARPS * PK_QR * 4;
static_assert(2 * (AD_SMEM + 1024) <= 228 * 1024, "two blocks per SM");

// byte offset of 16-byte part `part` (0..15) of row `row`
__device__ __forceinline__ uint32_t ad_part(int row, int part) {
  return (uint32_t)(row * 256 + ((part & 8) | ((part & 7) ^ (((row & 1) << 2) | ((row >> 1) & 3)))) * 16);
}

// The score that a tile's probabilities are taken relative to, exp(s - level): the tile's own largest, whose probability then
// is 1 and loses nothing when the probabilities are rounded to 16 bits for the product with V, but not more than AD_BELOW
// below the largest so far, so that sums stay within exp(AD_BELOW) of their usual size (tiles further down hardly count).
// With the running maximum alone the rounding loss grew with the tiles to a warp: 32 query and 8 kv heads, 1 x 1000 keys,
// bf16, error against fp64 1.91e-3 with one tile to a warp and 1.95e-3 with two.
constexpr float AD_BELOW = 4.f;
__device__ __forceinline__ float attn_level(float &top, float tile_max) {
  top = fmaxf(top, tile_max);
  return fmaxf(tile_max, top - AD_BELOW);
}

// One warp tile (16 keys, K at k_t, V at v_t) against up to 8 query rows, operands swapped: the keys are the M axis of
// S^T = K Q^T and the 128 output dimensions the M axis of O^T = V^T P^T, the query rows the 8 columns (with the rows on
// the M axis an m16 tile would be half padding or more).  Thread (g, t) holds columns (query rows) 2t, 2t + 1 of rows
// g and g + 8.  lim[e]: keys this lane's query row 2t + e sees, counted from the tile's first key.
struct AttnAccS {
  float m_run[2], l_part[2];       // per query row 2t, 2t + 1: level of the sums, this lane's share of the running sum
  float top[2];                    // ... the largest score
  float o[8][4];                   // O^T: m-tile dt = dimensions 16 dt .. + 15
  __device__ __forceinline__ void clear() {
    m_run[0] = m_run[1] = top[0] = top[1] = -INFINITY;
    l_part[0] = l_part[1] = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  }
};

template <class Op>
__device__ __forceinline__ void attn_tile_swap(AttnAccS &A, uint32_t k_t, uint32_t v_t, const uint4 (&qh)[4], const int (&lim)[2],
                                               bool mask) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // (the same permutation of the 32 dimensions of a k block on both operands: a lane's 16 bytes are dimensions 8t .. 8t + 7)
  float c[4] = {0.f, 0.f, 0.f, 0.f}, c2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int kb = 0; kb < 4; ++kb) {
    const uint4 K0 = lds128(k_t + ad_part(g, kb * 4 + t)), K1 = lds128(k_t + ad_part(g + 8, kb * 4 + t));
    Op::mma(c, K0.x, K1.x, K0.y, K1.y, qh[kb].x, qh[kb].y);
    Op::mma(c2, K0.z, K1.z, K0.w, K1.w, qh[kb].z, qh[kb].w);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    c[e] += c2[e];
    if (mask && g + (e >> 1) * 8 >= lim[e & 1]) c[e] = -INFINITY;
  }
  float corr[2];
#pragma unroll
  for (int hq = 0; hq < 2; ++hq) {
    // over the tile's 16 keys: the 8 lanes that share t
    float mx = fmaxf(c[hq], c[hq + 2]);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    const float m_new = attn_level(A.top[hq], mx);
    corr[hq] = m_new > -INFINITY ? __expf(A.m_run[hq] - m_new) : 1.f;
    A.m_run[hq] = m_new;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) c[e] = c[e] > -INFINITY ? __expf(c[e] - A.m_run[e & 1]) : 0.f;
  A.l_part[0] = A.l_part[0] * corr[0] + c[0] + c[2];
  A.l_part[1] = A.l_part[1] * corr[1] + c[1] + c[3];
  // P^T as the B operand (k = key, n = query row): lane (g, t) needs keys 2t, 2t + 1 (and + 8) of query
  // row g; they sit in lanes (2t, g / 2) and (2t + 1, g / 2), element g & 1 of each pair
  const uint32_t x = Op::pack2(c[0], c[1]), y = Op::pack2(c[2], c[3]);
  const int src_a = (2 * t) * 4 + (g >> 1), src_b = (2 * t + 1) * 4 + (g >> 1);
  const uint32_t xa = __shfl_sync(0xffffffffu, x, src_a), xb = __shfl_sync(0xffffffffu, x, src_b);
  const uint32_t ya = __shfl_sync(0xffffffffu, y, src_a), yb = __shfl_sync(0xffffffffu, y, src_b);
  const uint32_t sel = (g & 1) ? 0x7632u : 0x5410u;       // high or low halves of the two words
  const uint32_t b0 = __byte_perm(xa, xb, sel), b1 = __byte_perm(ya, yb, sel);
  // O^T += V^T P^T: A = V^T (m = dimension, k = key) through ldmatrix.trans of the key rows
  const int mi = lane >> 3, rr = (mi >> 1) * 8 + (lane & 7);
#pragma unroll
  for (int dt = 0; dt < 8; ++dt) {
    uint32_t a0, a1, a2, a3;
    ldmatrix_x4_trans(v_t + ad_part(rr, dt * 2 + (mi & 1)), a0, a1, a2, a3);
    A.o[dt][0] *= corr[0]; A.o[dt][1] *= corr[1]; A.o[dt][2] *= corr[0]; A.o[dt][3] *= corr[1];
    Op::mma(A.o[dt], a0, a1, a2, a3, b0, b1);
  }
}

// The same with 9 to 16 query rows, on the M axis: thread (g, t) holds rows g, g + 8 and keys (dimensions) 2t, 2t + 1 of
// every 8.  lim[h]: keys row g + 8 h sees.
struct AttnAccW {
  float m_run[2], l_part[2], top[2];
  float o[16][4];
  __device__ __forceinline__ void clear() {
    m_run[0] = m_run[1] = top[0] = top[1] = -INFINITY;
    l_part[0] = l_part[1] = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  }
};

template <class Op>
__device__ __forceinline__ void attn_tile_rows(AttnAccW &A, uint32_t k_t, uint32_t v_t, const uint4 (&qh)[4][2], const int (&lim)[2],
                                               bool mask) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float c[2][4], c2[2][4];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    c[nt][0] = c[nt][1] = c[nt][2] = c[nt][3] = 0.f;
    c2[nt][0] = c2[nt][1] = c2[nt][2] = c2[nt][3] = 0.f;
  }
#pragma unroll
  for (int kb = 0; kb < 4; ++kb) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const uint4 Kh = lds128(k_t + ad_part(nt * 8 + g, kb * 4 + t));
      Op::mma(c[nt], qh[kb][0].x, qh[kb][1].x, qh[kb][0].y, qh[kb][1].y, Kh.x, Kh.y);
      Op::mma(c2[nt], qh[kb][0].z, qh[kb][1].z, qh[kb][0].w, qh[kb][1].w, Kh.z, Kh.w);
    }
  }
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      c[nt][e] += c2[nt][e];
      if (mask && nt * 8 + 2 * t + (e & 1) >= lim[e >> 1]) c[nt][e] = -INFINITY;
    }
  }
  float corr[2];
#pragma unroll
  for (int hr = 0; hr < 2; ++hr) {
    float mx = fmaxf(fmaxf(c[0][2 * hr], c[0][2 * hr + 1]), fmaxf(c[1][2 * hr], c[1][2 * hr + 1]));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float m_new = attn_level(A.top[hr], mx);
    corr[hr] = m_new > -INFINITY ? __expf(A.m_run[hr] - m_new) : 1.f;
    A.m_run[hr] = m_new;
  }
  float psum[2] = {0.f, 0.f};
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      c[nt][e] = c[nt][e] > -INFINITY ? __expf(c[nt][e] - A.m_run[e >> 1]) : 0.f;
      psum[e >> 1] += c[nt][e];
    }
  }
  A.l_part[0] = A.l_part[0] * corr[0] + psum[0];
  A.l_part[1] = A.l_part[1] * corr[1] + psum[1];
  uint32_t ah[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) ah[i] = Op::pack2(c[i >> 1][(i & 1) * 2], c[i >> 1][(i & 1) * 2 + 1]);
  const int mi = lane >> 3, rr = (mi & 1) * 8 + (lane & 7);
#pragma unroll
  for (int d2 = 0; d2 < 8; ++d2) {
    uint32_t b0, b1, b2, b3;
    ldmatrix_x4_trans(v_t + ad_part(rr, d2 * 2 + (mi >> 1)), b0, b1, b2, b3);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      A.o[2 * d2 + h][0] *= corr[0]; A.o[2 * d2 + h][1] *= corr[0]; A.o[2 * d2 + h][2] *= corr[1]; A.o[2 * d2 + h][3] *= corr[1];
    }
    Op::mma(A.o[2 * d2], ah[0], ah[1], ah[2], ah[3], b0, b1);
    Op::mma(A.o[2 * d2 + 1], ah[0], ah[1], ah[2], ah[3], b2, b3);
  }
}

// The warps' level, sum and unnormalised output go to shared memory as [warp][query row][dimension].
__device__ __forceinline__ void attn_acc_store(AttnAccS &A, float *o_s, float *red_m, float *red_l, int nQ) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int hq = 0; hq < 2; ++hq) {
    float l = A.l_part[hq];
    l += __shfl_xor_sync(0xffffffffu, l, 4);
    l += __shfl_xor_sync(0xffffffffu, l, 8);
    l += __shfl_xor_sync(0xffffffffu, l, 16);
    if (g == 0) { red_m[warp * PK_QR + 2 * t + hq] = A.m_run[hq]; red_l[warp * PK_QR + 2 * t + hq] = l; }
  }
#pragma unroll
  for (int dt = 0; dt < 8; ++dt) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int q = 2 * t + (e & 1), d = dt * 16 + g + (e >> 1) * 8;
      if (q < nQ) o_s[(warp * PK_QR + q) * PK_OROW + d] = A.o[dt][e];
    }
  }
}
__device__ __forceinline__ void attn_acc_store(AttnAccW &A, float *o_s, float *red_m, float *red_l, int nQ) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int hr = 0; hr < 2; ++hr) {
    float l = A.l_part[hr];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    const int q = g + 8 * hr;
    if (t == 0) { red_m[warp * PK_QR + q] = A.m_run[hr]; red_l[warp * PK_QR + q] = l; }
    if (q < nQ) {
#pragma unroll
      for (int dt = 0; dt < 16; ++dt)
        *reinterpret_cast<float2 *>(o_s + (warp * PK_QR + q) * PK_OROW + dt * 8 + 2 * t) = make_float2(A.o[dt][2 * hr], A.o[dt][2 * hr + 1]);
    }
  }
}

// The key units of a launch: `items` = (sequence, kv head, row block) triples of `per_item` units each, one line of
// items * per_item units in equal shares for n_blocks blocks.
struct AttnShares {
  int per_item, n_blocks;
  long long total;
  __device__ __forceinline__ int begin(int block) const { return (int)(total * block / n_blocks); }
  // the block that holds unit u
  __device__ __forceinline__ int holder(int u) const { return (int)((((long long)u + 1) * n_blocks - 1) / total); }
};

// Loads from the shared memory of another block of the cluster (cluster_address).
__device__ __forceinline__ float4 ld_cluster4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_cluster2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
constexpr int AD_MAX_CLUSTER = 8;

// Where the form of a model's layer puts its results: the O projection's activation blocks.
struct AttnBlocks {
  uint4 *blocks;
  ActTiles T;
};

// CLUSTER: one cluster to an item, its units cut into equal pieces for the cluster's blocks, which merge their results through
// distributed shared memory: into `part_o` = out [B*R][nq][128], or, the fused form, into the O projection's activation
// blocks.  One launch, no partial results in memory.  (Merging by the last block of an item to arrive at a counter in
// memory instead: a layer of 8 sequences 2 us slower than with the merge as a launch of its own.)  See attn_cluster_ranks.
// qkv [B*R][ldq]: FUSED: the raw q | k | v rows of the QKV projection (AttnFuse); else q heads already normalised and
// rotated (not scaled) and K and V of the new rows already in the cache.  Cache [b][kv head][max_seq][128], 16 bit.
// part_o / part_ml: `nsplit` slots per (row, head); the pieces of an item take slots 0, 1, ...; the rest are marked empty.
template <class Op, bool FUSED = false, bool CLUSTER = false>
__global__ void __launch_bounds__(AD_THREADS, 2)
attn_decode_kernel(const float *qkv, int ldq, const void *kc, const void *vc, int max_seq,
                   int nq, int nkv, int B, int R, int RB, const int *__restrict__ pos0_ptr, int pos0_val, float *part_o,
                   float *part_ml, int nsplit, AttnFuse F = AttnFuse{nullptr, nullptr, nullptr, 0.f},
                   AttnBlocks O = AttnBlocks{nullptr, ActTiles{}}) {
  extern __shared__ __align__(1024) unsigned char sc[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int G = nq / nkv, n_rb = (R + RB - 1) / RB;
  // The next kernel may become resident (see pdl_enter).  With the fused step a3 the keys in front of the new rows come from
  // earlier passes: the first tiles are requested before the projection in front is waited for.  The position is older
  // than the last plainly launched kernel (the rotary table's).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!FUSED) asm volatile("griddepcontrol.wait;" ::: "memory");
  bool waited = !FUSED;
  const int pos0 = pos0_ptr ? *pos0_ptr : pos0_val;
  AttnShares sh;
  sh.per_item = (pos0 + R + AD_UNIT - 1) / AD_UNIT;
  sh.total = (long long)B * nkv * n_rb * sh.per_item;
  sh.n_blocks = (int)min((long long)gridDim.x, sh.total);             // no empty shares: pieces of an item are consecutive blocks
  int n_ranks = 1, rank = 0;
  if (CLUSTER) {
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n_ranks));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  }
  if (!CLUSTER && (int)blockIdx.x >= sh.n_blocks) {
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");    // this grid's end stands for the end of those before it
    return;
  }
  const int u_item = CLUSTER ? (int)blockIdx.x / n_ranks * sh.per_item : 0;
  const int u_end = CLUSTER ? u_item + sh.per_item * (rank + 1) / n_ranks : sh.begin(blockIdx.x + 1);
  const uint32_t ring = smem_u32(sc + AD_RING) + warp * AD_STAGES * AD_SLOT, q_t = smem_u32(sc + AD_Q);
  float *const o_s = reinterpret_cast<float *>(sc + AD_OS), *const red_m = reinterpret_cast<float *>(sc + AD_RED);
  float *const red_l = red_m + AD_WARPS * PK_QR;
  const float scale = rsqrtf((float)PK_D);

  for (int u = CLUSTER ? u_item + sh.per_item * rank / n_ranks : sh.begin(blockIdx.x); CLUSTER || u < u_end;) {
    // one piece: units [t0, t1) of an item
    const int item = CLUSTER ? (int)blockIdx.x / n_ranks : u / sh.per_item, t0 = u - item * sh.per_item, t1 = min(sh.per_item, t0 + u_end - u);
    const int piece = CLUSTER ? 0 : blockIdx.x - sh.holder(item * sh.per_item);
    u += t1 - t0;
    const int rb = item % n_rb, kvh = (item / n_rb) % nkv, b = item / n_rb / nkv;
    const int r0 = rb * RB, r1 = min(R, r0 + RB), nQ = (r1 - r0) * G;
    const int n_keys = min(pos0 + r1, t1 * AD_UNIT);                   // the block's last row sees position pos0 + r1 - 1
    const size_t head_off = ((size_t)b * nkv + kvh) * max_seq * PK_D;
    const typename Op::T *kb = reinterpret_cast<const typename Op::T *>(kc) + head_off;
    const typename Op::T *vb = reinterpret_cast<const typename Op::T *>(vc) + head_off;
    const int n_cached = FUSED ? min(n_keys, pos0) : n_keys;          // keys that come from the cache
    // this warp's tile of unit i: keys i * 64 + 16 warp ..; rows past the cached keys are filled with zeros
    // (P = 0 times stale bits must stay 0)
    auto fetch = [&](int i, int slot) {
      if (i < t1) {
        const int key0 = i * AD_UNIT + warp * AD_KEYS;
        const uint32_t dst = ring + slot * AD_SLOT;
        const int part = lane & 15;
#pragma unroll
        for (int j = 0; j < AD_KEYS / 2; ++j) {
          const int row = 2 * j + (lane >> 4), key = key0 + row, bytes = key < n_cached ? 16 : 0;
          const size_t src = (size_t)(key < n_cached ? key : 0) * PK_D + part * 8;
          const uint32_t off = ad_part(row, part);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + off), "l"(kb + src), "r"(bytes) : "memory");
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + AD_KEYS * 256 + off), "l"(vb + src), "r"(bytes) : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");             // an empty group past the last tile keeps the counts uniform
    };
#pragma unroll
    for (int s = 0; s < AD_STAGES; ++s) fetch(t0 + s, s);
    if (!waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      waited = true;
    }

    // query rows (beyond nQ zero): row qi = (position r0 + qi / G, head kvh*G + qi % G), scaled by 1/sqrt(d)
    for (int qi = warp; qi < PK_QR; qi += AD_WARPS) {
      typename Op::T *qh = reinterpret_cast<typename Op::T *>(sc + AD_Q + qi * PK_QROW);
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (qi < nQ) {
        const float *src = qkv + (size_t)(b * R + r0 + qi / G) * ldq + (size_t)(kvh * G + qi % G) * PK_D;
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = src[lane + 32 * j];
        if (FUSED) head_norm_rope<PK_D>(F.w_qn, F.table + (size_t)(r0 + qi / G) * (PK_D / 2), F.eps, lane, v);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) qh[lane + 32 * j] = Op::from_float(v[j] * scale);
    }
    // fused form: the pass's rows r_lo .. r_hi - 1 sit at positions inside this piece; their K and V come from the
    // projection's output, and the piece of the row block that owns a position appends it to the cache
    const int r_lo = FUSED ? max(0, t0 * AD_UNIT - pos0) : 0, r_hi = FUSED ? max(r_lo, min(r1, t1 * AD_UNIT - pos0)) : 0;
    if (FUSED) {
      for (int task = warp; task < 2 * (r_hi - r_lo); task += AD_WARPS) {
        const int r = r_lo + (task >> 1), is_v = task & 1;
        const float *src = qkv + (size_t)(b * R + r) * ldq + (size_t)(nq + (is_v ? nkv : 0) + kvh) * PK_D;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = src[lane + 32 * j];
        if (!is_v) head_norm_rope<PK_D>(F.w_kn, F.table + (size_t)r * (PK_D / 2), F.eps, lane, v);
        typename Op::T *row = reinterpret_cast<typename Op::T *>(sc + AD_NEW) + ((is_v ? AD_MAX_NEW : 0) + r - r_lo) * PK_D;
        typename Op::T *cache = const_cast<typename Op::T *>(is_v ? vb : kb) + (size_t)(pos0 + r) * PK_D;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const typename Op::T h = Op::from_float(v[j]);
          row[lane + 32 * j] = h;
          if (r >= r0) cache[lane + 32 * j] = h;
        }
      }
    }
    __syncthreads();                                                    // query rows and new rows written
    // the pass's own rows of a tile (its copies filled them with zeros)
    auto place_new = [&](int key0, uint32_t dst) {
      if (!FUSED || key0 + AD_KEYS <= pos0 || key0 >= n_keys) return;
      const int first = max(0, pos0 - key0), n_t = min(AD_KEYS, n_keys - key0);
      for (int c = lane + first * 32; c < n_t * 32; c += 32) {
        const int row = c >> 5, part = c & 15, is_v = (c >> 4) & 1;
        const uint4 val = *reinterpret_cast<const uint4 *>(sc + AD_NEW + ((is_v ? AD_MAX_NEW : 0) + key0 + row - pos0 - r_lo) * 256 + part * 16);
        sts128(dst + (is_v ? AD_KEYS * 256 : 0) + ad_part(row, part), val);
      }
      __syncwarp();
    };
    // the key loop of one form of the tile arithmetic: multiply(K tile, V tile, keys the row positions see, mask needed)
    auto key_loop = [&](auto &&multiply) {
      int slot = 0;
      for (int i = t0; i < t1; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(AD_STAGES - 1) : "memory");
        __syncwarp();
        const int key0 = i * AD_UNIT + warp * AD_KEYS;
        const uint32_t k_t = ring + slot * AD_SLOT;
        if (key0 < n_keys) {
          place_new(key0, k_t);
          multiply(k_t, k_t + AD_KEYS * 256, key0, key0 + AD_KEYS > pos0 + r0 + 1 || key0 + AD_KEYS > n_keys);
        }
        __syncwarp();                                                   // the slot is free
        fetch(i + AD_STAGES, slot);
        if (++slot == AD_STAGES) slot = 0;
      }
    };
    // keys a query row sees, from a tile's first key: up to its position and the end of the piece
    auto limit = [&](int q, int key0) { return min(n_keys, pos0 + r0 + q / G + 1) - key0; };
    if (nQ <= 8) {
      AttnAccS A;
      A.clear();
      uint4 qs[4];
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) qs[k4] = lds128(q_t + g * PK_QROW + k4 * 64 + t * 16);
      const int lim0[2] = {limit(2 * t, 0), limit(2 * t + 1, 0)};
      key_loop([&](uint32_t k_t, uint32_t v_t, int key0, bool mask) {
        const int lim[2] = {lim0[0] - key0, lim0[1] - key0};
        attn_tile_swap<Op>(A, k_t, v_t, qs, lim, mask);
      });
      attn_acc_store(A, o_s, red_m, red_l, nQ);
    } else {
      AttnAccW A;
      A.clear();
      uint4 qh[4][2];
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        qh[k4][0] = lds128(q_t + g * PK_QROW + k4 * 64 + t * 16);
        qh[k4][1] = lds128(q_t + (g + 8) * PK_QROW + k4 * 64 + t * 16);
      }
      const int lim0[2] = {limit(g, 0), limit(g + 8, 0)};
      key_loop([&](uint32_t k_t, uint32_t v_t, int key0, bool mask) {
        const int lim[2] = {lim0[0] - key0, lim0[1] - key0};
        attn_tile_rows<Op>(A, k_t, v_t, qh, lim, mask);
      });
      attn_acc_store(A, o_s, red_m, red_l, nQ);
    }
    __syncthreads();
    // per query row: the piece's largest level and its sum, and the factor each warp's share is scaled by (a warp without keys: 0)
    if ((int)threadIdx.x < nQ) {
      const int qi = threadIdx.x;
      float m = -INFINITY;
#pragma unroll
      for (int w = 0; w < AD_WARPS; ++w) m = fmaxf(m, red_m[w * PK_QR + qi]);
      float l = 0.f;
#pragma unroll
      for (int w = 0; w < AD_WARPS; ++w) {
        const float mw = red_m[w * PK_QR + qi];
        const float f = mw > -INFINITY ? __expf(mw - m) : 0.f;
        l += red_l[w * PK_QR + qi] * f;
        red_l[w * PK_QR + qi] = f;
      }
      if (CLUSTER) reinterpret_cast<float2 *>(sc + AD_RING + PK_QR * PK_D * 4)[qi] = make_float2(m, l);          // (the ring is free)
      const size_t slot = ((size_t)(b * R + r0 + qi / G) * nq + kvh * G + qi % G) * nsplit + piece;
      if (!CLUSTER) *reinterpret_cast<float2 *>(part_ml + slot * 2) = make_float2(m, l);
      if (!CLUSTER && t1 == sh.per_item)                                // the item's last piece
        for (int e = piece + 1; e < nsplit; ++e) *reinterpret_cast<float2 *>(part_ml + (slot + e - piece) * 2) = make_float2(-INFINITY, 0.f);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < nQ * (PK_D / 4); idx += AD_THREADS) {
      const int qi = idx / (PK_D / 4), d4 = idx % (PK_D / 4);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < AD_WARPS; ++w) {
        const float f = red_l[w * PK_QR + qi];
        if (f != 0.f) {
          const float4 v = *reinterpret_cast<const float4 *>(o_s + (w * PK_QR + qi) * PK_OROW + d4 * 4);
          acc.x += v.x * f; acc.y += v.y * f; acc.z += v.z * f; acc.w += v.w * f;
        }
      }
      if (CLUSTER) {
        reinterpret_cast<float4 *>(sc + AD_RING)[idx] = acc;
        continue;
      }
      const size_t slot = ((size_t)(b * R + r0 + qi / G) * nq + kvh * G + qi % G) * nsplit + piece;
      *reinterpret_cast<float4 *>(part_o + slot * PK_D + d4 * 4) = acc;
    }
    if (CLUSTER) {
      asm volatile("barrier.cluster.arrive.release;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
      // a thread to PER values of a query row: 4 of the output, or 8 (a unit) of the blocks
      constexpr int PER = FUSED ? 8 : 4, V = PER / 4;
      for (int idx = rank * AD_THREADS + threadIdx.x; idx < nQ * (PK_D / PER); idx += n_ranks * AD_THREADS) {
        const int qi = idx / (PK_D / PER), row = b * R + r0 + qi / G, head = kvh * G + qi % G;
        const uint32_t o_a = smem_u32(sc + AD_RING) + idx * PER * 4, ml_a = smem_u32(sc + AD_RING + PK_QR * PK_D * 4) + qi * 8;
        float2 ml[AD_MAX_CLUSTER];
        float4 o[AD_MAX_CLUSTER][V];
        float m = -INFINITY;
#pragma unroll
        for (int s = 0; s < AD_MAX_CLUSTER; ++s)
          if (s < n_ranks) {
            ml[s] = ld_cluster2(cluster_address(ml_a, s));
#pragma unroll
            for (int i = 0; i < V; ++i) o[s][i] = ld_cluster4(cluster_address(o_a + i * 16, s));
          }
#pragma unroll
        for (int s = 0; s < AD_MAX_CLUSTER; ++s)
          if (s < n_ranks && ml[s].y > 0.f) m = fmaxf(m, ml[s].x);
        float l = 0.f, f[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) f[i] = 0.f;
#pragma unroll
        for (int s = 0; s < AD_MAX_CLUSTER; ++s)
          if (s < n_ranks && ml[s].y > 0.f) {
            const float w = __expf(ml[s].x - m);
            l += ml[s].y * w;
#pragma unroll
            for (int i = 0; i < V; ++i) {
              f[4 * i] += o[s][i].x * w; f[4 * i + 1] += o[s][i].y * w;
              f[4 * i + 2] += o[s][i].z * w; f[4 * i + 3] += o[s][i].w * w;
            }
          }
        const float inv = 1.f / l;
#pragma unroll
        for (int i = 0; i < PER; ++i) f[i] *= inv;
        if constexpr (FUSED) {
          const int k = head * PK_D + idx % (PK_D / PER) * PER;
          store_hi_lo(f, O.blocks + O.T.unit(row, k / TG_KB, k % TG_KB / 8), O.T.lo_offset());
        } else {
          reinterpret_cast<float4 *>(part_o)[((size_t)row * nq + head) * (PK_D / 4) + idx % (PK_D / 4)] = make_float4(f[0], f[1], f[2], f[3]);
        }
      }
      asm volatile("barrier.cluster.arrive.release;" ::: "memory");       // no block leaves while another reads from it
      asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
      break;
    }
    __syncthreads();                                                    // outputs, factors and query rows consumed
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Blocks of a launch (two per SM, one wave) and the slots a (row, head) needs for its pieces; at most max_slots.
struct AttnDecodePlan { int n_blocks, nsplit; };
inline AttnDecodePlan attn_decode_plan(int n_sms, int items, int max_units, int max_slots) {
  // a share of total / n units touches at most n / items + 2 pieces of an item (n / items where that is whole), and
  // an item has no more pieces than units
  auto pieces = [&](int n) { return std::min(max_units, n % items == 0 ? n / items : n / items + 2); };
  AttnDecodePlan p;
  p.n_blocks = 2 * n_sms;
  if ((long long)items * max_units < p.n_blocks) p.n_blocks = items * max_units;
  if (pieces(p.n_blocks) > max_slots) p.n_blocks = items * std::min(max_slots, max_units);
  p.nsplit = pieces(p.n_blocks);
  return p;
}

// The same step for an fp32 cache in plain FMAs (fp32 accuracy on the tensor cores would take three products): the tile arithmetic of the pass kernel's fp32
// attention stage, one 64-key tile in shared memory per block and two blocks per SM, so that one
// block's copies run under the other's arithmetic.
using StepF32Map = AttnF32Map<64>;
constexpr int ATTN_F32_SMEM = StepF32Map::NEW;           // K and V tile, Q, partial scores, running max / sum / rescale factor

__global__ void __launch_bounds__(PK_THREADS, 2)
attn_f32_kernel(const float *qkv, int ldq, const float *__restrict__ kc, const float *__restrict__ vc, int max_seq,
                int nq, int nkv, int R, int RB, int CH, const int *__restrict__ pos0_ptr, int pos0_val, float *__restrict__ part_o,
                float *__restrict__ part_ml, int nsplit) {
  pdl_enter();
  extern __shared__ __align__(1024) unsigned char sc[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = nq / nkv, n_rb = (R + RB - 1) / RB;
  const int split = blockIdx.x, kvh = blockIdx.y / n_rb, rb = blockIdx.y % n_rb, b = blockIdx.z;
  const int r0 = rb * RB, r1 = min(R, r0 + RB), nQ = (r1 - r0) * G;
  const int pos0 = pos0_ptr ? *pos0_ptr : pos0_val;
  const int j0 = split * CH, j1 = min(j0 + CH, pos0 + r1);      // the last row of the block sees position pos0 + r1 - 1
  if (j0 >= j1) {                                                 // empty slice: mark and leave
    for (int qi = threadIdx.x; qi < nQ; qi += PK_THREADS) {
      const size_t slot = ((size_t)(b * R + r0 + qi / G) * nq + kvh * G + qi % G) * nsplit + split;
      part_ml[slot * 2] = -INFINITY;
      part_ml[slot * 2 + 1] = 0.f;
    }
    return;
  }
  // Q rows, scaled by 1/sqrt(d): row qi = (position r0 + qi / G, head kvh*G + qi % G)
  const float scale = rsqrtf((float)PK_D);
  for (int qi = warp; qi < nQ; qi += PK_WARPS) {
    const float *src = qkv + (size_t)(b * R + r0 + qi / G) * ldq + (size_t)(kvh * G + qi % G) * PK_D;
    float *dst = reinterpret_cast<float *>(sc + StepF32Map::Q) + qi * PK_D;
#pragma unroll
    for (int j = 0; j < 4; ++j) dst[lane + 32 * j] = __ldcg(src + lane + 32 * j) * scale;
  }
  float *const m_run = reinterpret_cast<float *>(sc + StepF32Map::STAT), *const l_run = m_run + PK_QR;
  if ((int)threadIdx.x < PK_QR) { m_run[threadIdx.x] = -INFINITY; l_run[threadIdx.x] = 0.f; }
  const float *kb = kc + (((size_t)b * nkv + kvh) * max_seq + j0) * PK_D;
  const float *vb = vc + (((size_t)b * nkv + kvh) * max_seq + j0) * PK_D;
  float acc[PK_QR][4];
#pragma unroll
  for (int q = 0; q < PK_QR; ++q) acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f;
  const int n_keys = j1 - j0;
  // The K and the V tile are loaded as two groups of asynchronous copies, each re-issued for the
  // next tile as soon as the step that reads it is over: K of tile i + 1 arrives under the
  // softmax step and P V of tile i, V of tile i + 1 under the scores of tile i + 1.
  auto fetch = [&](const float *rows, int tile0, int dst_off, int row_bytes) {
    const int n_t = min(PK_TK, n_keys - tile0);
#pragma unroll 1
    for (int c = threadIdx.x; c < n_t * 32; c += PK_THREADS) {
      const int row = c >> 5, u = c & 31;
      if (tile0 < n_keys) cp_async16(smem_u32(sc) + dst_off + row * row_bytes + u * 16, rows + (size_t)(tile0 + row) * PK_D + u * 4);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");      // an empty group past the last tile keeps the counts uniform
  };
  fetch(kb, 0, StepF32Map::K, PK_F_KROW);
  fetch(vb, 0, StepF32Map::V, PK_D * 4);
#pragma unroll 1
  for (int tile0 = 0; tile0 < n_keys; tile0 += PK_TK) {
    const int n_t = min(PK_TK, n_keys - tile0);
    asm volatile("cp.async.wait_group 1;" ::: "memory");      // K of this tile (V may still be on its way)
    __syncthreads();                                      // ... from every thread; the first time also Q and the statistics
    attn_f32_scores<StepF32Map>(sc, nQ, n_t);
    __syncthreads();                                      // K consumed
    fetch(kb, tile0 + PK_TK, StepF32Map::K, PK_F_KROW);
    // every key comes from the cache: key index i sits at position j0 + i
    attn_f32_softmax<StepF32Map>(sc, nQ, G, n_t, tile0, 0x7fffffff, j0, 0, pos0 + r0);
    asm volatile("cp.async.wait_group 1;" ::: "memory");      // V of this tile (the next K may still be on its way)
    __syncthreads();                                      // probabilities and V from every thread
    attn_f32_pv<StepF32Map>(sc, acc, nQ, n_t);
    __syncthreads();                                      // V and the probabilities consumed
    fetch(vb, tile0 + PK_TK, StepF32Map::V, PK_D * 4);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  attn_f32_combine<StepF32Map>(sc, acc, nQ, G, b * R + r0, kvh * G, nq, nsplit, split, part_o, part_ml);
}

}  // namespace dmtd
