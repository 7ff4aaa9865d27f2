// Causal attention of a chunk of new positions per sequence (the prefill, Section 2.2: all prompt rows through all
// layers; the scoring pass of Eq. 1-5) on the 5th-generation tensor cores, for a 16-bit KV cache and head_dim 128.
//
// A block takes 128 query rows of one (sequence, kv head): 128 / G consecutive positions x the G query heads of the kv
// head, and walks the keys they see in tiles of 128.  Per tile: S = Q K^T (M = 128 rows, N = 128 keys, accumulators in
// tensor memory), softmax by four warps (a thread owns a row: no shuffles), P back into tensor memory as the A operand
// of O += P V, accumulated in tensor memory over all tiles.  When a row's maximum grows, O would have to be scaled
// between two tiles; a row keeps an older maximum as its reference instead as long as the new one is less than 2^8
// above it (p then reaches 256, far inside both 16-bit types, and the sums are the same), so that O is read back
// and scaled in a few tiles only.
//
// Q, K and V lie in shared memory as rows of 64 values with the 128-byte swizzle, two halves of the head dimension one
// behind the other: K-major operands of S, and the same bytes are the N-major B operand of P V.  K and V tiles come
// by 16-byte asynchronous copies (the cache's rows are 256 bytes; the swizzle keeps the copies free of bank
// conflicts), K of the next tile under the softmax of this one, V under the next S.  One tile of each and half of the
// tensor memory (S 128 columns, P over them, O 128): two blocks per SM, one's products under the other's softmax.
//
// Bound: the chain of one tile, 4030 cycles (S 770, softmax 1870, hand-over 550, P V 850) with two blocks per SM beside
// each other, i.e. 2015 per tile and SM against 1350 of the tensor pipe.  1024 positions behind 8000 keys: 209 us
// (680 TFLOP/s); one sequence of 512 tokens (32 query and 8 kv heads): 18 us per layer, 69 us with the kernel
// before this one, which ran the same tiles on mma.sync, each warp re-reading K and V from shared memory for 16 rows.
//
// Warps 0-3 load Q, run the softmax and store; warp 4 issues the MMAs; warp 5 copies K and V.  Every barrier wait is bounded; the
// tensor-memory allocation waits only for grids in front of this one (see pdl_enter in the kernel).
#pragma once

#include "gemm_tc05.cuh"
#include "kernels.cuh"
#include "pass_attention.cuh"

namespace dmtd {

constexpr int AP_M = 128;                        // query rows per block
constexpr int AP_TK = 128;                       // keys per tile
constexpr int AP_LOADERS = 32;                   // copying threads (six warps a block: 168 registers a thread, seven would leave 128)
constexpr int AP_THREADS = AP_M + 32 + AP_LOADERS;
constexpr int AP_HALF = 128 * 128;               // bytes of one half (64 of the 128 dimensions) of 128 rows
constexpr int AP_Q = 0, AP_K = 2 * AP_HALF, AP_V = 4 * AP_HALF, AP_BARS = 6 * AP_HALF;
constexpr int AP_SMEM = AP_BARS + 64;
constexpr int AP_TMEM_COLS = 256;                // S (P over it) and O
static_assert(TG_MIN_SMEM + AP_SMEM + 2 * 1024 > 228 * 1024 && 2 * (TG_MIN_SMEM + 1024) > 228 * 1024,
              "a GEMM block shares its SM with no other holder of tensor memory");
constexpr float AP_LOG2E = 1.4426950408889634f;
constexpr float AP_RESCALE_LOG2 = 8.f;           // a row's reference maximum may be this far (in powers of two) behind

struct AttnPrefillParams {
  const float *qkv;            // [B*R][ldq]: q heads normalised and rotated (not scaled)
  const void *kc, *vc;         // cache [b][kv head][max_seq][128], the chunk's K and V already in it
  int ldq, max_seq, nq, nkv, R;
  const int *pos0;
  float *out;                  // [B*R][ld] fp32, or
  int ld;
  uint4 *blocks;               // (if not null) the activation blocks of the O projection
  ActTiles T;
  int *error;
  long long wait_limit;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// byte offset of 16-byte part `part` (8 values; 0..15) of row `row` in a swizzled tile of two halves
__device__ __forceinline__ uint32_t ap_part(int row, int part) {
  return (uint32_t)((part >> 3) * AP_HALF + row * 128 + (((part & 7) ^ (row & 7)) << 4));
}
// shared-memory operand descriptor, 128-byte swizzle: 8-row groups 1024 bytes apart; lbo: between groups of 64 values
// along the contiguous axis (N-major operand only)
__device__ __forceinline__ uint64_t ap_desc(uint32_t addr, uint32_t lbo) {
  return umma_smem_desc(addr, lbo, 1024) | (2ull << 61);
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(addr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ float exp2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two floats at a time (a scheduler has one softmax warp of each block: issue slots count)
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

template <class Op>
__global__ void __launch_bounds__(AP_THREADS, 2) attn_prefill_kernel(const __grid_constant__ AttnPrefillParams P) {
  extern __shared__ __align__(1024) unsigned char sc[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = P.nq / P.nkv, lgG = 31 - __clz(G), QB = AP_M >> lgG;  // G is a power of two (it divides 128); positions per block
  const int kvh = blockIdx.y, b = blockIdx.z;
  const int r0 = blockIdx.x * QB, r1 = min(P.R, r0 + QB);
  const uint32_t smem = smem_u32(sc);
  // tile i completes phase i of every barrier
  const uint32_t bar_k = smem + AP_BARS, bar_v = bar_k + 8;           // K / V tile in shared memory
  const uint32_t bar_s = bar_k + 16, bar_p = bar_k + 24, bar_o = bar_k + 32;   // S computed; P stored; P V computed
  const uint32_t bar_q = bar_k + 40;                                  // Q in shared memory (once)
  uint32_t *const tmem_slot = reinterpret_cast<uint32_t *>(sc + AP_BARS + 48);
  volatile int *const gave_up = reinterpret_cast<volatile int *>(sc + AP_BARS + 52);

  if (threadIdx.x == 0) {
    mbar_init(bar_k, AP_LOADERS);
    mbar_init(bar_v, AP_LOADERS);
    mbar_init(bar_s, 1);
    mbar_init(bar_p, AP_M);
    mbar_init(bar_o, 1);
    mbar_init(bar_q, AP_M);
    *gave_up = 0;
    fence_mbar_init();
  }
  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(AP_TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // The dependent grid (the O projection's GEMM) takes tensor memory before it waits for this one, and an allocation waits
  // without a limit: this block lets it in only now that it holds its own columns.
  pdl_enter();
  const uint32_t tmem_s = *tmem_slot, tmem_o = tmem_s + 128;
  const int pos0 = *P.pos0;
  const int n_keys = pos0 + r1, n_tiles = (n_keys + AP_TK - 1) / AP_TK;     // the block's last position sees keys [0, pos0 + r1)

  if (warp >= 5) {
    // ---- copies: K(i) once S(i - 1) is computed, V(i) once P V (i - 1) is
    const int lt = threadIdx.x - (AP_M + 32);
    const size_t head_off = ((size_t)b * P.nkv + kvh) * P.max_seq * 128;
    const typename Op::T *kb = reinterpret_cast<const typename Op::T *>(P.kc) + head_off;
    const typename Op::T *vb = reinterpret_cast<const typename Op::T *>(P.vc) + head_off;
    // rows past the last key are filled with zeros (P = 0 times stale bits must stay 0)
    auto fetch = [&](const typename Op::T *base, int tile0, uint32_t dst) {
      const int part = lt & 15;
#pragma unroll 8
      for (int row = lt >> 4; row < AP_TK; row += AP_LOADERS / 16) {
        const int key = tile0 + row;
        const int bytes = key < n_keys ? 16 : 0;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + ap_part(row, part)),
                     "l"(base + (size_t)min(key, n_keys - 1) * 128 + part * 8), "r"(bytes)
                     : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    bool ok = true;
    for (int i = 0; i < n_tiles && ok; ++i) {
      if (i > 0) ok = tg_wait(bar_s, (i - 1) & 1, P);
      if (!ok) break;
      fetch(kb, i * AP_TK, smem + AP_K);
      if (i > 0) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");          // long done when P V (i - 1) is
        fence_proxy_async();
        mbar_arrive(bar_k);
        ok = tg_wait(bar_o, (i - 1) & 1, P);
        if (!ok) break;
        fetch(vb, i * AP_TK, smem + AP_V);
      } else {
        fetch(vb, i * AP_TK, smem + AP_V);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        fence_proxy_async();
        mbar_arrive(bar_k);
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      fence_proxy_async();
      mbar_arrive(bar_v);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp == 4) {
    // ---- MMA issuer
    constexpr uint32_t fmt = std::is_same<typename Op::T, __half>::value ? 0u : 1u;       // A and B of one type
    const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
    const uint32_t idesc_pv = idesc | (1u << 16);                                         // B is N-major
    bool ok = __all_sync(0xffffffffu, tg_wait(bar_q, 0, P));
    for (int i = 0; i < n_tiles && ok; ++i) {
      ok = __all_sync(0xffffffffu, tg_wait(bar_k, i & 1, P));
      if (i > 0) ok = __all_sync(0xffffffffu, ok && tg_wait(bar_o, (i - 1) & 1, P));      // P lies over S
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = (kk >> 2) * AP_HALF + (kk & 3) * 32;
          const uint64_t da = ap_desc(smem + AP_Q + off, 16), db = ap_desc(smem + AP_K + off, 16);
          const uint32_t acc = kk > 0 ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_s),
              "l"(da), "l"(db), "r"(idesc), "r"(acc)
              : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_s) : "memory");
      }
      __syncwarp();
      ok = __all_sync(0xffffffffu, tg_wait(bar_v, i & 1, P) && tg_wait(bar_p, i & 1, P));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {                              // 16 keys per MMA: two groups of 8 rows of V, 8 columns of P
          const uint64_t db = ap_desc(smem + AP_V + kk * 2048, AP_HALF);
          const uint32_t acc = (i > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_o),
              "r"(tmem_s + kk * 8), "l"(db), "r"(idesc_pv), "r"(acc)
              : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_o) : "memory");
      }
      __syncwarp();
    }
    if (!ok && lane == 0) { *gave_up = 1; __threadfence_block(); }
  } else {
    // ---- softmax: thread = query row = lane of tensor memory
    {
      // Q tile: row i = (position r0 + i / G, head kvh * G + i % G), scaled by 1/sqrt(d); rows past the chunk zero
      const float scale = rsqrtf(128.f);
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        const int qrow = warp * 32 + j, qr = r0 + (qrow >> lgG);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (qr < P.R)
          v = reinterpret_cast<const float4 *>(P.qkv + (size_t)(b * P.R + qr) * P.ldq + (size_t)(kvh * G + (qrow & (G - 1))) * 128)[lane];
        *reinterpret_cast<uint2 *>(sc + AP_Q + ap_part(qrow, lane >> 1) + (lane & 1) * 8) =
            make_uint2(Op::pack2(v.x * scale, v.y * scale), Op::pack2(v.z * scale, v.w * scale));
      }
      fence_proxy_async();
      mbar_arrive(bar_q);
    }
    const int row = threadIdx.x, r = r0 + (row >> lgG), my_pos = pos0 + r;
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    const uint32_t t_s = tmem_s + lane_off, t_o = tmem_o + lane_off;
    float m_ref = -INFINITY, l = 0.f;                                 // reference maximum (times log2 e) and running sum
    bool ok = true;
    for (int i = 0; i < n_tiles; ++i) {
      ok = __all_sync(0xffffffffu, tg_wait(bar_s, i & 1, P));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // keys of the tile this row sees: [0, lim); only the block's last tiles are cut
      const int lim = min(min(my_pos + 1, n_keys) - i * AP_TK, AP_TK);
      const bool cut = (i + 1) * AP_TK > pos0 + r0 + 1;                 // the same for all rows of the block
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};      // four chains: a dependent maximum takes four cycles
#pragma unroll
      for (int c0 = 0; c0 < AP_TK; c0 += 64) {
        uint32_t s[64];
        tmem_ld32(t_s + c0, *reinterpret_cast<uint32_t(*)[32]>(s));
        tmem_ld32(t_s + c0 + 32, *reinterpret_cast<uint32_t(*)[32]>(s + 32));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (cut) {
#pragma unroll
          for (int j = 0; j < 64; ++j) mx4[j & 3] = fmaxf(mx4[j & 3], c0 + j < lim ? __uint_as_float(s[j]) : -INFINITY);
        } else {
#pragma unroll
          for (int j = 0; j < 64; ++j) mx4[j & 3] = fmaxf(mx4[j & 3], __uint_as_float(s[j]));
        }
      }
      float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      mx *= AP_LOG2E;
      float alpha = 1.f;
      if (i == 0) {
        m_ref = mx;                                                   // key 0 is visible to every row
      } else {
        const bool grow = mx > m_ref + AP_RESCALE_LOG2;
        if (grow) { alpha = exp2_approx(m_ref - mx); m_ref = mx; l *= alpha; }
        if (__any_sync(0xffffffffu, grow)) {
          ok = __all_sync(0xffffffffu, tg_wait(bar_o, (i - 1) & 1, P));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
          for (int c0 = 0; c0 < 128; c0 += 16) {
            uint32_t o[16];
            tmem_ld16(t_o + c0, o);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
            tmem_st16(t_o + c0, o);
          }
        }
      }
      const uint64_t log2e2 = f2_pack(AP_LOG2E, AP_LOG2E), neg_m2 = f2_pack(-m_ref, -m_ref);
      uint64_t sum2[2] = {0ull, 0ull};
      // P over S: columns 16 q .. + 15 of P (keys 32 q ..) lie over columns of S that have been read by then
#pragma unroll
      for (int c0 = 0; c0 < AP_TK; c0 += 64) {
        uint32_t s[64];
        tmem_ld32(t_s + c0, *reinterpret_cast<uint32_t(*)[32]>(s));
        tmem_ld32(t_s + c0 + 32, *reinterpret_cast<uint32_t(*)[32]>(s + 32));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t p[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int k = 32 * h + 2 * j;
            float a, c;
            f2_unpack(f2_fma(f2_pack(__uint_as_float(s[k]), __uint_as_float(s[k + 1])), log2e2, neg_m2), a, c);
            a = exp2_approx(a);
            c = exp2_approx(c);
            if (cut) {
              a = c0 + k < lim ? a : 0.f;
              c = c0 + k + 1 < lim ? c : 0.f;
            }
            sum2[j & 1] = f2_add(sum2[j & 1], f2_pack(a, c));
            p[j] = Op::pack2(a, c);
          }
          tmem_st16(t_s + c0 / 2 + 16 * h, p);
        }
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(bar_p);
      float l0, l1;
      f2_unpack(f2_add(sum2[0], sum2[1]), l0, l1);
      l += l0 + l1;
    }
    // ---- O / l: fp32 rows, or hi and lo units of the O projection's activations
    if (ok && n_tiles > 0) ok = __all_sync(0xffffffffu, tg_wait(bar_o, (n_tiles - 1) & 1, P)) && !*gave_up;
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const float inv = 1.f / l;
      const int m = b * P.R + r, k0 = (kvh * G + (row & (G - 1))) * 128;
#pragma unroll 1
      for (int c0 = 0; c0 < 128; c0 += 16) {
        uint32_t o[16];
        tmem_ld16(t_o + c0, o);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (r < P.R) {
          float f[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) f[j] = __uint_as_float(o[j]) * inv;
          if (P.blocks) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int k = k0 + c0 + 8 * h;
              const float g[8] = {f[8 * h], f[8 * h + 1], f[8 * h + 2], f[8 * h + 3], f[8 * h + 4], f[8 * h + 5], f[8 * h + 6], f[8 * h + 7]};
              store_hi_lo(g, P.blocks + P.T.unit(m, k >> 6, (k >> 3) & 7), P.T.lo_offset());
            }
          } else {
            float4 *dst = reinterpret_cast<float4 *>(P.out + (size_t)m * P.ld + k0 + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j) dst[j] = make_float4(f[4 * j], f[4 * j + 1], f[4 * j + 2], f[4 * j + 3]);
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 4) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_s), "r"(AP_TMEM_COLS) : "memory");
  }
}

}  // namespace dmtd
