// Per-step kernels of the DMTD decode path (one launch per step of the layer).
// Every projection accumulates into its output with fp32 reductions, so split-K work
// division needs no second pass; the buffers that start at zero are cleared by the
// preceding "prep" kernel.
#pragma once

#include "common.cuh"

namespace dmtd {

// First statement of a kernel that is launched with programmatic stream serialisation: the kernel after it may become
// resident now (it does the same, or touches nothing but weights and the cache rows of earlier passes before it waits);
// nothing is read or written here before the kernels in front are complete.  Kernels without it are launched
// plainly: they start when everything before them is complete.
// What an earlier grid of such a chain writes (activations, partial results, the cache) changes while this one is
// running: such parameters are not __restrict__, which would allow loads that assume the opposite or are moved in front of
// the wait.  Weights, norm gains and the rotary table are; where a buffer is read by volatile instructions only (asynchronous
// copies, __ldcg), which keep their order to the wait, it may be.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int GEMV_THREADS = 256;
constexpr int GEMV_WARPS = GEMV_THREADS / 32;

// ------------------------------------------------------------------------------------
// Weight repacking (runs once, at create)
// ------------------------------------------------------------------------------------

// src [N][K] bf16 row-major -> atoms of tiles [tile0, tile0 + ceil(N/16)) of a stream that
// has n_tiles_total row tiles.  One thread per 16-byte chunk.
__global__ void pack_bf16_kernel(const __nv_bfloat16 *__restrict__ src, int N, int K,
                                 uint4 *__restrict__ dst, int tile0, int n_tiles_total, int aps,
                                 int n_slabs) {
  int tiles_local = (N + 15) / 16;
  long long total = (long long)n_slabs * tiles_local * aps * 64;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < total;
       c += (long long)gridDim.x * blockDim.x) {
    int lane_pos = (int)(c % 64);
    long long atom_idx = c / 64;
    int a = (int)(atom_idx % aps);
    int tl = (int)((atom_idx / aps) % tiles_local);
    int s = (int)(atom_idx / aps / tiles_local);
    int half = lane_pos >> 5, lane = lane_pos & 31, g = lane >> 2, t = lane & 3;
    int row = tl * 16 + half * 8 + g;
    int k = (s * aps + a) * 32 + t * 8;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (row < N) v = *reinterpret_cast<const uint4 *>(src + (size_t)row * K + k);
    dst[(((long long)s * n_tiles_total + tile0 + tl) * aps + a) * 64 + half * 32 + lane] = v;
  }
}

template <typename T>
__global__ void to_float_kernel(const T *__restrict__ src, float *__restrict__ dst, int n) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = (float)src[i];
}

// ------------------------------------------------------------------------------------
// a1: embedding gather.  x[m][:] = E[token of row m]; row m = b*R + r sits at position
// *pos0 + r of sequence b.
// ------------------------------------------------------------------------------------
// The blocks past the rows write the rotary table of the same positions (rope_table_kernel's).
struct RopeTable {
  const double *inv_freq;
  float2 *table;
  int half;
};
// cos/sin of pos * theta^(-2i/d), computed in double so that long contexts do not lose angle precision; entry idx of
// the table [R][d/2] of (cos, sin).
__device__ __forceinline__ void rope_entry(const RopeTable &T, int pos0, int R, int idx) {
  if (idx >= R * T.half) return;
  double s, c;
  sincos((double)(pos0 + idx / T.half) * T.inv_freq[idx % T.half], &s, &c);
  T.table[idx] = make_float2((float)c, (float)s);
}
// grid (rows + blocks of the table), 128 threads
__global__ void embed_kernel(PackedMat E, const int *__restrict__ tokens, int max_seq,
                             const int *__restrict__ pos0, int R, int n_rows, float *x, int ldx,
                             int accumulate, DevState *st, RopeTable rope) {
  if (blockIdx.x >= n_rows) return rope_entry(rope, *pos0, R, (blockIdx.x - n_rows) * blockDim.x + threadIdx.x);
  int m = blockIdx.x, b = m / R, r = m % R;
  int tok = tokens[(size_t)b * max_seq + *pos0 + r];
  if (tok < 0 || tok >= E.N) {
    if (threadIdx.x == 0) atomicMax(&st->error, 1);
    tok = min(max(tok, 0), E.N - 1);
  }
  float *xr = x + (size_t)m * ldx;
  if (E.wf) {
    const float *e = E.wf + (size_t)tok * E.K;
    for (int k = threadIdx.x; k < E.K; k += blockDim.x) xr[k] = accumulate ? xr[k] + e[k] : e[k];
    return;
  }
  int T = tok >> 4, half = (tok >> 3) & 1, g = tok & 7;
  for (int c = threadIdx.x; c < E.K / 8; c += blockDim.x) {   // one 16-byte chunk = 8 values
    int k = c * 8, atom = k >> 5, t = (k >> 3) & 3;
    int s = atom / E.aps, a = atom % E.aps;
    uint4 v = E.w[(((long long)s * E.n_tiles + T) * E.aps + a) * 64 + half * 32 + g * 4 + t];
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float lo = bf16_bits_to_float(w[j] & 0xffffu), hi = bf16_bits_to_float(w[j] >> 16);
      if (accumulate) { lo += xr[k + 2 * j]; hi += xr[k + 2 * j + 1]; }
      xr[k + 2 * j] = lo;
      xr[k + 2 * j + 1] = hi;
    }
  }
}

// ------------------------------------------------------------------------------------
// Activation preparation for a projection: act[m][:] = x[m][:] / rms(x[m]) * w, and clear
// the accumulator row the projection will add into.  Grid (rows, slices): every block clears
// PREP_ZERO_COLS columns of its row's accumulator, the first block of a row also does the norm.
// ------------------------------------------------------------------------------------
constexpr int PREP_ZERO_COLS = 4096;
__global__ void prep_norm_kernel(const float *x, int ldx, const float *__restrict__ w,
                                 int K, float eps, float *act, int lda,
                                 float *zero_buf, int zero_ld, int zero_cols) {
  pdl_enter();
  const int m = blockIdx.x;
  if (zero_buf) {
    const int c0 = blockIdx.y * PREP_ZERO_COLS, c1 = min(zero_cols, c0 + PREP_ZERO_COLS);
    float *row = zero_buf + (size_t)m * zero_ld;
    const bool aligned = (reinterpret_cast<uintptr_t>(row) & 15) == 0;
    for (int k = c0 + threadIdx.x * 4; k < c1; k += blockDim.x * 4) {
      if (aligned && k + 4 <= c1) *reinterpret_cast<float4 *>(row + k) = make_float4(0.f, 0.f, 0.f, 0.f);
      else for (int j = k; j < c1; ++j) row[j] = 0.f;
    }
  }
  if (blockIdx.y != 0) return;
  const float *xr = x + (size_t)m * ldx;
  float ss = 0.f;
  for (int k = threadIdx.x; k < K; k += blockDim.x) ss += xr[k] * xr[k];
  __shared__ float red[32];
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  float inv = rsqrtf(red[0] / (float)K + eps);
  for (int k = threadIdx.x; k < K; k += blockDim.x) act[(size_t)m * lda + k] = xr[k] * inv * w[k];
}

// act[m][i] = silu(g) * u with g = gu[m][i], u = gu[m][I + i]  (the SwiGLU gate).
__global__ void prep_swiglu_kernel(const float *gu, int ldgu, int I,
                                   float *act, int lda) {
  pdl_enter();
  int m = blockIdx.y;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= I) return;
  float g = gu[(size_t)m * ldgu + i], u = gu[(size_t)m * ldgu + I + i];
  act[(size_t)m * lda + i] = g / (1.f + expf(-g)) * u;
}

// ------------------------------------------------------------------------------------
// Projection, bf16 weights: out[m][n] += sum_k W[n][k] * act[m][k].
//
// The atom stream is cut into equal contiguous ranges, one per warp of the grid, so every
// warp streams the same number of bytes whatever N and K are.  A warp walks its range
// segment by segment (a segment = atoms of one row tile inside one k-slab), accumulates with
// mma.m16n8k16 (weights = A operand straight from global memory in register order,
// activations = B operand from shared memory as bf16 hi/lo column pairs), and adds each
// finished segment into `out` with fp32 reductions.  NT n8-tiles cover 4*NT activation rows
// per sweep; more rows are swept in turn.
// ------------------------------------------------------------------------------------
template <int NT>
__global__ void __launch_bounds__(GEMV_THREADS)
gemv_bf16_kernel(PackedMat W, const float *act, int lda, int M,
                 float *out, int ldo) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int KS = W.aps * 32;
  const int row_bytes = ((KS * 2) % 128 == 64) ? KS * 2 : KS * 2 + 64;   // conflict-free LDS.128
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;

  const long long A = packed_atoms(W);
  const long long c0 = A * blockIdx.x / gridDim.x, c1 = A * (blockIdx.x + 1) / gridDim.x;
  const long long w0 = c0 + (c1 - c0) * warp / GEMV_WARPS, w1 = c0 + (c1 - c0) * (warp + 1) / GEMV_WARPS;
  if (c0 >= c1) return;
  const long long slab_atoms = (long long)W.n_tiles * W.aps;
  const int s_first = (int)(c0 / slab_atoms), s_last = (int)((c1 - 1) / slab_atoms);

  for (int m0 = 0; m0 < M; m0 += 4 * NT) {
    for (int s = s_first; s <= s_last; ++s) {
      __syncthreads();
      // stage rows m0 .. m0+4NT-1, k in slab s, as columns (2r: hi, 2r+1: lo)
      for (int idx = threadIdx.x; idx < 4 * NT * (KS / 4); idx += GEMV_THREADS) {
        int r = idx / (KS / 4), k4 = (idx % (KS / 4)) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m0 + r < M) v = *reinterpret_cast<const float4 *>(act + (size_t)(m0 + r) * lda + s * KS + k4);
        __nv_bfloat16 h[4], l[4];
        split_bf16(v.x, h[0], l[0]); split_bf16(v.y, h[1], l[1]);
        split_bf16(v.z, h[2], l[2]); split_bf16(v.w, h[3], l[3]);
        *reinterpret_cast<uint2 *>(smem_raw + (size_t)(2 * r) * row_bytes + k4 * 2) =
            *reinterpret_cast<uint2 *>(h);
        *reinterpret_cast<uint2 *>(smem_raw + (size_t)(2 * r + 1) * row_bytes + k4 * 2) =
            *reinterpret_cast<uint2 *>(l);
      }
      __syncthreads();
      long long a_lo = max(w0, (long long)s * slab_atoms), a_hi = min(w1, (long long)(s + 1) * slab_atoms);
      while (a_lo < a_hi) {
        long long in_slab = a_lo - (long long)s * slab_atoms;
        int T = (int)(in_slab / W.aps), a_begin = (int)(in_slab % W.aps);
        int a_end = (int)min((long long)W.aps, a_begin + (a_hi - a_lo));
        float acc[NT][4];
#pragma unroll
        for (int i = 0; i < NT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
        const uint4 *wp = W.w + (a_lo - a_begin) * 64 + lane;
        const unsigned char *bp = smem_raw + (size_t)g * row_bytes + t * 16;
        int a = a_begin;
        for (; a + 4 <= a_end; a += 4) {
          uint4 A0[4], A1[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            A0[u] = ldg_stream(wp + (size_t)(a + u) * 64);
            A1[u] = ldg_stream(wp + (size_t)(a + u) * 64 + 32);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int i = 0; i < NT; ++i) {
              uint4 Bv = *reinterpret_cast<const uint4 *>(bp + (size_t)(8 * i) * row_bytes + (a + u) * 64);
              mma_bf16_16816(acc[i], A0[u].x, A1[u].x, A0[u].y, A1[u].y, Bv.x, Bv.y);
              mma_bf16_16816(acc[i], A0[u].z, A1[u].z, A0[u].w, A1[u].w, Bv.z, Bv.w);
            }
          }
        }
        for (; a < a_end; ++a) {
          uint4 A0 = ldg_stream(wp + (size_t)a * 64), A1 = ldg_stream(wp + (size_t)a * 64 + 32);
#pragma unroll
          for (int i = 0; i < NT; ++i) {
            uint4 Bv = *reinterpret_cast<const uint4 *>(bp + (size_t)(8 * i) * row_bytes + a * 64);
            mma_bf16_16816(acc[i], A0.x, A1.x, A0.y, A1.y, Bv.x, Bv.y);
            mma_bf16_16816(acc[i], A0.z, A1.z, A0.w, A1.w, Bv.z, Bv.w);
          }
        }
        // accumulator columns 2t (hi) and 2t+1 (lo) belong to activation row 4i+t
        int n_lo = T * 16 + g;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          int m = m0 + 4 * i + t;
          if (m < M) {
            if (n_lo < W.N) atomicAdd(out + (size_t)m * ldo + n_lo, acc[i][0] + acc[i][1]);
            if (n_lo + 8 < W.N) atomicAdd(out + (size_t)m * ldo + n_lo + 8, acc[i][2] + acc[i][3]);
          }
        }
        a_lo += a_end - a_begin;
      }
    }
  }
}

// Projection, fp32 weights (small verification models only), more rows than a decode pass of a few sequences has:
// out[m][n] += sum_k W[n][k] act[m][k] by tiles of BM activation rows x BN weight rows.  A thread holds 4 x 4 outputs; KG sets
// of threads share a tile, each a part of every piece of k, and add their sums at the end.  Both operands come as they lie
// (k fastest) by asynchronous copies, two pieces of 32 KG values in flight; four floats of padding to a row keep the 16-byte reads
// free of bank conflicts.  Bound by fp32 arithmetic at prefill sizes (two products per instruction, fma.f32x2), by the trips
// to memory of its few blocks at decode sizes, hence the small tiles with four thread sets.
// Measured, a layer with its other kernels, against one warp to a weight row, which read every activation row from L1 for each
// of them: hidden 256, 32 / 512 / 1000 rows 97 / 1090 / 2054 us -> 48 / 86 / 137; hidden 1024, 12 / 1000 rows 122 / 6892 -> 83 / 915.
// Sums over 128 values of k at a time, then of those sums: no further from fp64 than the lane-wise sums before.
constexpr int GF_PAD = 4;
template <int BM, int BN, int KG>
constexpr int gemm_f32_smem() { return 2 * (BM + BN) * (32 * KG + GF_PAD) * 4; }
template <int BM, int BN, int KG>
__global__ void __launch_bounds__(BM * BN / 16 * KG) gemm_f32_kernel(PackedMat W, const float *act, int lda, int M, float *out, int ldo) {
  constexpr int SET = BM * BN / 16, THREADS = SET * KG, BK = 32 * KG, LD = BK + GF_PAD, STAGE = (BM + BN) * LD;
  extern __shared__ __align__(16) float gf_smem[];
  const int tid = threadIdx.x, kg = tid / SET, tx = tid % SET % (BN / 4), ty = tid % SET / (BN / 4);
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * BM, K = W.K;
  const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(gf_smem);
  // rows [first, first + ROWS) of the stage: values k0 .. k0 + BK - 1 of the rows of `src` from row0 on; zeros past the end
  auto fetch_rows = [&](const float *src, size_t ld, int row0, int n_rows, int first, int rows, int k0, int stage) {
    for (int i = tid; i < rows * (BK / 4); i += THREADS) {
      const int r = i / (BK / 4), k = k0 + i % (BK / 4) * 4;
      const bool ok = row0 + r < n_rows && k < K;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem0 + (stage * STAGE + (first + r) * LD + i % (BK / 4) * 4) * 4),
                   "l"(src + (ok ? (size_t)(row0 + r) * ld + k : 0)), "r"(ok ? 16 : 0)
                   : "memory");
    }
  };
  auto fetch_w = [&](int k0, int stage) { fetch_rows(W.wf, K, n0, W.N, BM, BN, k0, stage); };
  auto fetch_act = [&](int k0, int stage) { fetch_rows(act, lda, m0, M, 0, BM, k0, stage); };
  fetch_w(0, 0);                            // weights: before the kernel in front is complete
  pdl_enter();
  fetch_act(0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  float sum[4][4];
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { sum[i][j] = 0.f; acc[i][j] = make_float2(0.f, 0.f); }
  const int n_pieces = (K + BK - 1) / BK;
#pragma unroll 1
  for (int p = 0; p < n_pieces; ++p) {
    if (p + 1 < n_pieces) { fetch_w((p + 1) * BK, (p + 1) & 1); fetch_act((p + 1) * BK, (p + 1) & 1); }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const float *a_s = gf_smem + (p & 1) * STAGE + kg * 32, *b_s = a_s + BM * LD;
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4 *>(a_s + (ty + i * (BM / 4)) * LD + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4 *>(b_s + (tx + j * (BN / 4)) * LD + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          fma_f32x2(acc[i][j], make_float2(a[i].x, a[i].y), make_float2(b[j].x, b[j].y));
          fma_f32x2(acc[i][j], make_float2(a[i].z, a[i].w), make_float2(b[j].z, b[j].w));
        }
    }
    if ((p & 3) == 3 || p + 1 == n_pieces) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { sum[i][j] += acc[i][j].x + acc[i][j].y; acc[i][j] = make_float2(0.f, 0.f); }
    }
    __syncthreads();                        // the stage is free
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (KG > 1) {
    // the other sets' sums, through the stages' memory
    if (kg > 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) gf_smem[((kg - 1) * 16 + i * 4 + j) * SET + tid % SET] = sum[i][j];
    }
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int g = 0; g < KG - 1; ++g)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sum[i][j] += gf_smem[(g * 16 + i * 4 + j) * SET + tid];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty + i * (BM / 4);
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx + j * (BN / 4);
      if (n < W.N) out[(size_t)m * ldo + n] += sum[i][j];
    }
  }
}

// The same for the few rows of a decode pass, together with the step in front of it: every block works the M activation
// rows out in shared memory (a few KB) - RMSNorm, the SwiGLU gate, or the merge of the attention's key slices - and
// multiplies its weight rows.  A layer of a small model is bound by the number of its launches and by the trips to memory
// that follow one another in each: five launches instead of ten, and in each of them one trip for everything that is read
// (the first weight row of a warp is requested before the kernel in front is waited for).  24 passes of the 4-layer fp32
// test shape (hidden 256), one sequence: 2.00 ms with ten launches a layer, 1.34 so; 16 sequences: 5.72 and 4.92.
// store: out = instead of out +=.
enum { F32_NORM = 0, F32_SWIGLU = 1, F32_SLICES = 2 };
constexpr int F32_FUSE_ROWS = 16, F32_FUSE_FLOATS = 12 * 1024;     // most rows, and rows x K (48 KB)
constexpr int F32_AHEAD = 6;                                        // 128-value pieces of a row in flight
struct F32In {
  const float *act;               // F32_NORM: [M][lda]; F32_SWIGLU: gate | up, K apart
  int lda;
  const float *norm_w;
  float eps;
  const float *part_o, *part_ml;  // F32_SLICES: [(row * nq + head) * nsplit + slice][K / nq] and (max, sum)
  int nsplit, nq;
};
template <int IN>
__global__ void __launch_bounds__(256) gemv_f32_fused_kernel(PackedMat W, F32In in, int M, float *out, int ldo, int store) {
  extern __shared__ __align__(16) float xs[];                       // [M][K]
  __shared__ float ss_part[8][F32_FUSE_ROWS];                       // F32_NORM: sums of squares, by a row's warps
  const int lane = threadIdx.x & 31, w8 = threadIdx.x >> 5, K = W.K;
  const int warp = blockIdx.x * 8 + w8, n_warps = gridDim.x * 8;
  const int row_warps = M >= 8 ? 1 : 8 / M, part = w8 % row_warps;  // warps that share an activation row
  float4 w0[F32_AHEAD];
#pragma unroll
  for (int c = 0; c < F32_AHEAD; ++c) {
    const int k = lane * 4 + 128 * c;
    w0[c] = warp < W.N && k < K ? *reinterpret_cast<const float4 *>(W.wf + (size_t)warp * K + k) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_enter();
  // lane i < 4: the value that row i's product is added to
  const float old = !store && warp < W.N && lane < min(4, M) ? out[(size_t)lane * ldo + warp] : 0.f;
  if (IN == F32_SLICES) {
    // one warp per (row, head), as attn_merge_kernel; the first slices' outputs are requested with the (max, sum) pairs
    constexpr int FIRST = 2;
    const int D = K / in.nq;
    for (int i = w8; i < M * in.nq; i += 8) {
      const float2 *ml = reinterpret_cast<const float2 *>(in.part_ml) + (size_t)i * in.nsplit;
      const float *po = in.part_o + (size_t)i * in.nsplit * D;
      float2 v = lane < in.nsplit ? ml[lane] : make_float2(0.f, 0.f);
      float first[FIRST][4];
#pragma unroll
      for (int s = 0; s < FIRST; ++s)
#pragma unroll
        for (int e = 0; e < 4; ++e) first[s][e] = s < in.nsplit && lane + 32 * e < D ? po[s * D + lane + 32 * e] : 0.f;
      float mx = v.y > 0.f ? v.x : -INFINITY;
      for (int s = lane + 32; s < in.nsplit; s += 32) {
        const float2 u = ml[s];
        if (u.y > 0.f) mx = fmaxf(mx, u.x);
      }
      mx = warp_max(mx);
      float l = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};                    // D is 64 or 128: two or four values per lane
      for (int s0 = 0; s0 < in.nsplit; s0 += 32) {
        if (s0) v = s0 + lane < in.nsplit ? ml[s0 + lane] : make_float2(0.f, 0.f);
        const float f = v.y > 0.f ? __expf(v.x - mx) : 0.f;
        l += f * v.y;
        unsigned live = __ballot_sync(0xffffffffu, v.y > 0.f);       // slices without keys hold nothing that may be used
        if (s0 == 0) {
#pragma unroll
          for (int s = 0; s < FIRST; ++s)
            if (live >> s & 1) {
              const float fs = __shfl_sync(0xffffffffu, f, s);
#pragma unroll
              for (int e = 0; e < 4; ++e) o[e] += fs * first[s][e];
            }
          live &= ~0u << FIRST;
        }
        while (live) {
          const int s = __ffs(live) - 1;
          live &= live - 1;
          const float fs = __shfl_sync(0xffffffffu, f, s);
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (lane + 32 * e < D) o[e] += fs * po[(size_t)(s0 + s) * D + lane + 32 * e];
        }
      }
      const float inv = 1.f / warp_sum(l);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (lane + 32 * e < D) xs[(size_t)i * D + lane + 32 * e] = o[e] * inv;
    }
  } else {
    // RMSNorm: the rows times the gain, 1 / rms goes to the product; a row's warps take its 128-value pieces in turn
    for (int m = w8 / row_warps; m < M; m += 8) {
      const float *xr = in.act + (size_t)m * in.lda;
      float ss = 0.f;
#pragma unroll 4
      for (int k = (part * 32 + lane) * 4; k < K; k += 128 * row_warps) {
        float4 v = *reinterpret_cast<const float4 *>(xr + k);
        const float4 u = *reinterpret_cast<const float4 *>((IN == F32_SWIGLU ? xr + K : in.norm_w) + k);
        if (IN == F32_SWIGLU) {
          v.x = v.x / (1.f + expf(-v.x)); v.y = v.y / (1.f + expf(-v.y));
          v.z = v.z / (1.f + expf(-v.z)); v.w = v.w / (1.f + expf(-v.w));
        } else {
          ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
        *reinterpret_cast<float4 *>(xs + (size_t)m * K + k) = make_float4(v.x * u.x, v.y * u.y, v.z * u.z, v.w * u.w);
      }
      if (IN == F32_NORM) {
        ss = warp_sum(ss);
        if (lane == 0) ss_part[part][m] = ss;
      }
    }
  }
  __syncthreads();
  float row_scale = 1.f;                                            // lane m: of row m
  if (IN == F32_NORM && lane < M) {
    float ss = 0.f;
    for (int i = 0; i < row_warps; ++i) ss += ss_part[i][lane];
    row_scale = rsqrtf(ss / (float)K + in.eps);
  }
  for (int n = warp; n < W.N; n += n_warps) {
    const float *wr = W.wf + (size_t)n * K;
    for (int m0 = 0; m0 < M; m0 += 4) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      auto add = [&](const float4 &w, int k) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (m0 + i < M) {
            const float4 a = *reinterpret_cast<const float4 *>(xs + (size_t)(m0 + i) * K + k);
            acc[i] += w.x * a.x + w.y * a.y + w.z * a.z + w.w * a.w;
          }
      };
      int k = lane * 4;
      if (n == warp) {
#pragma unroll
        for (int c = 0; c < F32_AHEAD; ++c, k += 128)
          if (k < K) add(w0[c], k);
      }
      for (; k < K; k += 128) add(*reinterpret_cast<const float4 *>(wr + k), k);
      float v = 0.f;                                                // lane i < 4: row m0 + i
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float t = warp_sum(acc[i]);
        if (lane == i) v = t;
      }
      const float scale = __shfl_sync(0xffffffffu, row_scale, (m0 + lane) & 31);
      if (lane < 4 && m0 + lane < M) {
        float *o = out + (size_t)(m0 + lane) * ldo + n;
        *o = v * scale + (store ? 0.f : n == warp && m0 == 0 ? old : *o);
      }
    }
  }
}

// ------------------------------------------------------------------------------------
// a3: per-head QK-norm, rotary embedding, KV append.
// ------------------------------------------------------------------------------------

// The table for the R positions of a call that embeds nothing.
__global__ void rope_table_kernel(const int *__restrict__ pos0, int R, RopeTable T) {
  rope_entry(T, *pos0, R, blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename KVT> __device__ __forceinline__ KVT to_kv(float v);
template <> __device__ __forceinline__ float to_kv<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 to_kv<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}
template <> __device__ __forceinline__ __half to_kv<__half>(float v) { return __float2half_rn(v); }

// One warp per (row, head); heads are q heads, then k heads, then v heads.  q is normalised
// and rotated in place (fp32); k is normalised, rotated and stored in the cache; v is stored.
// qkv [M][ldq] = (q | k | v) per row.  Cache layout [b][kv head][max_seq][D].
template <int D, typename KVT>
__global__ void qk_norm_rope_append_kernel(float *qkv, int ldq, int nq, int nkv, int R,
                                           const float *__restrict__ w_qn, const float *__restrict__ w_kn,
                                           float eps, const float2 *__restrict__ table,
                                           const int *__restrict__ pos0, KVT *kc,
                                           KVT *vc, int max_seq) {
  pdl_enter();
  constexpr int E = D / 32;                 // values per lane; value j pairs with j + E/2
  int lane = threadIdx.x & 31;
  int head = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (head >= nq + 2 * nkv) return;
  int m = blockIdx.x, b = m / R, r = m % R, pos = *pos0 + r;
  float *src = qkv + (size_t)m * ldq + (size_t)head * D;
  float v[E];
#pragma unroll
  for (int j = 0; j < E; ++j) v[j] = src[lane + 32 * j];
  if (head >= nq + nkv) {                   // v head: plain append
    int h = head - nq - nkv;
    KVT *dst = vc + (((size_t)b * nkv + h) * max_seq + pos) * D;
#pragma unroll
    for (int j = 0; j < E; ++j) dst[lane + 32 * j] = to_kv<KVT>(v[j]);
    return;
  }
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < E; ++j) ss += v[j] * v[j];
  ss = warp_sum(ss);
  float inv = rsqrtf(ss / (float)D + eps);
  const float *w = head < nq ? w_qn : w_kn;
#pragma unroll
  for (int j = 0; j < E; ++j) v[j] = v[j] * inv * w[lane + 32 * j];
  float o[E];
#pragma unroll
  for (int j = 0; j < E / 2; ++j) {
    float2 cs = table[(size_t)r * (D / 2) + lane + 32 * j];
    float a = v[j], bb = v[j + E / 2];
    o[j] = a * cs.x - bb * cs.y;
    o[j + E / 2] = bb * cs.x + a * cs.y;
  }
  if (head < nq) {
#pragma unroll
    for (int j = 0; j < E; ++j) src[lane + 32 * j] = o[j];
  } else {
    int h = head - nq;
    KVT *dst = kc + (((size_t)b * nkv + h) * max_seq + pos) * D;
#pragma unroll
    for (int j = 0; j < E; ++j) dst[lane + 32 * j] = to_kv<KVT>(o[j]);
  }
}

// Step a3 inside an attention kernel: it reads the raw q | k | v rows of the QKV projection itself; every block
// normalises and rotates its own query rows and the new K rows that fall into its keys (a few rows, recomputed by the
// blocks that share them), and the block that owns a position appends its K and V rows to the cache.
struct AttnFuse {
  const float *w_qn, *w_kn;        // QK-norm weights [D]
  const float2 *table;             // (cos, sin) of the pass's positions [R][D / 2]
  float eps;
};
// QK-norm and rotary embedding of one head vector, v[j] = element lane + 32 j.
template <int D>
__device__ __forceinline__ void head_norm_rope(const float *w, const float2 *cs_row, float eps, int lane, float (&v)[D / 32]) {
  constexpr int E = D / 32;
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < E; ++j) ss += v[j] * v[j];
  const float inv = rsqrtf(warp_sum(ss) / (float)D + eps);
#pragma unroll
  for (int j = 0; j < E; ++j) v[j] = v[j] * inv * w[lane + 32 * j];
#pragma unroll
  for (int j = 0; j < E / 2; ++j) {
    const float2 cs = cs_row[lane + 32 * j];
    const float a = v[j], b = v[j + E / 2];
    v[j] = a * cs.x - b * cs.y;
    v[j + E / 2] = b * cs.x + a * cs.y;
  }
}

// ------------------------------------------------------------------------------------
// a4: split-KV attention.  Each block handles one (sequence, kv head, block of RB new
// positions, slice of CH keys): the G query heads of that kv head for those positions form
// up to 16 query rows that share every key/value it reads.  Blocks write unnormalised
// partial outputs with their running max and sum; attn_merge_kernel combines the slices.
// ------------------------------------------------------------------------------------
__host__ __device__ constexpr int attn_warps(int T) { return T == 1 ? 8 : 4; }       // warps of an attn_partial_kernel block
constexpr int ATTN_QR = 16;       // query rows per block

template <typename KVT> __device__ __forceinline__ void load8(const KVT *p, float (&f)[8]);
template <> __device__ __forceinline__ void load8<float>(const float *p, float (&f)[8]) {
  float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
template <> __device__ __forceinline__ void load8<__nv_bfloat16>(const __nv_bfloat16 *p, float (&f)[8]) {
  uint4 v = *reinterpret_cast<const uint4 *>(p);
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    f[2 * j] = bf16_bits_to_float(w[j] & 0xffffu);
    f[2 * j + 1] = bf16_bits_to_float(w[j] >> 16);
  }
}

template <> __device__ __forceinline__ void load8<__half>(const __half *p, float (&f)[8]) {
  uint4 v = *reinterpret_cast<const uint4 *>(p);
  const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 x = __half22float2(h[j]);
    f[2 * j] = x.x;
    f[2 * j + 1] = x.y;
  }
}
// NQ: query rows the block is compiled for, 4, 8 or 16 (the scores, the probabilities and the outputs of all NQ rows are
// worked out).  A warp takes 8 T keys at a time:
//   T = 1, 8 warps, four lanes to a key: slices of 64 keys of launches that are resident at once.  Bound by the trips to memory that follow one another, so K and V come in one, and
//   the older keys (previous passes appended them) are requested before the kernel in front is waited for.
//   T = 4, 4 warps, a lane to a key: longer slices, and more blocks than that.  Bound by instructions, so one softmax step
//     serves 32 keys, and by the blocks an SM holds: four with 64 dimensions, three with 128.
// Isolated, 36 keys of one head and 2 query rows took 27 us with 16 rows and one load at a time, 11 us with T = 4 in 8-key
// loads.  32 x 8192 keys, 8 kv heads of bf16 rows: 234 us with T = 4, 460 with T = 1.
template <int D, typename KVT, int NQ, bool FUSED, int T>
__global__ void __launch_bounds__(attn_warps(T) * 32, T == 1 ? 1 : D == 64 ? 4 : 3)
attn_partial_kernel(const float *qkv, int ldq, const KVT *kc,
                    const KVT *vc, int max_seq, int nq, int nkv, int R, int RB, int CH,
                    const int *__restrict__ pos0_ptr, int pos0_val, float *part_o,
                    float *part_ml, int nsplit, AttnFuse F) {
  constexpr int E = D / 32, NC = D / 32, W = attn_warps(T), TK = 8 * T;   // V: dims lane * E ..; K: NC chunks of 8 dims per lane
  const int G = nq / nkv;
  const int split = blockIdx.x, n_rb = (R + RB - 1) / RB;
  const int kvh = blockIdx.y / n_rb, rb = blockIdx.y % n_rb, b = blockIdx.z;
  const int r0 = rb * RB, r1 = min(R, r0 + RB), nQ = (r1 - r0) * G;
  // the position, and keys before it, are older than the last plainly launched kernel (the rotary table's)
  const int pos0 = pos0_ptr ? *pos0_ptr : pos0_val;
  const int j0 = split * CH, j1 = min(j0 + CH, pos0 + r1);      // keys [j0, j1); last row sees pos0+r1-1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  __shared__ float q_s[NQ][D];
  __shared__ __align__(16) float p_s[W][NQ][TK];
  __shared__ float red_m[W][NQ], red_l[W][NQ];
  extern __shared__ __align__(16) float o_s[];                   // [W][NQ][D]

  if (j0 >= j1) {                                                 // empty slice: mark and leave
    pdl_enter();
    for (int qi = threadIdx.x; qi < nQ; qi += blockDim.x) {
      int r = r0 + qi / G, h = kvh * G + qi % G;
      size_t slot = ((size_t)(b * R + r) * nq + h) * nsplit + split;
      part_ml[slot * 2] = -INFINITY;
      part_ml[slot * 2 + 1] = 0.f;
    }
    return;
  }
  const float scale = rsqrtf((float)D);
  const size_t head_off = ((size_t)b * nkv + kvh) * max_seq * D;
  const KVT *kbase = kc + head_off, *vbase = vc + head_off;
  KVT *const new_k = reinterpret_cast<KVT *>(o_s + W * NQ * D), *const new_v = new_k + (size_t)R * D;
  auto k_row = [&](int j) { return FUSED && j >= pos0 ? new_k + (size_t)(j - pos0) * D : kbase + (size_t)j * D; };
  auto v_row = [&](int j) { return FUSED && j >= pos0 ? new_v + (size_t)(j - pos0) * D : vbase + (size_t)j * D; };
  float kf[NC][8], vf[8][E];
  // T = 1: of the keys [jb, jb + 8) those in [lo, hi)
  auto load_tile = [&](int jb, int lo, int hi) {
    const int jk = jb + (lane >> 2);
    if (jk >= lo && jk < hi) {
      const KVT *k = k_row(jk);
#pragma unroll
      for (int c = 0; c < NC; ++c) load8<KVT>(k + (c * 4 + (lane & 3)) * 8, kf[c]);
    }
#pragma unroll
    for (int jj = 0; jj < 8; ++jj)
      if (jb + jj >= lo && jb + jj < hi) {
        const KVT *v = v_row(jb + jj);
#pragma unroll
        for (int e = 0; e < E; ++e) vf[jj][e] = (float)v[lane * E + e];
      }
  };
  if (T == 1) {
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int e = 0; e < 8; ++e) kf[c][e] = 0.f;
#pragma unroll
    for (int jj = 0; jj < 8; ++jj)
#pragma unroll
      for (int e = 0; e < E; ++e) vf[jj][e] = 0.f;
    load_tile(j0 + warp * TK, j0, min(j1, pos0));
  }
  pdl_enter();

  if (FUSED) {
    // step a3 (see AttnFuse): the pass's rows r_lo .. r_hi - 1 sit at positions inside this slice
    const int r_lo = max(0, j0 - pos0), r_hi = min(r1, j1 - pos0);
    const int n_kv = 2 * max(0, r_hi - r_lo);
    for (int task = warp; task < n_kv + NQ; task += W) {
      const bool is_q = task >= n_kv;
      const int qi = task - n_kv, r = is_q ? r0 + qi / G : r_lo + (task >> 1), is_v = !is_q && (task & 1);
      float v[E];
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = 0.f;
      if (!is_q || qi < nQ) {
        const int head = is_q ? kvh * G + qi % G : nq + (is_v ? nkv : 0) + kvh;
        const float *src = qkv + (size_t)(b * R + r) * ldq + (size_t)head * D;
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = src[lane + 32 * e];
        if (!is_v) head_norm_rope<D>(is_q ? F.w_qn : F.w_kn, F.table + (size_t)r * (D / 2), F.eps, lane, v);
      }
      if (is_q) {
#pragma unroll
        for (int e = 0; e < E; ++e) q_s[qi][lane + 32 * e] = v[e] * scale;
      } else {
        KVT *cache = const_cast<KVT *>(is_v ? vbase : kbase) + (size_t)(pos0 + r) * D;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const KVT h = to_kv<KVT>(v[e]);
          (is_v ? new_v : new_k)[(size_t)r * D + lane + 32 * e] = h;
          if (r >= r0) cache[lane + 32 * e] = h;         // the row block that owns the position appends it
        }
      }
    }
  } else {
    for (int idx = threadIdx.x; idx < NQ * D; idx += blockDim.x) {
      int qi = idx / D, dd = idx % D;
      float v = 0.f;
      if (qi < nQ) {
        int r = r0 + qi / G, h = kvh * G + qi % G;
        v = qkv[(size_t)(b * R + r) * ldq + (size_t)h * D + dd] * scale;
      }
      q_s[qi][dd] = v;
    }
  }
  __syncthreads();

  float m_run[NQ], l_run[NQ], o_acc[NQ][E];                       // l_run: of this lane's own keys
#pragma unroll
  for (int qi = 0; qi < NQ; ++qi) {
    m_run[qi] = -INFINITY; l_run[qi] = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) o_acc[qi][e] = 0.f;
  }

  for (int jb = j0 + warp * TK; jb < j1; jb += W * TK) {
    float s[NQ];
    auto dot8 = [](const float (&k)[8], const float *q) {
      const float4 a = *reinterpret_cast<const float4 *>(q), b = *reinterpret_cast<const float4 *>(q + 4);
      return k[0] * a.x + k[1] * a.y + k[2] * a.z + k[3] * a.w + k[4] * b.x + k[5] * b.y + k[6] * b.z + k[7] * b.w;
    };
    if constexpr (T == 1) {
      if (jb != j0 + warp * TK) load_tile(jb, j0, min(j1, pos0));
      if (jb + TK > pos0) load_tile(jb, pos0, j1);                // keys of this pass
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) {
        s[qi] = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) s[qi] += dot8(kf[c], &q_s[qi][(c * 4 + (lane & 3)) * 8]);
        s[qi] += __shfl_xor_sync(0xffffffffu, s[qi], 1);
        s[qi] += __shfl_xor_sync(0xffffffffu, s[qi], 2);
      }
    } else {
      const KVT *k = k_row(min(jb + lane, j1 - 1));
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) s[qi] = 0.f;
#pragma unroll 4
      for (int c = 0; c < D / 8; ++c) {
        float kr[8];
        load8<KVT>(k + c * 8, kr);
#pragma unroll
        for (int qi = 0; qi < NQ; ++qi) s[qi] += dot8(kr, &q_s[qi][c * 8]);
      }
    }
    const int jt = T == 1 ? lane >> 2 : lane, j = jb + jt;
#pragma unroll
    for (int qi = 0; qi < NQ; ++qi) {
      if (qi < nQ) {                                  // uniform across the warp
        const int pos = pos0 + r0 + qi / G;
        const bool ok = j < j1 && j <= pos;
        float mx = ok ? s[qi] : -INFINITY;
#pragma unroll
        for (int x = T == 1 ? 4 : 1; x < 32; x <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
        const float m_new = fmaxf(m_run[qi], mx);
        float p = 0.f, corr = 1.f;
        if (m_new > -INFINITY) {
          corr = __expf(m_run[qi] - m_new);           // exp(-inf) = 0 on the first block
          p = ok ? __expf(s[qi] - m_new) : 0.f;
        }
        l_run[qi] = l_run[qi] * corr + p;
        m_run[qi] = m_new;
#pragma unroll
        for (int e = 0; e < E; ++e) o_acc[qi][e] *= corr;
        if (T > 1 || (lane & 3) == 0) p_s[warp][qi][jt] = p;
      }
    }
    __syncwarp();
    const int n_here = min(TK, j1 - jb);
#pragma unroll 1
    for (int j8 = 0; j8 < n_here; j8 += 8) {
      if (T > 1) {
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {                          // past the last key: its row again, with probability 0
          const KVT *vr = v_row(jb + min(j8 + jj, n_here - 1)) + lane * E;
#pragma unroll
          for (int e = 0; e < E; ++e) vf[jj][e] = (float)vr[e];
        }
      }
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) {
        if (qi < nQ) {
          float p[8];
          *reinterpret_cast<float4 *>(p) = *reinterpret_cast<const float4 *>(&p_s[warp][qi][j8]);
          *reinterpret_cast<float4 *>(p + 4) = *reinterpret_cast<const float4 *>(&p_s[warp][qi][j8 + 4]);
#pragma unroll
          for (int jj = 0; jj < 8; ++jj)
#pragma unroll
            for (int e = 0; e < E; ++e) o_acc[qi][e] += p[jj] * vf[jj][e];
        }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int qi = 0; qi < NQ; ++qi)
#pragma unroll
    for (int x = T == 1 ? 4 : 1; x < 32; x <<= 1) l_run[qi] += __shfl_xor_sync(0xffffffffu, l_run[qi], x);

  // combine the warps of the block
#pragma unroll
  for (int qi = 0; qi < NQ; ++qi) {
    if (lane == 0) { red_m[warp][qi] = m_run[qi]; red_l[warp][qi] = l_run[qi]; }
#pragma unroll
    for (int e = 0; e < E; ++e) o_s[((size_t)warp * NQ + qi) * D + lane * E + e] = o_acc[qi][e];
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nQ * D; idx += blockDim.x) {
    int qi = idx / D, dd = idx % D;
    float m = -INFINITY;
#pragma unroll
    for (int w = 0; w < W; ++w) m = fmaxf(m, red_m[w][qi]);
    float l = 0.f, o = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      float f = red_m[w][qi] > -INFINITY ? __expf(red_m[w][qi] - m) : 0.f;
      l += red_l[w][qi] * f;
      o += o_s[((size_t)w * NQ + qi) * D + dd] * f;
    }
    int r = r0 + qi / G, h = kvh * G + qi % G;
    size_t slot = ((size_t)(b * R + r) * nq + h) * nsplit + split;
    part_o[slot * D + dd] = o;
    if (dd == 0) { part_ml[slot * 2] = m; part_ml[slot * 2 + 1] = l; }
  }
}

// One warp per (row, head): act[m][h*D + :] = sum_s w_s o_s / sum_s w_s l_s, w_s = exp(m_s - max m).
template <int D>
__global__ void attn_merge_kernel(const float *part_o, const float *part_ml,
                                  int nsplit, int n_rows_heads, int nq, float *act, int lda) {
  pdl_enter();
  constexpr int E = D / 32;
  int lane = threadIdx.x & 31;
  int idx = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (idx >= n_rows_heads) return;
  int m = idx / nq, h = idx % nq;
  const float *ml = part_ml + (size_t)idx * nsplit * 2;
  float mx = -INFINITY;
  for (int s = 0; s < nsplit; ++s)
    if (ml[2 * s + 1] > 0.f) mx = fmaxf(mx, ml[2 * s]);
  float l = 0.f, o[E];
#pragma unroll
  for (int e = 0; e < E; ++e) o[e] = 0.f;
  for (int s = 0; s < nsplit; ++s) {
    float ls = ml[2 * s + 1];
    if (ls > 0.f) {
      float f = __expf(ml[2 * s] - mx);
      l += ls * f;
      const float *po = part_o + ((size_t)idx * nsplit + s) * D + lane * E;
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] += po[e] * f;
    }
  }
  float inv = 1.f / l;
#pragma unroll
  for (int e = 0; e < E; ++e) act[(size_t)m * lda + (size_t)h * D + lane * E + e] = o[e] * inv;
}

// ------------------------------------------------------------------------------------
// a8: the lower->upper boundary of a full pass.  Only the newest row of each sequence goes
// on into the decoding layers (Section 2.2); the refill rows' outputs are dropped.
// ------------------------------------------------------------------------------------
__global__ void select_last_kernel(const float *x_lo, int R, int H, float *x_up) {
  pdl_enter();
  int b = blockIdx.x;
  const float *src = x_lo + ((size_t)b * R + (R - 1)) * H;
  for (int k = threadIdx.x; k < H; k += blockDim.x) x_up[(size_t)b * H + k] = src[k];
}

// ------------------------------------------------------------------------------------
// The ExDy variant (Section 2.1, the paragraph after Eq. 4): the short passes also run the first
// L_e encoding layers, and the output of those layers, h_enc, stands where the default has the
// embedding.  h_enc of a position that has not been through the thinking layers yet is kept
// (pending row = position - lo_len) and fed to them at the next full pass.
// ------------------------------------------------------------------------------------
// pend[b][newest - lo_len][:] = x_up[b][:]
__global__ void save_pending_kernel(const float *x_up, float *__restrict__ pend, int pend_cap, int H,
                                    const DevState *st) {
  const int b = blockIdx.x, r = st->newest - st->lo_len;
  if (r < 0 || r >= pend_cap) return;
  float *dst = pend + ((size_t)b * pend_cap + r) * H;
  for (int k = threadIdx.x; k < H; k += blockDim.x) dst[k] = x_up[(size_t)b * H + k];
}

// x_lo[b][r][:] = pend[b][r][:] for r < R - 1, x_up[b][:] for the newest row r = R - 1
__global__ void gather_pending_kernel(const float *__restrict__ pend, int pend_cap, const float *x_up, int R, int H,
                                      float *x_lo) {
  const int b = blockIdx.x / R, r = blockIdx.x % R;
  const float *src = r < R - 1 ? pend + ((size_t)b * pend_cap + r) * H : x_up + (size_t)b * H;
  float *dst = x_lo + (size_t)blockIdx.x * H;
  for (int k = threadIdx.x; k < H; k += blockDim.x) dst[k] = src[k];
}

// dst[i] = src[i] / dst[i] += src[i], n floats (n a multiple of 4)
__global__ void copy_rows_kernel(const float *__restrict__ src, float *__restrict__ dst, size_t n4, int accumulate) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    float4 v = reinterpret_cast<const float4 *>(src)[i];
    if (accumulate) {
      const float4 d = reinterpret_cast<const float4 *>(dst)[i];
      v.x += d.x; v.y += d.y; v.z += d.z; v.w += d.w;
    }
    reinterpret_cast<float4 *>(dst)[i] = v;
  }
}

// Eq. 3-4 over a chunk of rows of the masked parallel forward: row (b, r) sits at position
// p0 + r; at a mask position (inside the prompt, or (p - (P-1)) mod tau == 0: the anchors of
// Section 2.2) the decoding layers read h_think (x), or base + h_think with the literal sum of
// Eq. 4; elsewhere they read base (h_emb, or h_enc when encoding layers are reused).
__global__ void masked_select_kernel(float *x, const float *__restrict__ base, int R, int H, int p0, int P,
                                     int tau, int literal_sum) {
  const int r = blockIdx.x % R, p = p0 + r;
  const bool m = p < P || (p - (P - 1)) % tau == 0;
  float *xr = x + (size_t)blockIdx.x * H;
  const float *br = base + (size_t)blockIdx.x * H;
  if (m && !literal_sum) return;
  for (int k = threadIdx.x; k < H; k += blockDim.x) xr[k] = m ? br[k] + xr[k] : br[k];
}

// ------------------------------------------------------------------------------------
// a9 (second half): greedy pick, lowest index on ties; a10: feed the token back.
// ARGMAX_SLICES blocks per sequence each find the best of their slice of the vocabulary; the last of them to arrive
// picks among the slices, and the last of all advances the schedule's counters: one launch where a block of its own for
// each step took three.  The token goes to position n_known of the token buffer unless a forced token already sits
// there (teacher forcing), and to out_argmax if given.
// ------------------------------------------------------------------------------------
constexpr int ARGMAX_SLICES = 64;       // 151 936 logits of one sequence: 10 us with 16 slices

__device__ __forceinline__ void argmax_block_reduce(float best, int bi, float *sv, int *si) {
  sv[threadIdx.x] = best; si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = blockDim.x >> 1; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      float v2 = sv[threadIdx.x + s]; int i2 = si[threadIdx.x + s];
      if (v2 > sv[threadIdx.x] || (v2 == sv[threadIdx.x] && i2 < si[threadIdx.x])) {
        sv[threadIdx.x] = v2; si[threadIdx.x] = i2;
      }
    }
    __syncthreads();
  }
}

// a0: schedule counters after a pass (Section 2.2).  kind: 0 = prefill of P rows, 1 = full
// pass, 2 = decoding-layers-only pass.
__device__ __forceinline__ void advance_state(DevState *st, int kind, int P) {
  if (kind == 0) {
    st->n_known = P + 1; st->lo_len = P; st->up_len = P; st->cycle = 1;
    st->slot = 1 % st->tau; st->n_emitted = 1;
  } else {
    if (kind == 1) { st->lo_len = st->n_known; st->cycle += 1; }
    st->up_len = st->n_known;
    st->n_known += 1;
    st->slot = (st->slot + 1) % st->tau;
    st->n_emitted += 1;
  }
  st->newest = st->n_known - 1;
}

struct PickParams {
  float *part_val;                // [sequences][ARGMAX_SLICES]
  int *part_idx;
  unsigned int *arrived;          // [sequences + 1], zero between launches
  int *tokens;                    // null: the position holds its token already
  int max_seq;
  int *out_argmax;                // may be null
  int kind, P;                    // for advance_state
};

// grid (sequences, ARGMAX_SLICES), 256 threads
__global__ void argmax_kernel(const float *logits, int ldl, int V, DevState *st, SampleParams sp, PickParams pp) {
  pdl_enter();
  const int b = blockIdx.x, per = ((V + gridDim.y - 1) / gridDim.y + 3) & ~3;      // whole 16-byte loads
  const int i0 = blockIdx.y * per, i1 = min(V, i0 + per);
  const float *z = logits + (size_t)b * ldl;
  float best = -INFINITY;
  int bi = 0x7fffffff;
  const int position = st->n_known;                  // where the picked token will sit
  if (ldl % 4 == 0) {
    // four logits per load (the slice starts on a 16-byte boundary); indices rise within a thread, so the
    // first of equal values stays
    for (int i = i0 + 4 * threadIdx.x; i < i1; i += 4 * blockDim.x) {
      if (i + 4 <= i1) {
        const float4 q = *reinterpret_cast<const float4 *>(z + i);
        const float e[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float v = pick_value(e[j], i + j, position, b, sp);
          if (v > best) { best = v; bi = i + j; }
        }
      } else {
        for (int j = i; j < i1; ++j) {
          const float v = pick_value(z[j], j, position, b, sp);
          if (v > best) { best = v; bi = j; }
        }
      }
    }
  } else {
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      float v = pick_value(z[i], i, position, b, sp);
      if (v > best) { best = v; bi = i; }
    }
  }
  __shared__ float sv[256];
  __shared__ int si[256];
  argmax_block_reduce(best, bi, sv, si);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    pp.part_val[b * gridDim.y + blockIdx.y] = sv[0];
    pp.part_idx[b * gridDim.y + blockIdx.y] = si[0];
    __threadfence();                                  // this block's pair, and its read of n_known, before its arrival
    last = atomicInc(&pp.arrived[b], gridDim.y - 1) == gridDim.y - 1;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  best = -INFINITY;
  bi = 0x7fffffff;
  for (int i = threadIdx.x; i < gridDim.y; i += blockDim.x) {
    const float v = __ldcg(&pp.part_val[b * gridDim.y + i]);
    const int ix = __ldcg(&pp.part_idx[b * gridDim.y + i]);
    if (v > best || (v == best && ix < bi)) { best = v; bi = ix; }
  }
  argmax_block_reduce(best, bi, sv, si);
  if (threadIdx.x == 0) {
    const int pick = si[0] == 0x7fffffff ? 0 : si[0];
    if (pp.tokens) pp.tokens[(size_t)b * pp.max_seq + position] = pick;
    if (pp.out_argmax) pp.out_argmax[b] = pick;
    __threadfence();
    if (atomicInc(&pp.arrived[gridDim.x], gridDim.x - 1) == gridDim.x - 1) advance_state(st, pp.kind, pp.P);
  }
}

__global__ void set_int_kernel(int *p, int v) { *p = v; }

// out[b][i] = tokens[b][first + i], i < n  (the tokens a decode call produced)
__global__ void gather_tokens_kernel(const int *__restrict__ tokens, int max_seq, int first, int n,
                                     int ld_out, int *__restrict__ out) {
  int b = blockIdx.x;
  for (int i = threadIdx.x; i < n; i += blockDim.x) out[(size_t)b * ld_out + i] = tokens[(size_t)b * max_seq + first + i];
}

}  // namespace dmtd
