// Attention of one query row per sequence (bf16, head width 64): the last layer of an encoder whose items are pooled by
// token 0.  Only row 0 of that layer's output is read and only row 0 receives a gradient, so the layer needs keys and
// values of every token but one query: ctx = softmax(q K^T / sqrt(dh)) V, one row per item, and in the backward pass
// dV_j = P_j dctx, dK_j = dS_j q, dq = sum_j dS_j K_j.  No products to speak of: both kernels are bound by reading K and V
// (and writing dK and dV) once.  One block per item, one warp per head; eight lanes hold a 128-byte row, so a load
// instruction covers four rows, and consecutive heads' warps read consecutive pieces of the same rows.
// 1024 items of 64 tokens, width 768: 50 us forward and 90 us backward (61 and 92 with every chunk of rows requested when the
// one before had been worked on), against 86 and 200 us with all 64 queries; the
// products of the layer's projections shrink by a third as well (the encoder pass of two such layers 5.28 -> 4.80 ms).
#include "layers.h"
#include "tc_common.cuh"

namespace {

constexpr int DH = 64;
constexpr int kClsBlocks = kNumSMs * 4;          // blocks of the backward pass: one row of column sums each

__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 t = tc::unpack_bf16x2(w[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  return make_uint4(tc::pack_bf16x2(f[0], f[1]), tc::pack_bf16x2(f[2], f[3]), tc::pack_bf16x2(f[4], f[5]), tc::pack_bf16x2(f[6], f[7]));
}
__device__ __forceinline__ float dot8(const uint4& v, const float (&q)[8]) {
  float f[8];
  unpack8(v, f);
  float a = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) a = fmaf(f[i], q[i], a);
  return a;
}
// sum over the eight lanes that share a row
__device__ __forceinline__ float row_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 4);
}
__device__ __forceinline__ float all_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// the warp's scores sc[0 .. len) -> exp2(c (s - max)); returns their sum
__device__ __forceinline__ float softmax_scores(float* sc, int len, float c, int lane) {
  float m = -INFINITY;
  for (int j = lane; j < len; j += 32) m = fmaxf(m, sc[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float l = 0.f;
  for (int j = lane; j < len; j += 32) {
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"((sc[j] - m) * c));
    sc[j] = e;
    l += e;
  }
  return all_sum(l);
}

constexpr int ROWS = 4;                          // row groups of a chunk: 16 rows of 128 bytes
constexpr int CHUNK = 4 * ROWS;

// this lane's pieces of the rows j0 .. of one head's slice (zeros at and past len).  The next chunk is requested before the
// current one is worked on, across the softmax too: a warp waits for a chunk once, not once per chunk.  That costs the forward
// kernel registers and so blocks on an SM, which texts of a chunk or little more need: those fetch as they go (!AHEAD).
__device__ __forceinline__ void fetch_chunk(const bf16* __restrict__ base, int64_t ld, int j0, int len, int sub, uint4 (&v)[ROWS]) {
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const int j = j0 + 4 * i + sub;
    v[i] = j < len ? *reinterpret_cast<const uint4*>(base + j * ld) : make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ void take(uint4 (&v)[ROWS], const uint4 (&next)[ROWS]) {
#pragma unroll
  for (int i = 0; i < ROWS; ++i) v[i] = next[i];
}

template <bool AHEAD, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS) attn_cls_fwd_kernel(const bf16* __restrict__ q, const bf16* __restrict__ kv,
                                                          bf16* __restrict__ ctx, int n, int l_t, int d, float c,
                                                          const int32_t* __restrict__ seq_len, const int32_t* __restrict__ seq_off) {
  if (!chain_begin()) return;
  extern __shared__ float scores[];              // [heads][l_t]
  const int h = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane >> 3, p = lane & 7;
  float* sc = scores + h * l_t;
  const int64_t ld = 2 * (int64_t)d;
  for (int u = blockIdx.x; u < n; u += gridDim.x) {
    const int64_t row0 = seq_off ? (int64_t)seq_off[u] : (int64_t)u * l_t;
    const int len = seq_len ? seq_len[u] : l_t;
    const int64_t col = (int64_t)h * DH + p * 8;
    float qv[8];
    unpack8(*reinterpret_cast<const uint4*>(q + (int64_t)u * d + col), qv);
    const bf16* kb = kv + row0 * ld + col;
    float o[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    auto score = [&](int j0, const uint4 (&v)[ROWS]) {
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const float s = row_sum(dot8(v[i], qv));
        const int j = j0 + 4 * i + sub;
        if (p == 0 && j < len) sc[j] = s;
      }
    };
    auto add_values = [&](int j0, const uint4 (&v)[ROWS]) {
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const int j = j0 + 4 * i + sub;
        const float w = j < len ? sc[j] : 0.f;
        float f[8];
        unpack8(v[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) o[e] = fmaf(w, f[e], o[e]);
      }
    };
    float l;
    if constexpr (AHEAD) {
      uint4 v[ROWS], next[ROWS];
      fetch_chunk(kb, ld, 0, len, sub, v);
      for (int j0 = 0; j0 < len; j0 += CHUNK) {
        if (j0 + CHUNK < len) fetch_chunk(kb, ld, j0 + CHUNK, len, sub, next);
        else fetch_chunk(kb + d, ld, 0, len, sub, next);             // the first values
        score(j0, v);
        take(v, next);
      }
      __syncwarp();
      l = softmax_scores(sc, len, c, lane);
      __syncwarp();
      for (int j0 = 0; j0 < len; j0 += CHUNK) {
        if (j0 + CHUNK < len) fetch_chunk(kb + d, ld, j0 + CHUNK, len, sub, next);
        add_values(j0, v);
        take(v, next);
      }
    } else {
      for (int j0 = 0; j0 < len; j0 += CHUNK) {
        uint4 v[ROWS];
        fetch_chunk(kb, ld, j0, len, sub, v);
        score(j0, v);
      }
      __syncwarp();
      l = softmax_scores(sc, len, c, lane);
      __syncwarp();
      for (int j0 = 0; j0 < len; j0 += CHUNK) {
        uint4 v[ROWS];
        fetch_chunk(kb + d, ld, j0, len, sub, v);
        add_values(j0, v);
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      o[e] += __shfl_xor_sync(0xffffffffu, o[e], 8);
      o[e] += __shfl_xor_sync(0xffffffffu, o[e], 16);
      o[e] /= l;
    }
    if (sub == 0) *reinterpret_cast<uint4*>(ctx + (int64_t)u * d + col) = pack8(o);
    __syncwarp();                                // the scores are free for the next item
  }
}

__global__ void __launch_bounds__(512) attn_cls_bwd_kernel(const bf16* __restrict__ q, const bf16* __restrict__ kv,
                                                          const bf16* __restrict__ dctx, bf16* __restrict__ dq,
                                                          bf16* __restrict__ dkv, float* __restrict__ part, int n, int l_t, int d,
                                                          float c, float scale, const int32_t* __restrict__ seq_len,
                                                          const int32_t* __restrict__ seq_off) {
  if (!chain_begin()) return;
  extern __shared__ float scores[];              // [heads][2][l_t]: scores, later probabilities; dP, later dS
  const int h = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane >> 3, p = lane & 7;
  float* sc = scores + h * 2 * l_t;
  float* sd = sc + l_t;
  const int64_t ld = 2 * (int64_t)d;
  const int64_t col = (int64_t)h * DH + p * 8;
  float aq[8], ak[8], av[8];                     // column sums of dq, dK, dV over this block's items
#pragma unroll
  for (int e = 0; e < 8; ++e) aq[e] = ak[e] = av[e] = 0.f;
  for (int u = blockIdx.x; u < n; u += gridDim.x) {
    const int64_t row0 = seq_off ? (int64_t)seq_off[u] : (int64_t)u * l_t;
    const int len = seq_len ? seq_len[u] : l_t;
    float qv[8], gv[8];
    unpack8(*reinterpret_cast<const uint4*>(q + (int64_t)u * d + col), qv);
    unpack8(*reinterpret_cast<const uint4*>(dctx + (int64_t)u * d + col), gv);
    const bf16* kb = kv + row0 * ld + col;
    uint4 kk[ROWS], vv[ROWS], next_k[ROWS], next_v[ROWS];
    fetch_chunk(kb, ld, 0, len, sub, kk);
    fetch_chunk(kb + d, ld, 0, len, sub, vv);
    for (int j0 = 0; j0 < len; j0 += CHUNK) {
      const bool more = j0 + CHUNK < len;
      fetch_chunk(kb, ld, more ? j0 + CHUNK : 0, len, sub, next_k);          // at the end: the first keys once more, from L2
      if (more) fetch_chunk(kb + d, ld, j0 + CHUNK, len, sub, next_v);
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const float s = row_sum(dot8(kk[i], qv)), t = row_sum(dot8(vv[i], gv));
        const int j = j0 + 4 * i + sub;
        if (p == 0 && j < len) { sc[j] = s; sd[j] = t; }
      }
      take(kk, next_k);
      take(vv, next_v);
    }
    __syncwarp();
    const float inv = 1.f / softmax_scores(sc, len, c, lane);
    float delta = 0.f;
    for (int j = lane; j < len; j += 32) {       // each lane meets its own scores again: no barrier needed before
      const float pr = sc[j] * inv;
      sc[j] = pr;
      delta = fmaf(pr, sd[j], delta);
    }
    delta = all_sum(delta);
    float sum_p = 0.f, sum_ds = 0.f;
    for (int j = lane; j < len; j += 32) {
      const float ds = sc[j] * (sd[j] - delta) * scale;
      sd[j] = ds;
      sum_p += sc[j];
      sum_ds += ds;
    }
    sum_p = all_sum(sum_p);
    sum_ds = all_sum(sum_ds);
    __syncwarp();
    float o[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    bf16* db = dkv + row0 * ld + col;
    for (int j0 = 0; j0 < len; j0 += CHUNK) {
      if (j0 + CHUNK < len) fetch_chunk(kb, ld, j0 + CHUNK, len, sub, next_k);
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const int j = j0 + 4 * i + sub;
        if (j < len) {
          const float pr = sc[j], ds = sd[j];
          float f[8], dk[8], dv[8];
          unpack8(kk[i], f);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            o[e] = fmaf(ds, f[e], o[e]);
            dk[e] = ds * qv[e];
            dv[e] = pr * gv[e];
          }
          *reinterpret_cast<uint4*>(db + j * ld) = pack8(dk);
          *reinterpret_cast<uint4*>(db + d + j * ld) = pack8(dv);
        }
      }
      take(kk, next_k);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      o[e] += __shfl_xor_sync(0xffffffffu, o[e], 8);
      o[e] += __shfl_xor_sync(0xffffffffu, o[e], 16);
      aq[e] += o[e];
      ak[e] = fmaf(sum_ds, qv[e], ak[e]);
      av[e] = fmaf(sum_p, gv[e], av[e]);
    }
    if (sub == 0) *reinterpret_cast<uint4*>(dq + (int64_t)u * d + col) = pack8(o);
    __syncwarp();
  }
  if (sub < 3) {
    float* out = part + (int64_t)blockIdx.x * 3 * d + (int64_t)sub * d + col;
#pragma unroll
    for (int e = 0; e < 8; ++e) out[e] = sub == 0 ? aq[e] : (sub == 1 ? ak[e] : av[e]);
  }
}

// X[row(u), :] += r[u, :], fp32, row(u) = rows[u] or u * stride
__global__ void add_strided_rows_kernel(const float4* __restrict__ r, float4* __restrict__ X, int64_t n, int64_t stride, int words,
                                        const int32_t* __restrict__ rows) {
  if (!chain_begin()) return;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * words) return;
  const int64_t u = i / words;
  const int c = (int)(i - u * words);
  float4* x = X + (rows ? (int64_t)rows[u] : u * stride) * words + c;
  const float4 a = r[i];
  float4 b = *x;
  b.x += a.x; b.y += a.y; b.z += a.z; b.w += a.w;
  *x = b;
}

constexpr size_t kClsSmemMost = 96 * 1024;       // the kernels' limit is set to this, whatever a call needs: other threads launch them too
size_t cls_smem(int heads, int l_t, int arrays) { return (size_t)heads * l_t * arrays * sizeof(float); }

}  // namespace

bool attention_cls_supported(int l_t, int d, int n_heads) {
  return n_heads > 0 && n_heads <= 16 && d == n_heads * DH && cls_smem(n_heads, l_t, 2) <= kClsSmemMost;
}

gram_status attention_cls_forward(gram_ctx* ctx, const void* q, const void* kv, void* out, int n, int l_t, int d, int n_heads,
                                  const int32_t* seq_len, const int32_t* seq_off, cudaStream_t st) {
  if (n == 0) return GRAM_OK;
  const size_t smem = cls_smem(n_heads, l_t, 1);
  ProfScope prof(ctx, GRAM_K_ATTENTION, 4.0 * (double)n * l_t * d, 1, st, "attn_cls_fwd");
  // Short texts want blocks on the SM more than rows on their way.  32 768 rows, 12 heads, us as they go / ahead: texts of 8 tokens
  // 41 / 46, of 2 to 16 22 / 23, of 24 30 / 31, of 32 33 / 27, of 64 29 / 25, of 100 40 / 23.  Up to 12 heads 56 registers let three
  // blocks share an SM (with 64 registers and two: 48 tokens 31, 25 this way).
  auto kern = l_t < 24 ? attn_cls_fwd_kernel<false, 512, 0> : (n_heads <= 12 ? attn_cls_fwd_kernel<true, 384, 3> : attn_cls_fwd_kernel<true, 512, 2>);
  if (smem > 48 * 1024) GRAM_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClsSmemMost));
  launch_chain(kern, n, n_heads * 32, smem, st, (const bf16*)q, (const bf16*)kv, (bf16*)out, n, l_t, d,
                                                     1.4426950408889634f / sqrtf((float)DH), seq_len, seq_off);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

gram_status attention_cls_backward(gram_ctx* ctx, const void* q, const void* kv, const void* dctx, void* dq, void* dkv, float* part,
                                   int64_t part_cap_rows, int64_t* part_rows, int n, int l_t, int d, int n_heads,
                                   const int32_t* seq_len, const int32_t* seq_off, cudaStream_t st) {
  *part_rows = 0;
  if (n == 0) return GRAM_OK;
  int64_t blocks = n < kClsBlocks ? n : kClsBlocks;
  if (blocks > part_cap_rows) blocks = part_cap_rows;
  if (blocks < 1) return gram_set_error(ctx, "attention backward: no room for the column sums"), GRAM_ERR_WORKSPACE;
  const size_t smem = cls_smem(n_heads, l_t, 2);
  ProfScope prof(ctx, GRAM_K_ATTENTION, 10.0 * (double)n * l_t * d, 1, st, "attn_cls_bwd");
  if (smem > 48 * 1024) GRAM_CUDA(ctx, cudaFuncSetAttribute(attn_cls_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClsSmemMost));
  launch_chain(attn_cls_bwd_kernel, (unsigned)blocks, n_heads * 32, smem, st, (const bf16*)q, (const bf16*)kv, (const bf16*)dctx, (bf16*)dq,
                                                                    (bf16*)dkv, part, n, l_t, d, 1.4426950408889634f / sqrtf((float)DH),
                                                                    1.f / sqrtf((float)DH), seq_len, seq_off);
  GRAM_LAUNCH_CHECK(ctx);
  *part_rows = blocks;
  return GRAM_OK;
}

gram_status add_strided_rows(gram_ctx* ctx, const float* r, int64_t n, int64_t stride, const int32_t* rows, int d, float* X,
                             cudaStream_t st) {
  if (n == 0) return GRAM_OK;
  if (d % 4) return gram_set_error(ctx, "row sum: d must be a multiple of 4"), GRAM_ERR_ARG;
  ProfScope prof(ctx, GRAM_K_OTHER, 12.0 * (double)n * d, 1, st);
  launch_chain(add_strided_rows_kernel, (unsigned)ceil_div64(n * (d / 4), 256), 256, 0, st, (const float4*)r, (float4*)X, n, stride, d / 4, rows);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}
