// Matrix products.  bf16: a persistent, warp-specialised tcgen05 kernel (one TMA producer warp, one
// MMA-issuing warp, eight epilogue warps; operands staged in 128-byte-swizzled shared memory by TMA,
// fp32 accumulators double-buffered in tensor memory so that the epilogue of one tile overlaps the
// main loop of the next).  fp32: a plain tiled CUDA-core kernel for the small fp32 configuration.
#include <cuda.h>
#include <stdlib.h>

#include "gemm.h"
#include "tc_common.cuh"

namespace {
using namespace tc;

// ============================================================================================
// fp32 CUDA-core kernel: C(m, n) = sum_k A(m, k) * B(n, k), generic strides
// ============================================================================================
struct EpiDev {
  const float* bias;
  const float* res;
  const float* res_mean;
  const float* res_rstd;
  const float* res_gamma;
  const float* res_beta;
  void* pre;
  const void* dgelu_pre;
  void* copy_out;
  float* colsum_part;
  int gelu;
  int accumulate;
};

template <typename CT> __device__ __forceinline__ float ld_c(const CT* p);
template <> __device__ __forceinline__ float ld_c<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ld_c<bf16>(const bf16* p) { return __bfloat162float(*p); }
template <typename CT> __device__ __forceinline__ void st_c(CT* p, float v);
template <> __device__ __forceinline__ void st_c<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void st_c<bf16>(bf16* p, float v) { *p = __float2bfloat16(v); }

// one element; CT is C's type, OT the operands' type
template <typename CT, typename OT>
__device__ __forceinline__ void epilogue_store(const EpiDev& e, CT* C, int64_t ldc, int64_t m, int n, float acc) {
  float v = acc + (e.bias ? e.bias[n] : 0.f);
  const int64_t o = m * ldc + n;
  if (e.gelu) {
    if (e.pre) st_c<OT>(reinterpret_cast<OT*>(e.pre) + o, gelu_grad_f(v));
    v = gelu_f(v);
  }
  if (e.dgelu_pre) v *= ld_c<OT>(reinterpret_cast<const OT*>(e.dgelu_pre) + o);
  if (e.res) {
    float r = e.res[o];
    if (e.res_mean) r = (r - e.res_mean[m]) * e.res_rstd[m] * e.res_gamma[n] + e.res_beta[n];
    v += r;
  }
  if (e.accumulate) v += ld_c<CT>(C + o);
  st_c<CT>(C + o, v);
  if (e.copy_out) st_c<OT>(reinterpret_cast<OT*>(e.copy_out) + o, v);
}

// four consecutive columns n..n+3 of row m (n, ldc multiples of 4): the unit of the coalesced epilogue
__device__ __forceinline__ void ld4(const float* p, float (&x)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
}
__device__ __forceinline__ void ld4(const bf16* p, float (&x)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 f0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 f1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  x[0] = f0.x; x[1] = f0.y; x[2] = f1.x; x[3] = f1.y;
}
__device__ __forceinline__ void st4(float* p, const float (&x)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void st4(bf16* p, const float (&x)[4]) {
  __nv_bfloat162 h0 = __floats2bfloat162_rn(x[0], x[1]), h1 = __floats2bfloat162_rn(x[2], x[3]);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&h0), *reinterpret_cast<uint32_t*>(&h1));
}

// GELU and its derivative for the tensor-core epilogue.  erf comes from the rational approximation
// 7.1.26 of Abramowitz & Stegun, erf(y) = 1 - (a1 t + ... + a5 t^5) exp(-y^2), t = 1 / (1 + p y), whose
// absolute error is below 1.5e-7: far under the bf16 resolution of the values that are stored.  With
// y = |x| / sqrt(2) the exponential exp(-x^2 / 2) is also the Gaussian density the derivative needs.
__device__ __forceinline__ void gelu_parts(float x, float& cdf, float& pdf) {
  const float ax = fabsf(x);
  float ex, t;                                            // flush-to-zero forms: one MUFU each, no range fix-up
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(x * x * -0.72134752f));            // exp(-x^2 / 2)
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(fmaf(0.3275911f * 0.70710678f, ax, 1.f)));
  const float poly = t * (0.254829592f + t * (-0.284496736f + t * (1.421413741f + t * (-1.453152027f + t * 1.061405429f))));
  const float erf_abs = 1.f - poly * ex;                  // erf(|x| / sqrt 2)
  cdf = 0.5f * (1.f + copysignf(erf_abs, x));
  pdf = 0.39894228f * ex;
}

// The same for two values at a time with the packed fp32 instructions of sm_100 (two lanes of one 64-bit
// register): x holds the two pre-activations; on return g = gelu(x), dg = gelu'(x).  Half the instruction
// slots of the scalar form, which is what bounds the epilogue of the first feed-forward product.
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_const(float c) {
  const uint64_t u = (uint64_t)__float_as_uint(c);
  return u | (u << 32);
}
template <bool DERIVATIVE> __device__ __forceinline__ void gelu_pair(uint64_t x, uint64_t& g, uint64_t& dg) {
  float e0, e1, y0, y1;
  f2_unpack(f2_mul(f2_mul(x, x), f2_const(-0.72134752f)), e0, e1);
  asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(e0));                          // exp(-x^2 / 2)
  asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(e1));
  const uint64_t ex = f2_pack(e0, e1);
  f2_unpack(f2_fma(x & 0x7FFFFFFF7FFFFFFFull, f2_const(0.3275911f * 0.70710678f), f2_const(1.f)), y0, y1);
  asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(y0));
  asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(y1));
  const uint64_t t = f2_pack(y0, y1);
  uint64_t p = f2_fma(t, f2_const(1.061405429f), f2_const(-1.453152027f));
  p = f2_fma(p, t, f2_const(1.421413741f));
  p = f2_fma(p, t, f2_const(-0.284496736f));
  p = f2_fma(p, t, f2_const(0.254829592f));
  p = f2_mul(p, t);
  const uint64_t h = f2_fma(f2_mul(p, ex), f2_const(-0.5f), f2_const(0.5f));    // erf(|x| / sqrt 2) / 2
  const uint64_t cdf = f2_add(h | (x & 0x8000000080000000ull), f2_const(0.5f));   // 1/2 + sign(x) * h
  g = f2_mul(x, cdf);
  if (DERIVATIVE) dg = f2_fma(f2_mul(x, ex), f2_const(0.39894228f), cdf);
}
__device__ __forceinline__ uint32_t f2_to_bf16x2(uint64_t v) {
  float lo, hi;
  f2_unpack(v, lo, hi);
  return pack_bf16x2(lo, hi);
}

// what one lane reads before it may store anything for its 4 columns of one row: the residual, the
// saved GELU derivative or the old value of C (the tensor-core path takes at most one of the three)
struct EpiLoads {
  float aux[4];
};
template <typename CT>
__device__ __forceinline__ void epilogue_load4(const EpiDev& e, const CT* C, int64_t ldc, int64_t m, int n, EpiLoads& L) {
  const int64_t o = m * ldc + n;
  if (e.res) ld4(e.res + o, L.aux);
  else if (e.dgelu_pre) ld4(reinterpret_cast<const bf16*>(e.dgelu_pre) + o, L.aux);
  else if (e.accumulate) ld4(reinterpret_cast<const float*>(C) + o, L.aux);      // accumulation is offered for fp32 C only
}
template <typename CT>
__device__ __forceinline__ void epilogue_store4(const EpiDev& e, CT* C, int64_t ldc, int64_t m, int n, float (&v)[4],
                                                const EpiLoads& L, const float (&bias)[4], const float (&gam)[4],
                                                const float (&bet)[4], float mu, float rs) {
  const int64_t o = m * ldc + n;
  if (e.bias) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] += bias[i];
  }
  if (e.gelu) {
    float dg[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float c, p;
      gelu_parts(v[i], c, p);
      dg[i] = c + v[i] * p;        // gelu'(v), kept for the backward pass
      v[i] = v[i] * c;             // gelu(v)
    }
    if (e.pre) st4(reinterpret_cast<bf16*>(e.pre) + o, dg);
  }
  if (e.res) {
    if (e.res_mean) {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] += (L.aux[i] - mu) * rs * gam[i] + bet[i];
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] += L.aux[i];
    }
  } else if (e.dgelu_pre) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] *= L.aux[i];
  } else if (e.accumulate) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] += L.aux[i];
  }
  st4(C + o, v);
  if (e.copy_out) st4(reinterpret_cast<bf16*>(e.copy_out) + o, v);
}

// A tile of TILE x TILE results per block, TILE^2 / 16 threads with 4 x 4 results each; a k-block at a time through two
// shared-memory buffers, the next one fetched into registers (16-byte loads where the rows allow them) while the current
// ones are multiplied.  The configurations that run in fp32 are small, so what bounds these products is the chain of
// k-blocks of one block and the number of blocks, not the FMA rate: the K range is therefore cut over a cluster of up
// to 16 blocks, whose partial tiles are added through distributed shared memory in ascending order of the block's rank
// (the order depends on the sizes alone), each block finishing its share of the tile's rows.  One launch, no
// workspace.  Weight gradients of the check's model (64 x 64 to 256 x 64 over about 900 rows): 130 to 185 us each with
// one 64 x 64 block per tile and a synchronous load per k-block, 6 to 7 us now; the
// model's whole training step 2.49 -> 0.48 ms with the chain of launches below, 0.43 -> 0.39 with gradients' products in pairs
// (gemm_f32_pair_kernel).
// What a k-block waits for is its loads: 32 k at a time in the small tiles, and up to four groups of 64 threads with a k-block each,
// so that K = 128 can take one round of loads and no cluster; the groups' tiles are added in ascending order in shared memory.
// Which products get groups: f32_plan.
constexpr int F32_MAX_SPLIT = 16;
template <int TILE, int NG = 1> struct F32Cfg {
  static constexpr int SK = TILE == 32 ? 32 : 16;          // k of one k-block
  static constexpr int GROUP = TILE * TILE / 16;           // threads that hold one copy of the tile
  static constexpr int GROUPS = NG;                        // copies, each over its own k-blocks
  static constexpr int THREADS = GROUP * GROUPS;
  static constexpr int BUFS = GROUPS == 1 ? 2 : 1;         // operand buffers per group
  static constexpr int LD = TILE + 4;                      // keeps rows 16-byte aligned
  static constexpr int NV = TILE * SK / 4 / GROUP;         // 16-byte pieces per thread, operand and k-block
};

// piece `idx` of an operand's k-block: rows r0 .. of a matrix with leading dimension ld, k from k0; zeros outside
template <int TILE, bool KMAJOR>
__device__ __forceinline__ float4 f32_fetch(const float* __restrict__ X, int64_t ld, int64_t r0, int64_t rows, int64_t k0,
                                            int64_t kend, int idx, bool vec) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int KQ = F32Cfg<TILE>::SK / 4;                 // pieces of one row's k-block
  const int64_t r = r0 + (KMAJOR ? idx / KQ : 4 * (idx % (TILE / 4))), k = k0 + (KMAJOR ? 4 * (idx % KQ) : idx / (TILE / 4));
  if (r >= rows || k >= kend) return v;
  const float* p = KMAJOR ? X + r * ld + k : X + k * ld + r;
  const int64_t left = KMAJOR ? kend - k : rows - r;       // elements of the piece that exist
  if (vec && left >= 4) return *reinterpret_cast<const float4*>(p);
  v.x = p[0];
  if (left > 1) v.y = p[1];
  if (left > 2) v.z = p[2];
  if (left > 3) v.w = p[3];
  return v;
}
template <int TILE, bool KMAJOR>
__device__ __forceinline__ void f32_stage(float* s, int idx, float4 v) {
  constexpr int LD = F32Cfg<TILE>::LD;
  if (KMAJOR) {
    constexpr int KQ = F32Cfg<TILE>::SK / 4;
    float* q = s + 4 * (idx % KQ) * LD + idx / KQ;
    q[0] = v.x; q[LD] = v.y; q[2 * LD] = v.z; q[3 * LD] = v.w;
  } else {
    *reinterpret_cast<float4*>(s + (idx / (TILE / 4)) * LD + 4 * (idx % (TILE / 4))) = v;
  }
}

// The epilogue for four columns of a row at a time (vec_e launches: every matrix and vector it touches allows 16-byte
// accesses, and at most one of residual, GELU derivative and accumulation is asked for).  What it reads per element is
// fetched ahead (f32_aux), for all of a thread's rows before the first of them is stored: element by element, every load
// waits for the store before it.
__device__ __forceinline__ float4 f32_ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 f32_aux(const EpiDev& e, const float* C, int64_t o) {
  if (e.res) return f32_ld4(e.res + o);
  if (e.dgelu_pre) return f32_ld4(reinterpret_cast<const float*>(e.dgelu_pre) + o);
  if (e.accumulate) return f32_ld4(C + o);
  return make_float4(0.f, 0.f, 0.f, 0.f);
}
struct F32Cols { float4 bias, gamma, beta; };           // of the thread's four columns
__device__ __forceinline__ F32Cols f32_cols(const EpiDev& e, int n) {
  F32Cols c;
  c.bias = e.bias ? f32_ld4(e.bias + n) : make_float4(0.f, 0.f, 0.f, 0.f);
  c.gamma = e.res_mean ? f32_ld4(e.res_gamma + n) : make_float4(0.f, 0.f, 0.f, 0.f);
  c.beta = e.res_mean ? f32_ld4(e.res_beta + n) : make_float4(0.f, 0.f, 0.f, 0.f);
  return c;
}
__device__ __forceinline__ void f32_finish(const EpiDev& e, float* C, int64_t o, const float (&acc)[4], const float4& aux4,
                                           const F32Cols& c, float mu, float rs) {
  const float bias[4] = {c.bias.x, c.bias.y, c.bias.z, c.bias.w}, gam[4] = {c.gamma.x, c.gamma.y, c.gamma.z, c.gamma.w};
  const float bet[4] = {c.beta.x, c.beta.y, c.beta.z, c.beta.w}, aux[4] = {aux4.x, aux4.y, aux4.z, aux4.w};
  float v[4], dg[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[i] = acc[i] + bias[i];
    if (e.gelu) {
      dg[i] = gelu_grad_f(v[i]);
      v[i] = gelu_f(v[i]);
    }
    if (e.res) v[i] += e.res_mean ? (aux[i] - mu) * rs * gam[i] + bet[i] : aux[i];
    else if (e.dgelu_pre) v[i] *= aux[i];
    else if (e.accumulate) v[i] += aux[i];
  }
  if (e.gelu && e.pre) st4(reinterpret_cast<float*>(e.pre) + o, dg);
  st4(C + o, v);
  if (e.copy_out) st4(reinterpret_cast<float*>(e.copy_out) + o, v);
}

struct F32Prod {
  const float* A;
  int64_t lda;
  const float* B;
  int64_t ldb;
  float* C;
  int64_t ldc, M, K, k_per_part;
  int32_t N, vec_a, vec_b, vec_e;
  float* row_sums;               // row_sums[m] += the sum of A(m, k) over k (may be null; SUMS only)
  int32_t fold;                  // FOLD: k-blocks of a group that are added up in one chain
  EpiDev e;
};
template <int TILE, int NG> using F32Smem = float[NG][F32Cfg<TILE, NG>::BUFS][2][F32Cfg<TILE, NG>::SK * F32Cfg<TILE, NG>::LD];

// One tile of a product by one block, or by `parts` blocks of a cluster whose ranks begin at rank0, this one being number `part`.
// All threads of the blocks call it; with one part it does not touch the cluster's barrier.
// FOLD: after every `fold` k-blocks of a group their sum goes to the sum of those before, so that few parts of a long K are no longer
// a chain of additions than many.  SUMS: row_sums may be asked for.
template <int TILE, bool A_K, bool B_K, int NG, bool FOLD, bool SUMS>
__device__ __forceinline__ void f32_tile(const F32Prod& p, int64_t m0, int64_t n0, int part_no, int parts, int rank0, F32Smem<TILE, NG>& sm) {
  using Cfg = F32Cfg<TILE, NG>;
  constexpr int LD = Cfg::LD, NV = Cfg::NV, T = Cfg::GROUP, G = Cfg::GROUPS, SK = Cfg::SK, BUFS = Cfg::BUFS;
  static_assert(sizeof(sm) >= sizeof(float) * G * TILE * LD, "the partial tiles reuse the operand buffers");
  const float* __restrict__ A = p.A;
  const float* __restrict__ B = p.B;
  float* C = p.C;
  const EpiDev& e = p.e;
  const int64_t lda = p.lda, ldb = p.ldb, ldc = p.ldc, M = p.M, K = p.K;
  const int N = p.N, vec_a = p.vec_a, vec_b = p.vec_b, vec_e = p.vec_e;
  const int group = threadIdx.x / T, tid = threadIdx.x % T, tx = tid % (TILE / 4), ty = tid / (TILE / 4);
  const int64_t kb = (int64_t)part_no * p.k_per_part, ke = min(kb + p.k_per_part, K);
  static_assert(!SUMS || G > 1, "the row sums go through the groups' partial tiles");
  const bool sums = SUMS && p.row_sums != nullptr && n0 == 0;
  float asum = 0.f;                                        // of this thread's row of A
  float acc[4][4] = {}, folded[FOLD ? 4 : 1][4] = {};
  int chain = p.fold;
  float4 fa[NV], fb[NV];
  auto fetch = [&](int64_t k0) {                           // this group's k-block of the round that starts at k0 (zeros from ke on)
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      fa[i] = f32_fetch<TILE, A_K>(A, lda, m0, M, k0 + group * SK, ke, tid + i * T, vec_a);
      fb[i] = f32_fetch<TILE, B_K>(B, ldb, n0, N, k0 + group * SK, ke, tid + i * T, vec_b);
    }
  };
  fetch(kb);
  int buf = 0;
  for (int64_t k0 = kb; k0 < ke; k0 += SK * G, buf ^= BUFS - 1) {
    if (BUFS == 1 && k0 > kb) __syncthreads();             // the buffer has been read
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      f32_stage<TILE, A_K>(sm[group][buf][0], tid + i * T, fa[i]);
      f32_stage<TILE, B_K>(sm[group][buf][1], tid + i * T, fb[i]);
    }
    __syncthreads();                 // with two buffers also: everyone is done with the other one, which the next round fills
    if (k0 + SK * G < ke) fetch(k0 + SK * G);
    if (G > 1 && k0 + group * SK >= ke) continue;          // the last round may have fewer k-blocks than groups
    if (sums && tid < TILE) {
      float a[4] = {};                                     // every fourth k
#pragma unroll
      for (int k = 0; k < SK; ++k) a[k & 3] += sm[group][buf][0][k * LD + tid];
      asum += (a[0] + a[1]) + (a[2] + a[3]);
    }
#pragma unroll
    for (int k = 0; k < SK; ++k) {
      const float4 a4 = *reinterpret_cast<const float4*>(&sm[group][buf][0][k * LD + 4 * ty]);
      const float4 b4 = *reinterpret_cast<const float4*>(&sm[group][buf][1][k * LD + 4 * tx]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if constexpr (FOLD) {
      if (--chain == 0) {
        chain = p.fold;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) { folded[i][j] += acc[i][j]; acc[i][j] = 0.f; }
      }
    }
  }
  if constexpr (FOLD) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += folded[i][j];
  }
  float* part = &sm[0][0][0][0];
  // the groups' sum of four columns of row r of the tile
  auto group_sum = [&](int r, int c) {
    float4 v = *reinterpret_cast<const float4*>(part + r * LD + c);
#pragma unroll
    for (int g = 1; g < G; ++g) {
      const float4 x = *reinterpret_cast<const float4*>(part + g * (TILE * LD) + r * LD + c);
      v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
    }
    return v;
  };
  constexpr int TALL = Cfg::THREADS;
  if (G > 1) {                     // a row's sum of A takes the first column of the padding
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<float4*>(part + group * (TILE * LD) + (4 * ty + i) * LD + 4 * tx) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (sums && tid < TILE) part[group * (TILE * LD) + tid * LD + TILE] = asum;
    __syncthreads();
#pragma unroll
    for (int idx = threadIdx.x; idx < TILE * TILE / 4; idx += TALL) {
      const int r = idx / (TILE / 4), c = 4 * (idx % (TILE / 4));
      const float4 v4 = group_sum(r, c);
      if (sums && c == 0) {
        float s = part[r * LD + TILE];
#pragma unroll
        for (int g = 1; g < G; ++g) s += part[g * (TILE * LD) + r * LD + TILE];
        if (parts > 1) part[r * LD + TILE] = s;
        else if (m0 + r < M) p.row_sums[m0 + r] += s;
      }
      if (parts > 1) {
        *reinterpret_cast<float4*>(part + r * LD + c) = v4;  // only this thread reads these four places
        continue;
      }
      const int64_t m = m0 + r, n = n0 + c;
      if (m >= M || n >= N) continue;
      const float v[4] = {v4.x, v4.y, v4.z, v4.w};
      if (vec_e) {
        f32_finish(e, C, m * ldc + n, v, f32_aux(e, C, m * ldc + n), f32_cols(e, (int)n), e.res_mean ? e.res_mean[m] : 0.f,
                   e.res_mean ? e.res_rstd[m] : 1.f);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (n + j < N) epilogue_store<float, float>(e, C, ldc, m, (int)n + j, v[j]);
      }
    }
    if (parts == 1) return;
  }
  const int splits = parts;
  if (splits == 1) {
    if (vec_e) {
      const int64_t n = n0 + 4 * tx;
      if (n >= N) return;                        // N is a multiple of 4
      const F32Cols cols = f32_cols(e, (int)n);
      float4 aux[4];
      float mu[4], rs[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int64_t m = m0 + 4 * ty + i;
        const bool ok = m < M;
        aux[i] = ok ? f32_aux(e, C, m * ldc + n) : make_float4(0.f, 0.f, 0.f, 0.f);
        mu[i] = ok && e.res_mean ? e.res_mean[m] : 0.f;
        rs[i] = ok && e.res_mean ? e.res_rstd[m] : 1.f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int64_t m = m0 + 4 * ty + i;
        if (m < M) f32_finish(e, C, m * ldc + n, acc[i], aux[i], cols, mu[i], rs[i]);
      }
      return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t m = m0 + 4 * ty + i, n = n0 + 4 * tx + j;
        if (m < M && n < N) epilogue_store<float, float>(e, C, ldc, m, (int)n, acc[i][j]);
      }
    return;
  }
  if (G == 1) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<float4*>(part + (4 * ty + i) * LD + 4 * tx) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
  const int rows = TILE / splits, r0 = part_no * rows;             // this block's share of the tile's rows
  const int count = rows * (TILE / 4);                             // four columns of a row each
  struct Out {
    int r, c;
    int64_t m, n;
    bool ok;
    float4 aux;
    F32Cols cols;
    float mu, rs, sum;
  };
  auto output = [&](int idx) {
    Out o;
    o.r = r0 + idx / (TILE / 4);
    o.c = 4 * (idx % (TILE / 4));
    o.m = m0 + o.r;
    o.n = n0 + o.c;
    o.ok = o.m < M && o.n < N;
    o.aux = make_float4(0.f, 0.f, 0.f, 0.f);
    o.cols = {o.aux, o.aux, o.aux};
    o.mu = 0.f; o.rs = 1.f; o.sum = 0.f;
    if (vec_e && o.ok) {
      o.aux = f32_aux(e, C, o.m * ldc + o.n);
      o.cols = f32_cols(e, (int)o.n);
      if (e.res_mean) { o.mu = e.res_mean[o.m]; o.rs = e.res_rstd[o.m]; }
    }
    if (sums && o.c == 0 && o.m < M) o.sum = p.row_sums[o.m];
    return o;
  };
  Out o;
  int idx = threadIdx.x;
  if (idx < count) o = output(idx);                                // what the epilogue reads is fetched before the wait for the others
  gram_cluster_sync();
  while (idx < count) {
    const uint32_t at = smem_u32(part + o.r * LD + o.c);
    float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s0 = 0; s0 < F32_MAX_SPLIT; s0 += 8) {                // eight parts on their way at once, added in order
      if (s0 >= splits) break;
      float4 x[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        x[s] = make_float4(0.f, 0.f, 0.f, 0.f);
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 a;\n\tsetp.lt.s32 p, %5, %6;\n\tmapa.shared::cluster.u32 a, %4, %7;\n\t"
                     "@p ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [a];\n\t}"
                     : "+f"(x[s].x), "+f"(x[s].y), "+f"(x[s].z), "+f"(x[s].w)
                     : "r"(at), "r"(s0 + s), "r"(splits), "r"(rank0 + min(s0 + s, splits - 1))
                     : "memory");
      }
#pragma unroll
      for (int s = 0; s < 8; ++s)
        if (s0 + s < splits) { v[0] += x[s].x; v[1] += x[s].y; v[2] += x[s].z; v[3] += x[s].w; }
    }
    if (sums && o.c == 0) {
      const uint32_t at_sum = smem_u32(part + o.r * LD + TILE);
      float x[F32_MAX_SPLIT], a = 0.f;
#pragma unroll
      for (int s = 0; s < F32_MAX_SPLIT; ++s) {
        x[s] = 0.f;
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 a;\n\tsetp.lt.s32 p, %2, %3;\n\tmapa.shared::cluster.u32 a, %1, %4;\n\t"
                     "@p ld.shared::cluster.f32 %0, [a];\n\t}"
                     : "+f"(x[s])
                     : "r"(at_sum), "r"(s), "r"(splits), "r"(rank0 + min(s, splits - 1))
                     : "memory");
      }
#pragma unroll
      for (int s = 0; s < F32_MAX_SPLIT; ++s) a += x[s];
      if (o.m < M) p.row_sums[o.m] = o.sum + a;
    }
    if (o.ok) {
      if (vec_e) {
        f32_finish(e, C, o.m * ldc + o.n, v, o.aux, o.cols, o.mu, o.rs);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (o.n + q < N) epilogue_store<float, float>(e, C, ldc, o.m, (int)o.n + q, v[q]);
      }
    }
    idx += TALL;
    if (idx < count) o = output(idx);
  }
  // no block may leave while another still reads its partial tile
  gram_cluster_sync();
}

template <int TILE, bool A_K, bool B_K, int NG>
__global__ void __launch_bounds__(F32Cfg<TILE, NG>::THREADS) gemm_f32_kernel(const __grid_constant__ F32Prod p) {
  if (!chain_begin()) return;
  __shared__ __align__(16) F32Smem<TILE, NG> sm;           // [group][buffer][operand]; later the groups' partial tiles
  f32_tile<TILE, A_K, B_K, NG, false, false>(p, (int64_t)blockIdx.y * TILE, (int64_t)blockIdx.x * TILE, blockIdx.z, gridDim.z, 0, sm);
}
// Tiles of 64 x 64 with room for PER_SM blocks an SM: two have the registers to keep their loads apart, three take half as long again
// for a round of blocks, so three go where that makes fewer rounds by more than that.  256 columns over 768: 188 blocks 53.8 us
// with two and 59.0 with three, 440 blocks 107 and 82.
template <bool A_K, bool B_K, int PER_SM>
__global__ void __launch_bounds__(F32Cfg<64>::THREADS, PER_SM) gemm_f32_wide_kernel(const __grid_constant__ F32Prod p) {
  if (!chain_begin()) return;
  __shared__ __align__(16) F32Smem<64, 1> sm;
  f32_tile<64, A_K, B_K, 1, false, false>(p, (int64_t)blockIdx.y * 64, (int64_t)blockIdx.x * 64, blockIdx.z, gridDim.z, 0, sm);
}

// The two products that read one gradient dY [T, N]: dW [N, K] += dY^T X (product w; its row sums are the bias gradient) and
// dX [T, K] = dY W (product x), in one launch.  Neither fills the chip in the models that run in fp32, and each is a chain of launch,
// loads and exchange of partial sums: side by side they take little more than the longer one (64 x 256 and 256 x 64 over 900
// rows: 9.0 us where the two took 11.3 and the bias gradient's sums, two launches more, 5).  By this alone the check's step went from 429 to
// 386 us, 87 launches to 65, steps of other widths and sizes 2 to 11 % less.  Clusters of gridDim.x / clusters blocks;
// the first w_clusters work on product w, wp blocks a tile, the others on product x, xp blocks a tile.
struct F32Pair {
  F32Prod w, x;
  int32_t wp, xp, w_clusters, w_tiles, x_tiles;
};
template <bool FOLD>
__global__ void __launch_bounds__(F32Cfg<32, 4>::THREADS, 2) gemm_f32_pair_kernel(const __grid_constant__ F32Pair a) {
  if (!chain_begin()) return;
  __shared__ __align__(16) F32Smem<32, 4> sm;
  uint32_t blocks, rank;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(blocks));
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int cluster = blockIdx.x / blocks;
  const bool is_w = cluster < a.w_clusters;
  const int parts = is_w ? a.wp : a.xp, item = (cluster - (is_w ? 0 : a.w_clusters)) * (int)blocks + (int)rank;
  const int tile = item / parts, part = item % parts;
  const F32Prod& p = is_w ? a.w : a.x;
  const int tiles_n = (p.N + 31) / 32;
  const int64_t m0 = (int64_t)(tile / tiles_n) * 32, n0 = (int64_t)(tile % tiles_n) * 32;
  const bool there = tile < (is_w ? a.w_tiles : a.x_tiles);
  if (there && is_w) f32_tile<32, false, false, 4, FOLD, true>(a.w, m0, n0, part, parts, (int)rank - part, sm);
  else if (there) f32_tile<32, true, false, 4, FOLD, false>(a.x, m0, n0, part, parts, (int)rank - part, sm);
  if (blocks > 1 && !(there && parts > 1)) {               // the cluster's barrier counts every block
    gram_cluster_sync();
    gram_cluster_sync();
  }
}

F32Prod f32_prod(const float* A, int64_t lda, const float* B, int64_t ldb, float* C, int64_t ldc, int64_t M, int N, int64_t K,
                 int64_t k_per_part, const EpiDev& e) {
  auto al = [](const void* p) { return (uintptr_t)p % 16 == 0; };
  const int one_aux = (e.res != nullptr) + (e.dgelu_pre != nullptr) + (e.accumulate != 0) <= 1;
  F32Prod p = {};
  p.A = A; p.lda = lda; p.B = B; p.ldb = ldb; p.C = C; p.ldc = ldc; p.M = M; p.N = N; p.K = K;
  p.k_per_part = k_per_part;
  p.vec_a = lda % 4 == 0 && al(A);
  p.vec_b = ldb % 4 == 0 && al(B);
  p.vec_e = one_aux && N % 4 == 0 && ldc % 4 == 0 && al(C) && al(e.bias) && al(e.res) && al(e.res_gamma) && al(e.res_beta) && al(e.pre) &&
            al(e.dgelu_pre) && al(e.copy_out);
  p.e = e;
  return p;
}

template <int TILE, int NG, bool A_K, bool B_K>
cudaError_t launch_f32(const F32Prod& p, int splits, cudaStream_t st) {
  const int64_t blocks = ceil_div64(p.M, TILE) * ceil_div(p.N, TILE) * splits;
  void (*kern)(F32Prod);
  if constexpr (TILE == 64)
    kern = 3 * ceil_div64(blocks, 3 * kNumSMs) < 2 * ceil_div64(blocks, 2 * kNumSMs) ? gemm_f32_wide_kernel<A_K, B_K, 3> : gemm_f32_wide_kernel<A_K, B_K, 2>;
  else
    kern = gemm_f32_kernel<TILE, A_K, B_K, NG>;
  if (splits > 8) {                                        // clusters of more than 8 blocks are an opt-in
    const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (err != cudaSuccess) return err;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ceil_div(p.N, TILE), (unsigned)ceil_div64(p.M, TILE), (unsigned)splits);
  cfg.blockDim = dim3(F32Cfg<TILE, NG>::THREADS);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = (unsigned)splits;
  attr[1] = chain_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p);
}
template <int TILE, int NG>
cudaError_t launch_f32_major(bool a_k, bool b_k, const F32Prod& p, int splits, cudaStream_t st) {
  if (a_k && b_k) return launch_f32<TILE, NG, true, true>(p, splits, st);
  if (a_k) return launch_f32<TILE, NG, true, false>(p, splits, st);
  if (b_k) return launch_f32<TILE, NG, false, true>(p, splits, st);
  return launch_f32<TILE, NG, false, false>(p, splits, st);
}

// How a product of `blocks` tiles (64 x 64 if big, else 32 x 32) is cut: parts of the K range over a cluster, and groups of a
// block.
//  - K of at most four k-blocks: one round of loads by that many groups, no cluster.  160 x 512 over 128: 5.5 us over a cluster, 3.6;
//    320 x 256 over 64 5.4 and 3.9; K = 32 takes four groups too, whose threads share the tile's epilogue (160 x 128: 4.3 and 3.2).
//    Beyond two blocks of four groups an SM (1200 x 288 over 96, 342 tiles: 7.1 us without, 7.8 with) only as many as k-blocks.
//  - Else the K range is halved over a cluster while blocks are missing and a part keeps two k-blocks.  Groups on top where the
//    blocks leave SMs room: 64 x 64 over 4000 (64 blocks) 10.0 and 6.6, 192 x 64 (192 blocks) 10.8 and 8.6, but 256 x 64 over 1200
//    (256 blocks) 7.0 without, 9.8 with.
//    Eight parts with a round of four groups instead of sixteen with two k-blocks (192 x 64 over 912: 5.6 and 4.9).
//  - Tiles that need no parts but are no more than three an SM: four groups shorten a long K (1200 x 256 over 1024, 304 tiles: 46.8
//    and 41.6).
//  - Instead of all that, as few parts as let each take its K in one round of four groups: where the blocks above are more than 2.75
//    an SM, or take more than one round while these are at most one an SM, and these fit at once.  (Clusters of four and more do not
//    reach every SM: 258 blocks of the 296.)  With those parts and with the ones above, us: 160 x 256 over 160 4.7 and 5.4, 480 x 64 over 384
//    4.8 and 5.4, 64 x 512 over 768 6.5 and 7.9, 912 x 64 over 256 5.1 and 5.2, 912 x 128 over 192 6.3 and 7.0.  Everywhere that
//    they fit they would lose: 64 x 64 over 256 4.8 and 3.9 (eight parts of a k-block are one round too), 320 x 128 over 384 6.4 and 5.9,
//    576 x 128 over 512 (288 blocks) 1.4 times the time.
struct F32Plan {
  int parts, groups;
  int64_t k_per_part;
};
F32Plan f32_plan(int64_t blocks, int64_t K, bool big, int most_parts) {
  F32Plan p = {1, 1, K};
  const int sk = big ? F32Cfg<64>::SK : F32Cfg<32>::SK;
  auto groups_of = [&](int64_t k) { return k > 2 * sk || (K <= 4 * sk && blocks <= 2 * kNumSMs) ? 4 : (k > sk ? 2 : 1); };
  const bool one_round = !big && K <= 4 * sk && blocks * groups_of(K) <= 8 * kNumSMs;
  if (!one_round) {
    const int64_t enough = big ? kNumSMs : 4 * kNumSMs;
    while (p.parts < most_parts && blocks * p.parts * 2 <= enough && K >= 64 * p.parts) {
      if (p.parts == 8 && !big && blocks <= 16 && K > 16 * sk && K <= 32 * sk) break;
      p.parts *= 2;
    }
  }
  p.k_per_part = ceil_div64(ceil_div64(K, p.parts), sk) * sk;
  const int groups = groups_of(p.k_per_part);
  const int64_t all = blocks * p.parts;
  if (!big && (one_round || (groups == 4 ? 3 * all <= 4 * kNumSMs : all <= kNumSMs) || (p.parts == 1 && all <= 3 * kNumSMs && K >= 256))) p.groups = groups;
  if (!one_round && !big) {
    int parts = 1;
    while (parts < most_parts && K > 4 * sk * parts) parts *= 2;
    const int sms = parts > 2 ? kNumSMs * 7 / 8 : kNumSMs;
    const bool fits = K <= 4 * sk * parts && blocks * parts <= 2 * sms;
    if (fits && (4 * all > 11 * kNumSMs || (p.k_per_part > sk * p.groups && blocks * parts <= sms)))
      p = {parts, 4, ceil_div64(ceil_div64(K, parts), sk) * sk};
  }
  return p;
}

// ============================================================================================
// bf16 tcgen05 kernel
// ============================================================================================
constexpr int BM = 128, BK = 64;
constexpr int EPI_WARPS = 8;
constexpr int TC_THREADS = 64 + 32 * EPI_WARPS;   // warp 0: TMA, warp 1: MMA, warps 2-9: epilogue
constexpr int STAGE_LD = 32;                     // a warp's 32 x 32 fp32 transpose buffer (swizzled, no padding)
// A warp's 32 x 32 fp32 transpose buffer: rows of eight 16-byte slots, slot j of row r stored at j ^ (r & 7).
// Row-per-thread writes and eight-lanes-per-row reads are then both free of bank conflicts.
__device__ __forceinline__ void stage_write_row(float* stage, int lane, const uint32_t (&v)[32]) {
  float4* s4 = reinterpret_cast<float4*>(stage) + lane * 8;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    s4[j ^ (lane & 7)] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]),
                                     __uint_as_float(v[4 * j + 3]));
}
__device__ __forceinline__ float4 stage_read(const float* stage, int row, int slot) {
  return reinterpret_cast<const float4*>(stage)[row * 8 + (slot ^ (row & 7))];
}

struct TcArgs {
  void* C;
  int64_t ldc;
  int64_t M;
  int32_t N;
  int32_t num_kb;          // k-blocks of 64 over the whole K
  int32_t n_tiles_m, n_tiles_n, splits, kb_per_split;
  int32_t chain;           // k-blocks added up in one accumulator (EPI_SUM: fewer than kb_per_split)
  int32_t half_from;       // pair kernel: tiles from this one on are two work units of half the columns each (unit numbers go on)
  int64_t split_stride;    // elements between the partial outputs of two splits
  EpiDev epi;
  int32_t* status;
};

template <int BN> struct TcCfg {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = (BN == 256) ? 4 : (BN == 128 ? 6 : 8);
  static constexpr int TMEM_COLS = 2 * BN;           // two accumulator buffers
  static constexpr int EPI_BYTES = EPI_WARPS * 32 * STAGE_LD * 4;   // per-warp transpose buffers of the epilogue
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;
};

// The epilogue of one output tile for one epilogue warp: rows row0 .. row0+31 (TMEM lanes q*32..), columns
// [half*BN/PARTS, (half+1)*BN/PARTS) of the tile whose first column is n_first; columns from n_lim on (the matrix's edge, or
// the end of a half-width unit) are not touched.  A warp may read only its quarter of the TMEM lanes; PARTS warps
// share a quarter and split the columns.  Each 32 x 32 block is loaded one row per thread, turned through a
// padded shared-memory buffer, and then handled four rows per instruction with eight lanes per row, so that
// global loads and stores of a row are contiguous 128-byte pieces.  Returns false if the bounded wait for the
// accumulator gave up.
// DG: the epilogue is only "multiply by the saved GELU derivative, store bf16" (backward of the
// feed-forward layer); the derivative's values for the whole tile are then fetched into registers
// while the main loop of that tile is still running, which hides their HBM latency.
// Epilogue variants fixed at compile time (the general one reads the EpiDev flags at run time):
//   EPI_DG    multiply by the saved GELU derivative, bf16 out (values prefetched during the main loop)
//   EPI_BIAS  (+ bias), bf16 or fp32 out
//   EPI_GELU  + bias, GELU, saved derivative, both bf16 (pair kernel)
//   EPI_GELU_V  the same without the derivative (passes that no backward pass follows; pair kernel)
//   EPI_RES   (+ bias) + fp32 residual (LayerNorm on the fly when res_mean is set), fp32 out (+ bf16 copy)
//   EPI_SUM   fp32 out (added to C on request) of a K range that is cut into several accumulator chains (pair kernel)
//   EPI_RES_TS  the same without the bf16 copy, residual in and result out by bulk tensor copies (pair kernel)
enum { EPI_GENERAL = 0, EPI_DG = 1, EPI_BIAS = 2, EPI_GELU = 3, EPI_RES = 4, EPI_RES_TS = 5, EPI_GELU_V = 6, EPI_SUM = 7 };

template <int BN, typename CT, int MODE, int PARTS = 2>
__device__ __forceinline__ bool epilogue_tile(const TcArgs& a, CT* Cs, int64_t row0, int n_first, int n_lim, int half, int q, int lane,
                                              float* stage, uint32_t tmem_base, int buf, uint32_t tfull_addr,
                                              uint32_t parity, volatile int* abort_flag) {
  if constexpr (MODE == EPI_DG) {
    uint2 pf[BN / (32 * PARTS)][8];                       // packed bf16: 4 columns of one row per entry
    const int sub = lane >> 3, slot = lane & 7;
    const int64_t rows_left = a.M - (row0 + sub);
    const int64_t step = 4 * a.ldc;
    const int ncol0 = n_first + half * (BN / PARTS) + slot * 4;
    const int64_t o0 = (row0 + sub) * a.ldc + ncol0;
    const bf16* pre = reinterpret_cast<const bf16*>(a.epi.dgelu_pre) + o0;
#pragma unroll
    for (int blk = 0; blk < BN / (32 * PARTS); ++blk) {
      const bool col_ok = ncol0 + blk * 32 < n_lim;
#pragma unroll
      for (int rr = 0; rr < 8; ++rr)
        pf[blk][rr] = (col_ok && rr * 4 < rows_left) ? *reinterpret_cast<const uint2*>(pre + blk * 32 + rr * step) : make_uint2(0u, 0u);
    }
    if (!mbar_wait(tfull_addr, parity, abort_flag)) return false;
    tc_fence_after();
#pragma unroll
    for (int blk = 0; blk < BN / (32 * PARTS); ++blk) {
      const int c0 = half * (BN / PARTS) + blk * 32;
      uint32_t v[32];
      tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c0), v);
      tc_ld32_wait(v);
      stage_write_row(stage, lane, v);
      __syncwarp();
      if (ncol0 + blk * 32 < n_lim) {
        CT* cp = Cs + o0 + blk * 32;
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
          if (rr * 4 < rows_left) {
            const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pf[blk][rr].x));
            const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pf[blk][rr].y));
            const float4 t = stage_read(stage, rr * 4 + sub, slot);
            const float x[4] = {t.x * g0.x, t.y * g0.y, t.z * g1.x, t.w * g1.y};
            st4(cp, x);
          }
          cp += step;
        }
      }
      __syncwarp();
    }
    tc_fence_before();
    return true;
  } else if constexpr (MODE == EPI_RES) {
    // fp32 result = accumulator (+ bias) + residual (LayerNorm applied where it is read), plus an optional bf16 copy.
    // The residual is 4 bytes per element from HBM, and eight warps per SM keep too few loads in flight to hide its
    // latency if every 32-column block waits for its own: the loads of a block are therefore issued one block ahead,
    // the first block's before the wait for the accumulator.
    constexpr int NBLK = BN / PARTS / 32;
    const int sub = lane >> 3, slot = lane & 7;
    const int64_t rows_left = a.M - (row0 + sub);         // row rr*4 + sub exists iff rr*4 < rows_left
    const int64_t step = 4 * a.ldc;
    const int nbase = n_first + half * (BN / PARTS) + slot * 4;
    const int64_t obase = (row0 + sub) * a.ldc + nbase;
    float4 rnext[8];
    auto load_res = [&](int blk, float4 (&dst)[8]) {
      const bool col_ok = nbase + blk * 32 < n_lim;
      const float* rp = a.epi.res + obase + blk * 32;
#pragma unroll
      for (int rr = 0; rr < 8; ++rr)
        dst[rr] = (col_ok && rr * 4 < rows_left) ? __ldcs(reinterpret_cast<const float4*>(rp + rr * step)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    load_res(0, rnext);
    float mu_l = 0.f, rs_l = 1.f;
    const bool ln = a.epi.res_mean != nullptr;
    if (ln && row0 + lane < a.M) {
      mu_l = a.epi.res_mean[row0 + lane];
      rs_l = a.epi.res_rstd[row0 + lane];
    }
    if (!mbar_wait(tfull_addr, parity, abort_flag)) return false;
    tc_fence_after();
#pragma unroll 1
    for (int blk = 0; blk < NBLK; ++blk) {
      float4 r4[8];
#pragma unroll
      for (int rr = 0; rr < 8; ++rr) r4[rr] = rnext[rr];
      if (blk + 1 < NBLK) load_res(blk + 1, rnext);
      uint32_t v[32];
      tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + half * (BN / PARTS) + blk * 32), v);
      tc_ld32_wait(v);
      stage_write_row(stage, lane, v);
      __syncwarp();
      const int n = nbase + blk * 32;
      const bool col_ok = n < n_lim;                          // lanes of a warp may differ here when N is not a multiple of 32
      float b4[4] = {0.f, 0.f, 0.f, 0.f}, g4[4] = {0.f, 0.f, 0.f, 0.f}, be4[4] = {0.f, 0.f, 0.f, 0.f};
      if (col_ok) {
        if (a.epi.bias) ld4(a.epi.bias + n, b4);
        if (ln) {
          ld4(a.epi.res_gamma + n, g4);
          ld4(a.epi.res_beta + n, be4);
        }
      }
      CT* cp = Cs + obase + blk * 32;
      bf16* qp = a.epi.copy_out ? reinterpret_cast<bf16*>(a.epi.copy_out) + obase + blk * 32 : nullptr;
#pragma unroll
      for (int rr = 0; rr < 8; ++rr) {
        const int rl = rr * 4 + sub;
        // every lane takes part in the shuffles, whatever its columns
        const float mu = __shfl_sync(0xffffffffu, mu_l, rl), rs = __shfl_sync(0xffffffffu, rs_l, rl);
        if (col_ok && rr * 4 < rows_left) {
          const float4 t = stage_read(stage, rl, slot);
          float x[4] = {t.x + b4[0], t.y + b4[1], t.z + b4[2], t.w + b4[3]};
          if (ln) {
            x[0] += (r4[rr].x - mu) * rs * g4[0] + be4[0];
            x[1] += (r4[rr].y - mu) * rs * g4[1] + be4[1];
            x[2] += (r4[rr].z - mu) * rs * g4[2] + be4[2];
            x[3] += (r4[rr].w - mu) * rs * g4[3] + be4[3];
          } else {
            x[0] += r4[rr].x; x[1] += r4[rr].y; x[2] += r4[rr].z; x[3] += r4[rr].w;
          }
          st4(cp, x);
          if (qp) st4(qp, x);
        }
        cp += step;
        if (qp) qp += step;
      }
      __syncwarp();
    }
    tc_fence_before();
    return true;
  } else if constexpr (MODE == EPI_BIAS) {
    if (!mbar_wait(tfull_addr, parity, abort_flag)) return false;
    tc_fence_after();
    const int sub = lane >> 3, slot = lane & 7;
    const int64_t rows_left = a.M - (row0 + sub);         // row rr*4 + sub exists iff rr*4 < rows_left
#pragma unroll 1
    for (int c0 = half * (BN / PARTS); c0 < (half + 1) * (BN / PARTS); c0 += 32) {
      uint32_t v[32];
      tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c0), v);
      tc_ld32_wait(v);
      stage_write_row(stage, lane, v);
      __syncwarp();
      const int n = n_first + c0 + slot * 4;
      if (n < n_lim) {                                      // N is a multiple of 8
        float b4[4] = {0.f, 0.f, 0.f, 0.f};
        if (a.epi.bias) ld4(a.epi.bias + n, b4);
        const int64_t o0 = (row0 + sub) * a.ldc + n;      // element offset of this lane's first row
        const int64_t step = 4 * a.ldc;
        CT* cp = Cs + o0;
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
          if (rr * 4 < rows_left) {
            const float4 t = stage_read(stage, rr * 4 + sub, slot);
            const float x[4] = {t.x + b4[0], t.y + b4[1], t.z + b4[2], t.w + b4[3]};
            st4(cp, x);
          }
          cp += step;
        }
      }
      __syncwarp();
    }
    tc_fence_before();
    return true;
  } else {
    if (!mbar_wait(tfull_addr, parity, abort_flag)) return false;
    tc_fence_after();
    float mu_l = 0.f, rs_l = 1.f;               // LayerNorm statistics of row row0 + lane
    if (a.epi.res_mean && row0 + lane < a.M) {
      mu_l = a.epi.res_mean[row0 + lane];
      rs_l = a.epi.res_rstd[row0 + lane];
    }
#pragma unroll 1
    for (int c0 = half * (BN / PARTS); c0 < (half + 1) * (BN / PARTS); c0 += 32) {
      uint32_t v[32];
      tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c0), v);
      tc_ld32_wait(v);
      stage_write_row(stage, lane, v);
      __syncwarp();
      const int n = n_first + c0 + (lane & 7) * 4;
      const bool col_ok = n < n_lim;                // N is a multiple of 8
      float bias4[4] = {0.f, 0.f, 0.f, 0.f}, gam4[4] = {0.f, 0.f, 0.f, 0.f}, bet4[4] = {0.f, 0.f, 0.f, 0.f};
      if (col_ok) {
        if (a.epi.bias) ld4(a.epi.bias + n, bias4);
        if (a.epi.res_mean) {
          ld4(a.epi.res_gamma + n, gam4);
          ld4(a.epi.res_beta + n, bet4);
        }
      }
      // global loads of four rows are issued before the first store of those rows
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        EpiLoads L[4];
#pragma unroll
        for (int r4 = 0; r4 < 4; ++r4) {
          const int64_t m = row0 + (hh * 4 + r4) * 4 + (lane >> 3);
          if (m < a.M && col_ok) epilogue_load4<CT>(a.epi, Cs, a.ldc, m, n, L[r4]);
        }
#pragma unroll
        for (int r4 = 0; r4 < 4; ++r4) {
          const int rl = (hh * 4 + r4) * 4 + (lane >> 3);
          const float mu = __shfl_sync(0xffffffffu, mu_l, rl), rs = __shfl_sync(0xffffffffu, rs_l, rl);
          const int64_t m = row0 + rl;
          if (m < a.M && col_ok) {
            const float4 t = stage_read(stage, rl, lane & 7);
            float x[4] = {t.x, t.y, t.z, t.w};
            epilogue_store4<CT>(a.epi, Cs, a.ldc, m, n, x, L[r4], bias4, gam4, bet4, mu, rs);
          }
        }
      }
      __syncwarp();
    }
    tc_fence_before();
    return true;
  }
}

template <int BN, bool A_K, bool B_K, typename CT, int MODE = EPI_GENERAL>
__global__ void __launch_bounds__(TC_THREADS, 1) gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA,
                                                               const __grid_constant__ CUtensorMap tmB, TcArgs a) {
  using Cfg = TcCfg<BN>;
  constexpr int STAGES = Cfg::STAGES;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;                 // swizzled tiles need 1024-byte alignment
  uint8_t* gen_tiles = smem_raw + (tiles - raw);
  float* epi_stage = reinterpret_cast<float*>(gen_tiles + STAGES * Cfg::STAGE_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gen_tiles + STAGES * Cfg::STAGE_BYTES + Cfg::EPI_BYTES);
  const uint32_t bar0 = tiles + STAGES * Cfg::STAGE_BYTES + Cfg::EPI_BYTES;
  // barrier slots: full[STAGES], empty[STAGES], tmem_full[2], tmem_empty[2]; then tmem base, abort flag
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull_bar(b), 1);
      mbar_init(tempty_bar(b), 32 * EPI_WARPS);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)Cfg::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (!chain_begin()) return;              // barriers and tensor memory are set up before the wait

  const int64_t total = (int64_t)a.n_tiles_m * a.n_tiles_n * a.splits;
  bool failed = false;

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    int s = 0;
    uint32_t ph = 0;
    for (int64_t t = blockIdx.x; t < total && !failed; t += gridDim.x) {
      const int split = (int)(t / ((int64_t)a.n_tiles_m * a.n_tiles_n));
      const int64_t r = t - (int64_t)split * a.n_tiles_m * a.n_tiles_n;
      const int tm = (int)(r / a.n_tiles_n), tn = (int)(r % a.n_tiles_n);
      const int kb0 = split * a.kb_per_split, kb1 = min(kb0 + a.kb_per_split, a.num_kb);
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait_warp(empty_bar(s), ph ^ 1u, abort_flag)) { failed = true; break; }
        const uint32_t sa = tiles + s * Cfg::STAGE_BYTES, sb = sa + Cfg::A_BYTES;
        if (elect_one()) {
          mbar_expect_tx(full_bar(s), Cfg::STAGE_BYTES);
          if (A_K) {
            tma_load_2d(sa, &tmA, kb * BK, tm * BM, full_bar(s));
          } else {
#pragma unroll
            for (int i = 0; i < BM / 64; ++i) tma_load_2d(sa + i * 8192, &tmA, tm * BM + i * 64, kb * BK, full_bar(s));
          }
          if (B_K) {
            tma_load_2d(sb, &tmB, kb * BK, tn * BN, full_bar(s));
          } else {
#pragma unroll
            for (int i = 0; i < BN / 64; ++i) tma_load_2d(sb + i * 8192, &tmB, tn * BN + i * 64, kb * BK, full_bar(s));
          }
        }
        __syncwarp();
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
    }
    if (failed && lane == 0) {
      *abort_flag = 1;
      gram_device_fail(a.status, GRAM_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer --------------------------------
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((A_K ? 0u : 1u) << 15) |
                               ((B_K ? 0u : 1u) << 16) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    int s = 0;
    uint32_t ph = 0;
    int64_t it = 0;
    for (int64_t t = blockIdx.x; t < total && !failed; t += gridDim.x, ++it) {
      const int split = (int)(t / ((int64_t)a.n_tiles_m * a.n_tiles_n));
      const int kb0 = split * a.kb_per_split, kb1 = min(kb0 + a.kb_per_split, a.num_kb);
      const int buf = (int)(it & 1);
      if (!mbar_wait_warp(tempty_bar(buf), (uint32_t)((it >> 1) & 1) ^ 1u, abort_flag)) { failed = true; break; }
      tc_fence_after();
      const uint32_t tmem_d = tmem_base + (uint32_t)(buf * BN);
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait_warp(full_bar(s), ph, abort_flag)) { failed = true; break; }
        tc_fence_after();
        const uint32_t sa = tiles + s * Cfg::STAGE_BYTES, sb = sa + Cfg::A_BYTES;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t da = A_K ? make_desc(sa + k * 32, 16, 1024) : make_desc(sa + k * 2048, 8192, 1024);
            const uint64_t db = B_K ? make_desc(sb + k * 32, 16, 1024) : make_desc(sb + k * 2048, 8192, 1024);
            tc_mma(tmem_d, da, db, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
          }
          tc_commit(empty_bar(s));            // the stage is free once these MMAs have read it
          if (kb == kb1 - 1) tc_commit(tfull_bar(buf));      // accumulator complete
        }
        __syncwarp();
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
    }
    if (failed && lane == 0) {
      *abort_flag = 1;
      gram_device_fail(a.status, GRAM_ERR_TIMEOUT);
    }
  } else {
    // ------------------------------ epilogue warps ----------------------------
    const int ew = warp - 2;
    const int q = warp & 3;
    const int half = ew >> 2;
    float* stage = epi_stage + ew * (32 * STAGE_LD);
    CT* C = reinterpret_cast<CT*>(a.C);
    int64_t it = 0;
    for (int64_t t = blockIdx.x; t < total && !failed; t += gridDim.x, ++it) {
      const int split = (int)(t / ((int64_t)a.n_tiles_m * a.n_tiles_n));
      const int64_t r = t - (int64_t)split * a.n_tiles_m * a.n_tiles_n;
      const int tm = (int)(r / a.n_tiles_n), tn = (int)(r % a.n_tiles_n);
      const int buf = (int)(it & 1);
      const int64_t row0 = (int64_t)tm * BM + q * 32;
      CT* Cs = C + (int64_t)split * a.split_stride;
      if (!epilogue_tile<BN, CT, MODE>(a, Cs, row0, tn * BN, a.N, half, q, lane, stage, tmem_base, buf, tfull_bar(buf),
                                     (uint32_t)((it >> 1) & 1), abort_flag)) {
        failed = true;
        break;
      }
      mbar_arrive(tempty_bar(buf));           // all epilogue threads free the accumulator buffer
    }
    if (failed && lane == 0) {
      *abort_flag = 1;
      gram_device_fail(a.status, GRAM_ERR_TIMEOUT);
    }
  }

  // ------------------------------ teardown --------------------------------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // a wait gave up: let copies and MMAs already issued drain (bounded) before memory is released
    if (warp == 0 && lane == 0) {
      for (int s = 0; s < STAGES; ++s) {
        uint64_t t0 = clock64();
        while (!mbar_try(full_bar(s), 0) && !mbar_try(full_bar(s), 1) && clock64() - t0 < WAIT_LIMIT_CYCLES / 64) {}
      }
    }
    if (warp == 1 && lane == 0) {
      uint64_t t0 = clock64();
      while (clock64() - t0 < WAIT_LIMIT_CYCLES / 64) {}
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS)
                 : "memory");
  }
}

// ============================================================================================
// The same product on pairs of SMs (tcgen05 cta_group::2): a cluster of two CTAs owns a 256 x 256
// output tile.  Each CTA stages its own 128 rows of A and its own 128 of the tile's 256 columns of B,
// the leader CTA (cluster rank 0) issues one M256 N256 K16 MMA per step that reads both CTAs' shared
// memory, and each CTA's tensor memory receives its 128 rows of the result.  Per CTA and k-block this
// moves 32 KB through shared memory instead of 48 KB, which is what bounds the single-CTA kernel.
// Protocol: each CTA's TMA loads signal the leader's "full" barrier (two arrivals with their byte
// counts); the leader's commits arrive on the "empty" and "accumulator full" barriers of both CTAs
// (one commit for the two); the epilogue warps of both CTAs arrive on the leader's
// "accumulator empty" barrier.  Every wait is bounded as in the single-CTA kernel; the CTAs meet at a
// cluster barrier before they exit so that neither releases shared or tensor memory the other may
// still touch.
// ============================================================================================
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_expect_tx_remote(uint32_t cluster_bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int32_t c0, int32_t c1,
                                                 uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1)
      : "memory");
}
// arrives on the barrier at this shared-memory offset in both CTAs of the pair
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accum)
      : "memory");
}

// 32 columns of a per-column vector from column n (zeros at and past N, or without a vector).  The tests are made once per
// block of columns, so that the arithmetic on it is one straight line: with a test per four columns a warp had two pairs of
// values to interleave and waited for their chains.
__device__ __forceinline__ void load_cols32(const float* __restrict__ p, int n, int N, float4 (&x)[8]) {
  if (p && n + 32 <= N) {
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = __ldg(reinterpret_cast<const float4*>(p + n + 4 * j));
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      x[j] = p && n + 4 * j < N ? __ldg(reinterpret_cast<const float4*>(p + n + 4 * j)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Epilogue of the pair kernel for bf16 results (EPI_BIAS, EPI_GELU, EPI_DG): one warp owns rows row0 .. row0+31
// and NB blocks of 32 columns from global column col0 (tile column c_local).  A thread keeps its own row: 32
// accumulators from tensor memory per block, the arithmetic, 64 bytes of bf16 written into a 32-row x 64-column
// box in shared memory (128-byte rows whose 16-byte pieces are XOR-swizzled as the 128-byte swizzle of the
// tensor map expects, which also keeps the writes free of bank conflicts).  Two blocks fill a box, and lane 0
// hands it to a bulk tensor store, which writes whole 128-byte lines and clips the box at the matrix edges.
// EPI_GELU fills a second box with the derivative (the two results are what bounds it: 805 MB in 257 us at 65 536 x 3072, of
// which 255 us stay without the arithmetic and 177 without the stores; one result alone, EPI_GELU_V, takes 239 us where the
// two take 282 at 70 000 rows); EPI_DG (NB = 2) first fetches the box of the saved derivative
// with a bulk tensor load (issued before the wait for the accumulator), multiplies in place and stores the same
// box.  The accumulator buffer is handed back as soon as the last block has been read.  sbuf: 4 KB (8 KB for
// EPI_GELU), 1024-byte aligned, private to the warp.  Returns false if a bounded wait gave up.
template <int MODE, int NB>
__device__ __forceinline__ bool epilogue_tile_ts(const TcArgs& a, const CUtensorMap* tmC, const CUtensorMap* tmP, int32_t row0,
                                                 int32_t col0, int32_t n_lim, int c_local, int q, int lane, uint32_t sbuf,
                                                 uint32_t tmem_base, int buf, uint32_t tfull_addr, uint32_t parity,
                                                 volatile int* abort_flag, uint32_t tempty_remote, uint32_t ld_bar,
                                                 uint32_t ld_parity) {
  static_assert(MODE != EPI_DG || NB == 2, "the derivative's box is fetched once per tile");
  const uint32_t swz = (uint32_t)(lane & 7);
  const uint32_t srow = sbuf + (uint32_t)lane * 128u;
  if constexpr (MODE == EPI_DG) {
    if (lane == 0) {
      bulk_wait_read_all();                                // the last tile's store has read the box
      mbar_expect_tx(ld_bar, 4096);
      tma_load_2d(sbuf, tmP, col0, row0, ld_bar);
    }
    __syncwarp();
  }
  if (!mbar_wait(tfull_addr, parity, abort_flag)) return false;
  tc_fence_after();
  if constexpr (MODE == EPI_DG) {
    if (!mbar_wait(ld_bar, ld_parity, abort_flag)) return false;
  }
  const bool rows_ok = row0 < a.M;                         // a box that starts below the matrix is not stored
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    uint32_t v[32];
    tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + c_local + b * 32), v);
    float4 bias[MODE == EPI_DG ? 1 : 8];
    if constexpr (MODE != EPI_DG) load_cols32(a.epi.bias, col0 + b * 32, a.N, bias);
    tc_ld32_wait(v);
    if (b == NB - 1) {                                     // every value of this tile is in registers now
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(tempty_remote);
    }
    const int nbx = col0 + (b >> 1) * 64;                  // first column of the box
    if (nbx >= n_lim || !rows_ok) continue;
    const uint32_t p0 = (uint32_t)(b & 1) * 4u;            // this block's first 16-byte piece of the row
    uint32_t oc[16];
    if constexpr (MODE == EPI_DG) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint4 g4 = lds128(srow + (((p0 + (uint32_t)c) ^ swz) << 4));
        const uint32_t gw[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 gg = unpack_bf16x2(gw[i]);
          oc[4 * c + i] = pack_bf16x2(__uint_as_float(v[8 * c + 2 * i]) * gg.x, __uint_as_float(v[8 * c + 2 * i + 1]) * gg.y);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        sts128(srow + (((p0 + (uint32_t)c) ^ swz) << 4), oc[4 * c], oc[4 * c + 1], oc[4 * c + 2], oc[4 * c + 3]);
    } else {
      constexpr bool GELU = MODE == EPI_GELU || MODE == EPI_GELU_V, DERIVATIVE = MODE == EPI_GELU;
      uint32_t op[DERIVATIVE ? 16 : 1];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 b4 = bias[j];
        if constexpr (GELU) {
          uint64_t g0, g1, d0, d1;
          gelu_pair<DERIVATIVE>(f2_add(f2_pack(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1])), f2_pack(b4.x, b4.y)), g0, d0);
          gelu_pair<DERIVATIVE>(f2_add(f2_pack(__uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])), f2_pack(b4.z, b4.w)), g1, d1);
          oc[2 * j] = f2_to_bf16x2(g0);
          oc[2 * j + 1] = f2_to_bf16x2(g1);
          if constexpr (DERIVATIVE) {
            op[2 * j] = f2_to_bf16x2(d0);
            op[2 * j + 1] = f2_to_bf16x2(d1);
          }
        } else {
          oc[2 * j] = pack_bf16x2(__uint_as_float(v[4 * j]) + b4.x, __uint_as_float(v[4 * j + 1]) + b4.y);
          oc[2 * j + 1] = pack_bf16x2(__uint_as_float(v[4 * j + 2]) + b4.z, __uint_as_float(v[4 * j + 3]) + b4.w);
        }
      }
      if ((b & 1) == 0) {                                  // the last store from the box(es) has read them
        if (lane == 0) bulk_wait_read_all();
        __syncwarp();
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        sts128(srow + (((p0 + (uint32_t)c) ^ swz) << 4), oc[4 * c], oc[4 * c + 1], oc[4 * c + 2], oc[4 * c + 3]);
      if constexpr (MODE == EPI_GELU) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          sts128(srow + 4096u + (((p0 + (uint32_t)c) ^ swz) << 4), op[4 * c], op[4 * c + 1], op[4 * c + 2], op[4 * c + 3]);
      }
    }
    if (b & 1) {
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store_2d(tmC, sbuf, nbx, row0);
        if constexpr (MODE == EPI_GELU) tma_store_2d(tmP, sbuf + 4096, nbx, row0);
        bulk_commit();
      }
      if constexpr (MODE == EPI_DG) {
        if (a.epi.colsum_part) {
          // column sums of the box as stored (rows and columns outside the matrix hold zeros): lane c adds
          // columns 2c, 2c+1 over the 32 rows in ascending order and writes row (row0 / 32) of the partial sums
          float s0 = 0.f, s1 = 0.f;
          const uint32_t piece = (uint32_t)(lane >> 2), word = (uint32_t)(lane & 3) * 4u;
#pragma unroll 8
          for (uint32_t r = 0; r < 32; ++r) {
            uint32_t w;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(sbuf + r * 128u + ((piece ^ (r & 7u)) << 4) + word) : "memory");
            const float2 f = unpack_bf16x2(w);
            s0 += f.x;
            s1 += f.y;
          }
          const int cc = nbx + 2 * lane;
          if (cc < n_lim) *reinterpret_cast<float2*>(a.epi.colsum_part + (int64_t)(row0 >> 5) * a.N + cc) = make_float2(s0, s1);
          __syncwarp();                                    // every lane has read the box before it is refilled
        }
      }
    }
  }
  return true;
}

// Epilogue of the pair kernel for the fp32 residual products (EPI_RES_TS): result = accumulator (+ bias) + residual,
// the residual being the fp32 stream or LayerNorm of it applied where it is read.  One warp owns rows row0 .. row0+31
// and four blocks of 32 columns from global column col0.  The residual is 4 bytes per element from HBM and the result
// 4 bytes back: both travel as 32-row x 32-column boxes (128-byte rows, 128-byte swizzle) by bulk tensor copies, so the
// warp issues no global load or store of its own and many boxes are in flight per SM.  A thread keeps its own row: 32
// accumulators from tensor memory, its row of the residual box from shared memory, the sum written back in place,
// and lane 0 hands the box to a bulk tensor store.  Three boxes per warp rotate (block k of the warp's running count
// uses box k % 3 and load barrier k % 3): the loads of a tile's first two blocks are issued before the wait for the
// accumulator, that of block b + 2 after the store of block b has been committed and the store before it has read its box.
// sbuf: 12 KB, 1024-byte aligned, private to the warp; nb: the warp's running block count.
__device__ __forceinline__ bool epilogue_tile_res(const TcArgs& a, const CUtensorMap* tmC, const CUtensorMap* tmR, int32_t row0,
                                                  int32_t col0, int32_t n_lim, int c_local, int q, int lane, uint32_t sbuf, uint32_t tmem_base,
                                                  int buf, uint32_t tfull_addr, uint32_t parity, volatile int* abort_flag,
                                                  uint32_t tempty_remote, uint32_t ld_bar0, uint32_t& nb) {
  int nv = 0;                                               // blocks of this warp that lie inside the matrix
  if (row0 < a.M) {
    nv = (n_lim - col0 + 31) / 32;
    nv = nv < 0 ? 0 : (nv > 4 ? 4 : nv);
  }
  auto request = [&](int b) {                               // residual box of block b of this tile -> box (nb + b) % 3
    const uint32_t k = nb + (uint32_t)b;
    const uint32_t bar = ld_bar0 + 8u * (k % 3u);
    mbar_expect_tx(bar, 4096);
    tma_load_2d(sbuf + (k % 3u) * 4096u, tmR, col0 + 32 * b, row0, bar);
  };
  if (lane == 0 && nv > 0) {
    bulk_wait_read_but_one();                               // every store but the latest has read its box
    request(0);
    if (nv > 1) request(1);
  }
  const bool ln = a.epi.res_mean != nullptr;
  float mu = 0.f, rs = 1.f;
  if (ln && row0 + lane < a.M) {
    mu = a.epi.res_mean[row0 + lane];
    rs = a.epi.res_rstd[row0 + lane];
  }
  if (!mbar_wait(tfull_addr, parity, abort_flag)) return false;
  tc_fence_after();
  if (nv == 0) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_remote(tempty_remote);
    return true;
  }
  const uint32_t swz = (uint32_t)(lane & 7);
#pragma unroll 1
  for (int b = 0; b < nv; ++b) {
    const uint32_t k = nb + (uint32_t)b;
    const uint32_t box = sbuf + (k % 3u) * 4096u, srow = box + (uint32_t)lane * 128u;
    const int n = col0 + b * 32;
    uint32_t v[32];
    tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + c_local + b * 32), v);
    float4 bias[8], gam[8], bet[8];
    load_cols32(a.epi.bias, n, a.N, bias);
    if (ln) {
      load_cols32(a.epi.res_gamma, n, a.N, gam);
      load_cols32(a.epi.res_beta, n, a.N, bet);
    }
    tc_ld32_wait(v);
    if (b == nv - 1) {                                      // every value of this tile is in registers now
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(tempty_remote);
    }
    if (!mbar_wait(ld_bar0 + 8u * (k % 3u), (k / 3u) & 1u, abort_flag)) return false;
    if (ln) {                                               // columns past N: zeros in, and the store clips them
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint32_t addr = srow + ((((uint32_t)c) ^ swz) << 4);
        const uint4 r = lds128(addr);
        sts128(addr, __float_as_uint(__uint_as_float(v[4 * c]) + bias[c].x + ((__uint_as_float(r.x) - mu) * rs * gam[c].x + bet[c].x)),
               __float_as_uint(__uint_as_float(v[4 * c + 1]) + bias[c].y + ((__uint_as_float(r.y) - mu) * rs * gam[c].y + bet[c].y)),
               __float_as_uint(__uint_as_float(v[4 * c + 2]) + bias[c].z + ((__uint_as_float(r.z) - mu) * rs * gam[c].z + bet[c].z)),
               __float_as_uint(__uint_as_float(v[4 * c + 3]) + bias[c].w + ((__uint_as_float(r.w) - mu) * rs * gam[c].w + bet[c].w)));
      }
    } else {
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint32_t addr = srow + ((((uint32_t)c) ^ swz) << 4);
        const uint4 r = lds128(addr);
        sts128(addr, __float_as_uint(__uint_as_float(v[4 * c]) + bias[c].x + __uint_as_float(r.x)),
               __float_as_uint(__uint_as_float(v[4 * c + 1]) + bias[c].y + __uint_as_float(r.y)),
               __float_as_uint(__uint_as_float(v[4 * c + 2]) + bias[c].z + __uint_as_float(r.z)),
               __float_as_uint(__uint_as_float(v[4 * c + 3]) + bias[c].w + __uint_as_float(r.w)));
      }
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_2d(tmC, box, n, row0);
      bulk_commit();
      if (b + 2 < nv) {
        bulk_wait_read_but_one();                           // the store of block b - 1 has read the box that block b + 2 takes
        request(b + 2);
      }
    }
    __syncwarp();
  }
  nb += (uint32_t)nv;
  return true;
}

// EW epilogue warps per CTA: 8 (two per TMEM lane quarter) or, for the light epilogues whose register use allows
// it, 16 (four per quarter, 64 columns each) with one pipeline stage fewer
// bytes of private shared memory per epilogue warp: one 4 KB store box, two for the GELU epilogue (value and derivative),
// three fp32 boxes for the residual epilogue
template <typename CT, int MODE> constexpr int warp_bytes() {
  return (sizeof(CT) == 4 && MODE == EPI_RES_TS) ? 12288 : ((sizeof(CT) == 2 && MODE == EPI_GELU) ? 8192 : 4096);
}
template <int EW, int WARP_BYTES = 4096> struct Tc2Cfg {
  static constexpr int BN = 256;                       // columns of the pair's tile
  static constexpr int A_BYTES = BM * BK * 2;          // this CTA's 128 rows of A
  static constexpr int B_BYTES = (BN / 2) * BK * 2;    // this CTA's 128 columns of B
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int EPI_BYTES = EW * WARP_BYTES;    // the epilogue warps' private buffers
  static constexpr int STAGES = (232448 - 1024 - 512 - EPI_BYTES) / STAGE_BYTES;   // 6 with 32 KB of buffers, 5 with 64 KB
  static constexpr int TMEM_COLS = 2 * BN;
  static constexpr int THREADS = 64 + 32 * EW;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + 1024 + 512;
};

// A work unit of the pair kernel: a tile, or half of its columns, over the k-blocks [kb0, kb1).  The last wave of tiles is
// seldom full: where its tiles fit one wave as halves they are handed out as such (300 tiles over 74 pairs are 4 waves and
// 4 tiles; the rest of the chip would wait for those).  25 600 x 768 x 3072 with the LayerNorm residual: 102 -> 94 us.
struct Tc2Unit {
  int32_t split, tm, n_first, width, kb0, kb1;
};
__device__ __forceinline__ Tc2Unit tc2_unit(const TcArgs& a, int64_t t) {
  Tc2Unit u;
  const int64_t per_split = (int64_t)a.n_tiles_m * a.n_tiles_n;
  int32_t right = 0;
  u.width = 256;
  if (t >= a.half_from) {                              // one part of the K range only
    right = (int32_t)((t - a.half_from) & 1);
    t = a.half_from + ((t - a.half_from) >> 1);
    u.width = 128;
  }
  u.split = (int32_t)(t / per_split);
  const int64_t r = t - (int64_t)u.split * per_split;
  u.tm = (int32_t)(r / a.n_tiles_n);
  u.n_first = (int32_t)(r % a.n_tiles_n) * 256 + right * 128;
  u.kb0 = u.split * a.kb_per_split;
  u.kb1 = min(u.kb0 + a.kb_per_split, a.num_kb);
  return u;
}
__device__ __forceinline__ int64_t tc2_units(const TcArgs& a) {
  const int64_t tiles = (int64_t)a.n_tiles_m * a.n_tiles_n * a.splits;
  return tiles + (tiles > a.half_from ? tiles - a.half_from : 0);
}

// Epilogue of EPI_SUM: the unit's K range arrives as several accumulators, each a chain of a.chain k-blocks, which the warp
// adds up in its registers (128 columns a thread) in ascending order before it writes its 32 rows x 128 columns.  The tensor
// core cuts off where this adds with rounding, so the length of a chain sets the precision; with the chains of one unit added
// here, the parts of the K range that go through memory need no longer be as many as the chains.  A unit of one chain is handed
// back to the MMAs sooner this way, but its first column is written later: from SUM_CHAIN_ALONE k-blocks on the former counts more,
// below it the unit takes the epilogue that writes a block of columns as it comes out of the accumulator (2304 x 768 in eight parts,
// us so / through these registers: chains of 8 k-blocks 26.3 / 29.4, of 16 36.1 / 36.1, of 32 57.5 / 56.3, of 128 179 / 173).
constexpr int SUM_CHAIN_ALONE = 16;
constexpr int SUM_CHAIN_MAX = 192;       // k-blocks of a chain, whatever the tiles and the workspace: 65 536 rows in six
__device__ __forceinline__ bool epilogue_unit_sum(const TcArgs& a, float* Cs, int64_t row0, int n_first, int n_lim, int half, int q, int lane,
                                                  float* stage, uint32_t tmem_base, int64_t it, int chains, uint32_t tfull0,
                                                  uint32_t tempty0_remote, volatile int* abort_flag) {
  float acc[4][32];
#pragma unroll
  for (int b = 0; b < 4; ++b)
#pragma unroll
    for (int k = 0; k < 32; ++k) acc[b][k] = 0.f;
#pragma unroll 1
  for (int c = 0; c < chains; ++c, ++it) {
    const uint32_t buf = (uint32_t)(it & 1);
    if (!mbar_wait(tfull0 + 8u * buf, (uint32_t)((it >> 1) & 1), abort_flag)) return false;
    tc_fence_after();
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      uint32_t v[32];
      tc_ld32_issue(tmem_base + ((uint32_t)(q * 32) << 16) + buf * 256u + (uint32_t)(half * 128 + b * 32), v);
      tc_ld32_wait(v);
#pragma unroll
      for (int k = 0; k < 32; ++k) acc[b][k] += __uint_as_float(v[k]);
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_remote(tempty0_remote + 8u * buf);
  }
  const int sub = lane >> 3, slot = lane & 7;
  const int64_t rows_left = a.M - (row0 + sub);
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    uint32_t v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __float_as_uint(acc[b][k]);
    stage_write_row(stage, lane, v);
    __syncwarp();
    const int n = n_first + half * 128 + b * 32 + slot * 4;
    if (n < n_lim) {                                   // N is a multiple of 8
      float* cp = Cs + (row0 + sub) * a.ldc + n;
#pragma unroll
      for (int rr = 0; rr < 8; ++rr) {
        if (rr * 4 < rows_left) {
          const float4 t = stage_read(stage, rr * 4 + sub, slot);
          float x[4] = {t.x, t.y, t.z, t.w}, o[4] = {0.f, 0.f, 0.f, 0.f};
          if (a.epi.accumulate) ld4(cp, o);
#pragma unroll
          for (int k = 0; k < 4; ++k) x[k] += o[k];
          st4(cp, x);
        }
        cp += 4 * a.ldc;
      }
    }
    __syncwarp();
  }
  return true;
}

// n_tiles_m counts 256-row tiles here.  tmC / tmP: maps of the bf16 result and of the GELU-derivative matrix
// (boxes of 32 rows x 64 columns, 128-byte swizzle) for the variants whose epilogue uses bulk tensor stores; unused otherwise.
template <bool A_K, bool B_K, typename CT, int MODE = EPI_GENERAL, int EW = EPI_WARPS>
__global__ void __launch_bounds__(64 + 32 * EW, 1) gemm_tc2_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                  const __grid_constant__ CUtensorMap tmB,
                                                                  const __grid_constant__ CUtensorMap tmC,
                                                                  const __grid_constant__ CUtensorMap tmP, TcArgs a) {
  constexpr bool RS = sizeof(CT) == 4 && MODE == EPI_RES_TS;       // fp32 residual epilogue through bulk tensor copies
  constexpr bool TS = RS || (sizeof(CT) == 2 && ((EW == 16 && MODE == EPI_DG) || MODE == EPI_BIAS || MODE == EPI_GELU || MODE == EPI_GELU_V));
  constexpr int WARP_BYTES = warp_bytes<CT, MODE>();
  using Cfg = Tc2Cfg<EW, WARP_BYTES>;
  constexpr int BN = Cfg::BN, STAGES = Cfg::STAGES;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;       // the same offset in both CTAs of the pair
  uint8_t* gen_tiles = smem_raw + (tiles - raw);
  float* epi_stage = reinterpret_cast<float*>(gen_tiles + STAGES * Cfg::STAGE_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gen_tiles + STAGES * Cfg::STAGE_BYTES + Cfg::EPI_BYTES);
  const uint32_t bar0 = tiles + STAGES * Cfg::STAGE_BYTES + Cfg::EPI_BYTES;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };                       // used in the leader
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };           // one per CTA
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };       // one per CTA
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };  // used in the leader
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto ld_bar = [&](int w) { return bar0 + 8u * (2 * STAGES + 6 + w); };      // one per epilogue warp (EPI_DG loads), three for EPI_RES_TS

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 2);              // the two CTAs' producers, each with its byte count
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull_bar(b), 1);
      mbar_init(tempty_bar(b), 2 * EW);          // one arrival per epilogue warp of either CTA
    }
    if (TS) {
      for (int w = 0; w < (RS ? 3 * EW : EW); ++w) mbar_init(ld_bar(w), 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)Cfg::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  gram_cluster_sync();                           // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (!chain_begin()) return;              // barriers and tensor memory are set up before the wait

  const int64_t total = tc2_units(a);
  const int64_t cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
  bool failed = false;

  if (warp == 0) {
    // ------------------------------ TMA producer (both CTAs) ------------------------------
    int s = 0;
    uint32_t ph = 0;
    const uint32_t lead_bar0 = map_to_cta(bar0, 0);          // the leader's barrier block, as seen from this CTA
    for (int64_t t = cluster_id; t < total && !failed; t += n_clusters) {
      const Tc2Unit u = tc2_unit(a, t);
      const int m0 = u.tm * 2 * BM + (int)rank * BM;             // this CTA's rows of A
      const int n0 = u.n_first + (int)rank * (u.width / 2);      // this CTA's columns of B: one or two boxes of 64
      const uint32_t bytes = Cfg::A_BYTES + (uint32_t)u.width * (BK * 2 / 2);
      for (int kb = u.kb0; kb < u.kb1; ++kb) {
        if (!mbar_wait_warp(empty_bar(s), ph ^ 1u, abort_flag)) { failed = true; break; }
        const uint32_t lead_full = lead_bar0 + 8u * s;           // the leader's full_bar(s)
        const uint32_t sa = tiles + s * Cfg::STAGE_BYTES, sb = sa + Cfg::A_BYTES;
        if (elect_one()) {
          mbar_arrive_expect_tx_remote(lead_full, bytes);
          if (A_K) {
            tma_load_2d_pair(sa, &tmA, kb * BK, m0, lead_full);
          } else {
#pragma unroll
            for (int i = 0; i < BM / 64; ++i) tma_load_2d_pair(sa + i * 8192, &tmA, m0 + i * 64, kb * BK, lead_full);
          }
          if (B_K) {
            tma_load_2d_pair(sb, &tmB, kb * BK, n0, lead_full);
            if (u.width == BN) tma_load_2d_pair(sb + 8192, &tmB, kb * BK, n0 + 64, lead_full);
          } else {
            tma_load_2d_pair(sb, &tmB, n0, kb * BK, lead_full);
            if (u.width == BN) tma_load_2d_pair(sb + 8192, &tmB, n0 + 64, kb * BK, lead_full);
          }
        }
        __syncwarp();
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
    }
    if (failed && lane == 0) {
      *abort_flag = 1;
      gram_device_fail(a.status, GRAM_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer (leader CTA only) ----------------------------
    // What bounded the main loop was this warp's own time per k-block, not its operands: with the copies left out, 643 of 647
    // cycles per k-block stayed (512 is what the MMAs take), and the wait for the operands was the barrier's latency.  With
    // the loop run by one lane and a commit per CTA: 65 536 x 2304 x 768 171 us, with all lanes and one commit 150 us
    // (1540 TFLOP/s); 65 536 x 768 x 3072 with the fp32 residual 242 -> 215 us.
    // The descriptors of stage 0 are built once: a later stage or k-step only adds to the 14-bit address field, which
    // cannot overflow inside shared memory.
    if (leader) {
      constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((A_K ? 0u : 1u) << 15) | ((B_K ? 0u : 1u) << 16) |
                                  ((uint32_t)((2 * BM) >> 4) << 24);
      int s = 0;
      uint32_t ph = 0;
      int64_t it = 0;
      const uint64_t da0 = A_K ? make_desc(tiles, 16, 1024) : make_desc(tiles, 8192, 1024);
      const uint64_t db0 = B_K ? make_desc(tiles + Cfg::A_BYTES, 16, 1024) : make_desc(tiles + Cfg::A_BYTES, 8192, 1024);
      constexpr uint32_t ka = (A_K ? 32 : 2048) >> 4, kbs = (B_K ? 32 : 2048) >> 4;
      for (int64_t t = cluster_id; t < total && !failed; t += n_clusters) {
        const Tc2Unit u = tc2_unit(a, t);
        const uint32_t idesc = idesc0 | ((uint32_t)(u.width >> 3) << 17);
        for (int c0 = u.kb0; c0 < u.kb1 && !failed; c0 += a.chain, ++it) {       // one accumulator each
          const int c1 = min(c0 + a.chain, u.kb1);
          const int buf = (int)(it & 1);
          if (!mbar_wait_warp(tempty_bar(buf), (uint32_t)((it >> 1) & 1) ^ 1u, abort_flag)) { failed = true; break; }
          tc_fence_after();
          const uint32_t tmem_d = tmem_base + (uint32_t)(buf * BN);
          for (int kb = c0; kb < c1; ++kb) {
            if (!mbar_wait_warp(full_bar(s), ph, abort_flag)) { failed = true; break; }
            tc_fence_after();
            const uint32_t soff = (uint32_t)(s * (Cfg::STAGE_BYTES >> 4));
            const uint64_t da = da0 + soff, db = db0 + soff;
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                tc_mma_pair(tmem_d, da + (uint64_t)(k * ka), db + (uint64_t)(k * kbs), idesc, (kb > c0 || k > 0) ? 1u : 0u);
              tc_commit_pair(empty_bar(s));                      // the stage is free in both CTAs once these MMAs are done
              if (kb == c1 - 1) tc_commit_pair(tfull_bar(buf));    // accumulator complete in both CTAs
            }
            __syncwarp();
            if (++s == STAGES) { s = 0; ph ^= 1u; }
          }
        }
      }
      if (failed && lane == 0) {
        *abort_flag = 1;
        gram_device_fail(a.status, GRAM_ERR_TIMEOUT);
      }
    }
  } else {
    // ------------------------------ epilogue warps (both CTAs) ------------------------------
    const int ew = warp - 2;
    const int q = warp & 3;
    const int half = ew >> 2;
    float* stage = epi_stage + ew * (32 * STAGE_LD);
    CT* C = reinterpret_cast<CT*>(a.C);
    int64_t it = 0;
    uint32_t res_blocks = 0;                      // EPI_RES_TS: this warp's running count of 32-column blocks
    for (int64_t t = cluster_id; t < total && !failed; t += n_clusters, ++it) {
      const Tc2Unit u = tc2_unit(a, t);
      const int n_lim = min(a.N, u.n_first + u.width);
      const int buf = (int)(it & 1);
      const int64_t row0 = (int64_t)u.tm * 2 * BM + (int64_t)rank * BM + q * 32;
      if constexpr (MODE == EPI_SUM) {
        const int chains = (u.kb1 - u.kb0 + a.chain - 1) / a.chain;
        if (!epilogue_unit_sum(a, reinterpret_cast<float*>(C) + (int64_t)u.split * a.split_stride, row0, u.n_first, n_lim, half, q, lane, stage,
                               tmem_base, it, chains, tfull_bar(0), map_to_cta(tempty_bar(0), 0), abort_flag)) {
          failed = true;
          break;
        }
        it += chains - 1;
      } else if constexpr (RS) {
        if (!epilogue_tile_res(a, &tmC, &tmP, (int32_t)row0, u.n_first + half * 128, n_lim, half * 128, q, lane,
                               tiles + STAGES * Cfg::STAGE_BYTES + (uint32_t)(ew * WARP_BYTES), tmem_base, buf, tfull_bar(buf),
                               (uint32_t)((it >> 1) & 1), abort_flag, map_to_cta(tempty_bar(buf), 0), ld_bar(3 * ew), res_blocks)) {
          failed = true;
          break;
        }
      } else if constexpr (TS) {
        constexpr int NB = 32 / EW;               // blocks of 32 columns per warp
        const bool ok = epilogue_tile_ts<MODE, NB>(a, &tmC, &tmP, (int32_t)row0, u.n_first + half * (NB * 32), n_lim, half * (NB * 32), q, lane,
                                    tiles + STAGES * Cfg::STAGE_BYTES + (uint32_t)(ew * WARP_BYTES), tmem_base, buf, tfull_bar(buf),
                                    (uint32_t)((it >> 1) & 1), abort_flag, map_to_cta(tempty_bar(buf), 0), ld_bar(ew),
                                    (uint32_t)(it & 1));
        if (!ok) {
          failed = true;
          break;
        }
      } else {
        CT* Cs = C + (int64_t)u.split * a.split_stride;
        if (!epilogue_tile<BN, CT, MODE, EW / 4>(a, Cs, row0, u.n_first, n_lim, half, q, lane, stage, tmem_base, buf, tfull_bar(buf),
                                                 (uint32_t)((it >> 1) & 1), abort_flag)) {
          failed = true;
          break;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(map_to_cta(tempty_bar(buf), 0));
      }
    }
    if (TS && lane == 0) bulk_wait_all();       // this warp's stores are complete before the CTA may exit
    if (failed && lane == 0) {
      *abort_flag = 1;
      gram_device_fail(a.status, GRAM_ERR_TIMEOUT);
    }
  }

  // ------------------------------ teardown --------------------------------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (warp == 1 && lane == 0) {           // let copies and MMAs already issued drain (bounded)
      uint64_t t0 = clock64();
      while (clock64() - t0 < WAIT_LIMIT_CYCLES / 64) {}
    }
    __syncthreads();
  }
  gram_cluster_sync();                        // the peer no longer reads this CTA's memory or signals its barriers
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS)
                 : "memory");
  }
}

// C(m, n) = sum over splits of part[s](m, n), in ascending s; then the epilogue.  Four columns per thread (N is a multiple of
// 8), four splits' loads on their way at once; PLAIN: the only epilogue is "add to fp32 C" or none (weight gradients).
// 3072 x 768 from six parts: 21 us with a column per thread and split after split, 13 this way (from a cold L2).
template <typename CT, bool PLAIN>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float* __restrict__ part, int splits, int64_t split_stride, int64_t M,
                                                           int N, CT* C, int64_t ldc, EpiDev e) {
  if (!chain_begin()) return;
  const int64_t n4 = M * N / 4;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = 4 * i / N;
    const int n = (int)(4 * i - m * N);
    const float* p = part + 4 * i;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < splits; s += 4) {
      float4 x[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        x[k] = s + k < splits ? *reinterpret_cast<const float4*>(p + (int64_t)(s + k) * split_stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 4; ++k) { a.x += x[k].x; a.y += x[k].y; a.z += x[k].z; a.w += x[k].w; }
    }
    if constexpr (PLAIN) {
      float4* c = reinterpret_cast<float4*>(C + m * ldc + n);
      if (e.accumulate) {
        const float4 o = *c;
        a.x += o.x; a.y += o.y; a.z += o.z; a.w += o.w;
      }
      *c = a;
    } else {
      epilogue_store<CT, bf16>(e, C, ldc, m, n, a.x);
      epilogue_store<CT, bf16>(e, C, ldc, m, n + 1, a.y);
      epilogue_store<CT, bf16>(e, C, ldc, m, n + 2, a.z);
      epilogue_store<CT, bf16>(e, C, ldc, m, n + 3, a.w);
    }
  }
}

// ------------------------------ host side --------------------------------------------------
template <int BN, bool A_K, bool B_K, typename CT, int MODE = EPI_GENERAL>
cudaError_t launch_tc(const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& args, int grid, cudaStream_t st) {
  auto kern = gemm_tc_kernel<BN, A_K, B_K, CT, MODE>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<BN>::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  launch_chain(kern, grid, TC_THREADS, TcCfg<BN>::SMEM_BYTES, st, ma, mb, args);
  return cudaGetLastError();
}

template <int BN, typename CT>
cudaError_t launch_tc_major(bool a_k, bool b_k, const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& args, int grid,
                            cudaStream_t st) {
  if (a_k && b_k) return launch_tc<BN, true, true, CT>(ma, mb, args, grid, st);
  if (a_k && !b_k) return launch_tc<BN, true, false, CT>(ma, mb, args, grid, st);
  if (!a_k && b_k) return launch_tc<BN, false, true, CT>(ma, mb, args, grid, st);
  return launch_tc<BN, false, false, CT>(ma, mb, args, grid, st);
}

template <bool A_K, bool B_K, typename CT, int MODE = EPI_GENERAL, int EW = EPI_WARPS>
cudaError_t launch_tc2(const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& args, int grid, cudaStream_t st,
                       const CUtensorMap* mc = nullptr, const CUtensorMap* mp = nullptr) {
  using Tc2 = Tc2Cfg<EW, warp_bytes<CT, MODE>()>;
  auto kern = gemm_tc2_kernel<A_K, B_K, CT, MODE, EW>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Tc2::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(Tc2::THREADS);
  cfg.dynamicSmemBytes = Tc2::SMEM_BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = chain_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, ma, mb, mc ? *mc : ma, mp ? *mp : (mc ? *mc : ma), args);
}
template <typename CT>
cudaError_t launch_tc2_major(bool a_k, bool b_k, const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& args, int grid,
                             cudaStream_t st) {
  if (a_k && b_k) return launch_tc2<true, true, CT>(ma, mb, args, grid, st);
  if (a_k && !b_k) return launch_tc2<true, false, CT>(ma, mb, args, grid, st);
  if (!a_k && b_k) return launch_tc2<false, true, CT>(ma, mb, args, grid, st);
  return launch_tc2<false, false, CT>(ma, mb, args, grid, st);
}

}  // namespace

static bool pair_enabled_env() {
  static const bool on = []() { const char* v = getenv("GRAM_GEMM_PAIR"); return !(v && v[0] == '0'); }();
  return on;
}
// GRAM_GEMM_RES_TS=0 in the environment keeps the register path of the fp32 residual epilogue (for comparisons)
static bool res_ts_env() {
  static const bool on = []() { const char* v = getenv("GRAM_GEMM_RES_TS"); return !(v && v[0] == '0'); }();
  return on;
}
bool gemm_fused_colsum(int dtype, int64_t M, int N) {
  const bool bn256 = (N % 256 == 0 || N > 1024);
  return dtype == GRAM_BF16 && pair_enabled_env() && bn256 && M >= 2 * BM && M < ((int64_t)1 << 31) && get_encode_fn() != nullptr;
}

gram_status gemm_ws_alloc(gram_ctx* ctx, GemmWorkspace* ws, size_t splitk_bytes) {
  ws->splitk_bytes = splitk_bytes;
  if (splitk_bytes) GRAM_CUDA(ctx, cudaMalloc(&ws->splitk, splitk_bytes));
  return GRAM_OK;
}
void gemm_ws_free(GemmWorkspace* ws) {
  cudaFree(ws->splitk);
  *ws = GemmWorkspace();
}

static EpiDev epi_dev(const GemmEpilogue& epi) {
  return EpiDev{epi.bias, epi.res, epi.res_mean, epi.res_rstd, epi.res_gamma, epi.res_beta, epi.pre, epi.dgelu_pre, epi.copy_out,
                epi.colsum_part, epi.gelu, epi.accumulate};
}

// Both products go together where their tiles are at most three blocks an SM: above, each fills the chip by itself.  Together against
// apart with the bias gradient's two launches, widths 16 to 128 over 100 to 14 000 rows: 0.59 of the time up to 148 tiles, 0.74 up to
// 370, 0.81 (0.98 at worst) up to 444, 0.96 (1.57 at worst) on from there to 900.
// Parts of the K ranges: the longer chain is halved while the blocks fit the SMs at once (a width of 128: 478 us a step, 499 with half
// as many blocks again) and it is more than one round of four k-blocks.  dW's chain runs over the rows, and dX's blocks, which are as
// many as the rows are, would leave it no parts: while it is longer than four rounds it is halved up to a block an SM whatever dX takes.
// us with the SMs shared out and this way: 192 x 64 over 4096 rows 32.6 and 16.6 (apart 21.0), over 6400 47.3 and 23.7, 288 x 96 over 2952
// 44.8 and 22.8, 384 x 128 48.3 and 32.0, 96 x 32 over 10 000 22.2 and 15.4; a line at two rounds or eight loses up to a fifth at single sizes.
// What a group adds up in one chain is no longer than in the product alone (`fold`; error against 64 bits of 192 x 64 over 6400 4.9e-7 -> 2.0e-7, which is
// the product alone): folding costs 3 to 5 % of a launch of many rounds, and launches that need none have a kernel of
// their own (steps of the check's size take up to 1 % less than with folding in all of them).  Both keep to the registers of two blocks an SM.
bool gemm_f32_grads_together(int64_t T, int N, int K) {
  const int64_t w = (int64_t)ceil_div(N, 32) * ceil_div(K, 32), x = ceil_div64(T, 32) * ceil_div(K, 32);
  return T > 0 && N > 0 && K > 0 && w + x <= 3 * kNumSMs;
}
gram_status gemm_f32_grads(gram_ctx* ctx, const float* dY, const float* X, float* dW, const char* dw_tag, float* db, const float* W, float* dX,
                           int64_t T, int N, int K, const GemmEpilogue& epi, cudaStream_t st) {
  if (!dY || !X || !dW || !W || !dX || !gemm_f32_grads_together(T, N, K)) return gram_set_error(ctx, "gemm: bad gradient products"), GRAM_ERR_ARG;
  ProfScope prof(ctx, GRAM_K_GEMM, 4.0 * (double)T * N * (double)K, 1, st, dw_tag ? dw_tag : "gemm_f32", epi.tag ? epi.tag : "gemm_f32");
  const int most = F32_MAX_SPLIT < gram_cluster_blocks(ctx) ? F32_MAX_SPLIT : gram_cluster_blocks(ctx);
  constexpr int SK = F32Cfg<32, 4>::SK, ROUND = 4 * SK;
  F32Pair a = {};
  a.w_tiles = ceil_div(N, 32) * ceil_div(K, 32);
  a.x_tiles = (int32_t)ceil_div64(T, 32) * ceil_div(K, 32);
  a.wp = a.xp = 1;
  for (;;) {
    const int64_t wk = a.wp < most ? ceil_div64(T, a.wp) : 0, xk = a.xp < most ? ceil_div(N, a.xp) : 0;
    const bool w_first = wk >= xk;
    if ((w_first ? wk : xk) <= ROUND) break;
    const int64_t w = (int64_t)a.w_tiles * a.wp, x = (int64_t)a.x_tiles * a.xp;
    if (w + x + (w_first ? w : x) > 2 * kNumSMs && !(w_first && wk > 4 * ROUND && 2 * w <= kNumSMs)) break;
    if (w_first) a.wp *= 2;
    else a.xp *= 2;
  }
  EpiDev ew = {};
  ew.accumulate = 1;
  a.w = f32_prod(dY, N, X, K, dW, K, N, K, T, ceil_div64(ceil_div64(T, a.wp), SK) * SK, ew);
  a.w.row_sums = db;
  auto fold_of = [&](int64_t tiles, int64_t k) {
    const F32Plan alone = f32_plan(tiles, k, false, most);
    return (int32_t)ceil_div64(alone.k_per_part, SK * alone.groups);
  };
  a.w.fold = fold_of(a.w_tiles, T);
  a.x = f32_prod(dY, N, W, K, dX, K, T, K, N, (int64_t)ceil_div(ceil_div(N, a.xp), SK) * SK, epi_dev(epi));
  a.x.fold = fold_of(a.x_tiles, N);
  const int blocks = a.wp > a.xp ? a.wp : a.xp;
  a.w_clusters = ceil_div(a.w_tiles * a.wp, blocks);
  auto folds = [](const F32Prod& p) { return p.k_per_part > (int64_t)p.fold * ROUND; };
  auto kern = folds(a.w) || folds(a.x) ? gemm_f32_pair_kernel<true> : gemm_f32_pair_kernel<false>;
  if (blocks > 8) GRAM_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(blocks * (a.w_clusters + ceil_div(a.x_tiles * a.xp, blocks))));
  cfg.blockDim = dim3(F32Cfg<32, 4>::THREADS);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)blocks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = chain_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  GRAM_CUDA(ctx, cudaLaunchKernelEx(&cfg, kern, a));
  return GRAM_OK;
}

gram_status gemm_launch(gram_ctx* ctx, GemmWorkspace* ws, int dtype, const void* A, int a_kmajor, int64_t lda,
                        const void* B, int b_kmajor, int64_t ldb, void* C, int c_f32, int64_t ldc, int64_t M, int N,
                        int64_t K, const GemmEpilogue& epi, int allow_splitk, cudaStream_t st) {
  if (M < 0 || N < 0 || K < 0) return gram_set_error(ctx, "gemm: negative size"), GRAM_ERR_ARG;
  if (M == 0 || N == 0) return GRAM_OK;
  if (!A || !B || !C) return gram_set_error(ctx, "gemm: null operand"), GRAM_ERR_ARG;
  const EpiDev e = epi_dev(epi);
  if (dtype == GRAM_F32) {
    if (!c_f32) return gram_set_error(ctx, "gemm: fp32 operands need an fp32 result"), GRAM_ERR_UNSUPPORTED;
    ProfScope prof(ctx, GRAM_K_GEMM, 2.0 * (double)M * N * (double)K, 1, st, epi.tag ? epi.tag : "gemm_f32");
    // 64 x 64 tiles once they give every SM a block, else 32 x 32
    const int64_t b64 = ceil_div64(M, 64) * ceil_div64(N, 64), b32 = ceil_div64(M, 32) * ceil_div64(N, 32);
    const bool big = b64 >= kNumSMs;
    const int most = F32_MAX_SPLIT < gram_cluster_blocks(ctx) ? F32_MAX_SPLIT : gram_cluster_blocks(ctx);
    const F32Plan p = f32_plan(big ? b64 : b32, K, big, most);
    if (ceil_div64(M, big ? 64 : 32) > 65535)
      return gram_set_error(ctx, "gemm: %lld rows are more than an fp32 product takes", (long long)M), GRAM_ERR_UNSUPPORTED;
    auto launch = big ? launch_f32_major<64, 1> : (p.groups == 4 ? launch_f32_major<32, 4> : (p.groups == 2 ? launch_f32_major<32, 2> : launch_f32_major<32, 1>));
    const cudaError_t ferr = launch(a_kmajor, b_kmajor, f32_prod((const float*)A, lda, (const float*)B, ldb, (float*)C, ldc, M, N, K, p.k_per_part, e), p.parts, st);
    if (ferr != cudaSuccess) return gram_set_error(ctx, "gemm launch failed: %s", cudaGetErrorString(ferr)), GRAM_ERR_CUDA;
    return GRAM_OK;
  }
  // ---- bf16 on the tensor cores ----
  if ((lda % 8) || (ldb % 8) || ((uintptr_t)A % 16) || ((uintptr_t)B % 16) || ((uintptr_t)C % 16) || (ldc % 8) ||
      K == 0)
    return gram_set_error(ctx, "gemm: bf16 operands need 16-byte aligned rows (sizes multiples of 8)"), GRAM_ERR_UNSUPPORTED;
  if (e.accumulate && !c_f32) return gram_set_error(ctx, "gemm: accumulation needs an fp32 result"), GRAM_ERR_UNSUPPORTED;
  if ((e.res != nullptr) + (e.dgelu_pre != nullptr) + (e.accumulate != 0) > 1)
    return gram_set_error(ctx, "gemm: at most one of residual, GELU derivative and accumulation per product"), GRAM_ERR_UNSUPPORTED;
  if ((N % 8) || (e.bias && ((uintptr_t)e.bias % 16)) || (e.res_gamma && (((uintptr_t)e.res_gamma % 16) || ((uintptr_t)e.res_beta % 16))))
    return gram_set_error(ctx, "gemm: N must be a multiple of 8 and the epilogue's vectors 16-byte aligned"), GRAM_ERR_UNSUPPORTED;
  const int BNsel = (N % 256 == 0 || N > 1024) ? 256 : (N > 64 ? 128 : 64);
  // pairs of SMs (256 x 256 tiles) when the problem has full-height tiles; GRAM_GEMM_PAIR=0 keeps single CTAs
  const bool pair = pair_enabled_env() && BNsel == 256 && M >= 2 * BM;
  CUtensorMap ma, mb;
  bool ok;
  if (a_kmajor) ok = make_map(&ma, A, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM);
  else ok = make_map(&ma, A, (uint64_t)M, (uint64_t)K, (uint64_t)lda, 64, BK);
  if (b_kmajor) ok = ok && make_map(&mb, B, (uint64_t)K, (uint64_t)N, (uint64_t)ldb, BK, (uint32_t)(pair ? 64 : BNsel));
  else ok = ok && make_map(&mb, B, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, 64, BK);
  if (!ok) return gram_set_error(ctx, "gemm: cuTensorMapEncodeTiled failed"), GRAM_ERR_CUDA;

  TcArgs args;
  args.M = M;
  args.N = N;
  args.num_kb = (int32_t)ceil_div64(K, BK);
  args.n_tiles_m = (int32_t)ceil_div64(M, pair ? 2 * BM : BM);
  args.n_tiles_n = ceil_div(N, BNsel);
  args.status = gram_status_word(ctx);
  const int64_t tiles = (int64_t)args.n_tiles_m * args.n_tiles_n;
  const int units = pair ? kNumSMs / 2 : kNumSMs;        // CTAs, or CTA pairs, that run at once
  int splits = 1;
  // weight gradients: a plain fp32 result, added to C or not
  const bool sum_form = pair && !a_kmajor && !b_kmajor && c_f32 && !e.bias && !e.gelu && !e.dgelu_pre && !e.res && !e.copy_out && !e.pre;
  // parts of the K range that go through memory: where the tiles do not fill the chip, as many as the workspace takes
  const int64_t per = (int64_t)M * N * (int64_t)sizeof(float);
  const int64_t most = allow_splitk && tiles < units && ws && ws->splitk ? (int64_t)(ws->splitk_bytes / per) : 1;
  int chains = 1;
  if (allow_splitk && tiles < units && args.num_kb >= 16 && (sum_form || most > 1)) {
    // chains of additions in the accumulator: between 2 and 4 per CTA (pair), each of at least eight k-blocks; among those, the
    // count that leaves the last wave fullest.  Longer chains cost precision: the tensor core adds into its fp32 accumulator by
    // cutting off, so the error of a chain grows with its length, while the chains themselves are added with rounding
    // (65 536 rows, 3072 x 768, against 64 bits: 1.2e-5 from 6 chains, 3.8e-5 from 2).
    int lo = (int)((2 * units + tiles - 1) / tiles), hi = (int)((4 * units + tiles - 1) / tiles);
    int cap = args.num_kb / 8;
    if (!sum_form && cap > most) cap = (int)most;          // each chain is a part here
    if (hi > cap) hi = cap;
    if (lo > hi) lo = hi;
    double best = -1.0;
    for (int ch = lo; ch <= hi && ch >= 1; ++ch) {
      const int64_t total = tiles * ch;
      const double fill = (double)total / (double)(ceil_div64(total, units) * units);
      if (fill > best + 1e-9) { best = fill; chains = ch; }
    }
  }
  // weight gradients add their chains in registers: neither the workspace nor a chip full of tiles lets a chain grow.  Longer ones
  // are cut evenly, so that the count still fills waves (36 tiles, 81 920 rows: 12 chains 268 us, the 7 that suffice 293).
  if (sum_form) chains *= ceil_div(ceil_div(args.num_kb, chains), SUM_CHAIN_MAX);
  splits = chains;
  args.kb_per_split = ceil_div(args.num_kb, splits);
  splits = ceil_div(args.num_kb, args.kb_per_split);
  args.chain = args.kb_per_split;
  if (sum_form && splits > 1) {
    // The chains of a unit are added in its epilogue's registers, so that the parts of the K range that go through memory are
    // only as many as fill the chip: of those counts, from one unit per pair of SMs up, the one that leaves the last wave
    // fullest, the smallest of equals (within two per cent: a part costs its write, its read and a place in the sum).
    // 42 500 rows, a layer's four weight gradients on average: product 98 -> 90 us, sum of the parts 11.4 -> 7.0.
    int best_sp = 1;
    double best = 0.0;
    for (int sp = (int)(splits < most ? splits : most); sp >= 1; --sp) {
      const int per_part = ceil_div(splits, sp);                         // chains of a part
      if (ceil_div(splits, per_part) != sp) continue;
      const int64_t total = tiles * sp;
      const double fill = (double)tiles * splits / ((double)ceil_div64(total, units) * units * per_part);
      if (fill >= 0.98 * best) { best_sp = sp; if (fill > best) best = fill; }
    }
    args.kb_per_split = ceil_div(splits, best_sp) * args.chain;
    splits = ceil_div(args.num_kb, args.kb_per_split);
  }
  args.splits = splits;
  const bool sum_regs = sum_form && (args.chain < args.kb_per_split || args.chain >= SUM_CHAIN_ALONE);
  // The last wave's tiles as halves where twice as many still fit one wave.
  args.half_from = INT32_MAX;
  int64_t work = tiles * splits;
  if (pair && splits == 1) {
    const int64_t rest = tiles % units;
    if (rest > 0 && 2 * rest <= units && tiles - rest < INT32_MAX) {
      args.half_from = (int32_t)(tiles - rest);
      work += rest;
    }
  }
  cudaError_t err;
  ProfScope prof(ctx, GRAM_K_GEMM, 2.0 * (double)M * N * (double)K, splits > 1 ? 2 : 1, st, epi.tag ? epi.tag : "gemm");
  const int grid = pair ? 2 * (int)(work < units ? work : units)
                        : (int)((tiles * splits < kNumSMs) ? tiles * splits : kNumSMs);
  if (splits > 1) {
    args.C = ws->splitk;
    args.ldc = N;
    args.split_stride = (int64_t)M * N;
    args.epi = EpiDev{nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0, 0};
    if (sum_regs) err = launch_tc2<false, false, float, EPI_SUM>(ma, mb, args, grid, st);
    else if (sum_form) err = launch_tc2<false, false, float, EPI_BIAS>(ma, mb, args, grid, st);
    else if (pair) err = launch_tc2_major<float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else if (BNsel == 256) err = launch_tc_major<256, float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else if (BNsel == 128) err = launch_tc_major<128, float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else err = launch_tc_major<64, float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    if (err != cudaSuccess) return gram_set_error(ctx, "gemm launch failed: %s", cudaGetErrorString(err)), GRAM_ERR_CUDA;
    int rb = (int)ceil_div64(M * N / 4, 256);
    if (rb > kNumSMs * 16) rb = kNumSMs * 16;
    const bool plain = c_f32 && !e.bias && !e.gelu && !e.dgelu_pre && !e.res && !e.copy_out && !e.pre;
    if (plain) launch_chain(splitk_reduce_kernel<float, true>, rb, 256, 0, st, ws->splitk, splits, (int64_t)M * N, M, N, (float*)C, ldc, e);
    else if (c_f32) launch_chain(splitk_reduce_kernel<float, false>, rb, 256, 0, st, ws->splitk, splits, (int64_t)M * N, M, N, (float*)C, ldc, e);
    else launch_chain(splitk_reduce_kernel<bf16, false>, rb, 256, 0, st, ws->splitk, splits, (int64_t)M * N, M, N, (bf16*)C, ldc, e);
    GRAM_LAUNCH_CHECK(ctx);
    return GRAM_OK;
  }
  args.C = C;
  args.ldc = ldc;
  args.split_stride = 0;
  args.epi = e;
  if (e.colsum_part && !(pair && e.dgelu_pre && !c_f32))
    return gram_set_error(ctx, "gemm: column-sum partials need the paired GELU-derivative variant"), GRAM_ERR_UNSUPPORTED;
  const bool dg_only = e.dgelu_pre && !e.bias && !e.res && !e.accumulate && !e.copy_out && !e.gelu && !c_f32 && a_kmajor &&
                       !b_kmajor;
  const bool others = e.gelu || e.dgelu_pre || e.res || e.accumulate || e.copy_out || e.pre;
  const bool m_bias = !others;
  const bool m_gelu = e.gelu && !e.dgelu_pre && !e.res && !e.accumulate && !e.copy_out && !c_f32 && a_kmajor && b_kmajor;
  const bool m_res = e.res && !e.gelu && !e.dgelu_pre && !e.accumulate && !e.pre && c_f32 && a_kmajor;
  if (pair) {
    // bf16 results leave through bulk tensor stores: maps of C and of the GELU-derivative matrix (boxes of 32 rows x 64 columns)
    const void* aux = e.gelu ? e.pre : e.dgelu_pre;          // null: the value alone
    const bool ts = !c_f32 && M < (int64_t)1 << 31 && (!aux || (uintptr_t)aux % 16 == 0);
    CUtensorMap mc, mp;
    bool ts_ok = ts && make_map(&mc, C, (uint64_t)N, (uint64_t)M, (uint64_t)ldc, 64, 32);
    if (ts_ok && aux) ts_ok = make_map(&mp, aux, (uint64_t)N, (uint64_t)M, (uint64_t)ldc, 64, 32);
    const CUtensorMap* pc = &mc;
    const CUtensorMap* pp = aux ? &mp : &mc;
    // the fp32 residual products with a short reduction (K <= 1024: the output projection of attention), where the epilogue's
    // memory traffic outlasts the main loop: result and residual as fp32 boxes of 32 rows x 32 columns through bulk tensor
    // copies (no bf16 copy on this path).  With longer K the register path keeps six pipeline stages instead of four and
    // is the faster one (65 536 x 768: 209 against 244 us at K = 3072, 162 against 191 at K = 2304).
    CUtensorMap mcf, mrf;
    const bool rs_ok = m_res && !e.copy_out && K <= 1024 && res_ts_env() && M < (int64_t)1 << 31 && (uintptr_t)e.res % 16 == 0 &&
                       make_map_f32(&mcf, C, (uint64_t)N, (uint64_t)M, (uint64_t)ldc, 32, 32) &&
                       make_map_f32(&mrf, e.res, (uint64_t)N, (uint64_t)M, (uint64_t)ldc, 32, 32);
    if (e.colsum_part && !(dg_only && ts_ok))
      return gram_set_error(ctx, "gemm: column-sum partials need the GELU-derivative variant with bulk stores"), GRAM_ERR_UNSUPPORTED;
    if (dg_only && ts_ok) err = launch_tc2<true, false, bf16, EPI_DG, 16>(ma, mb, args, grid, st, pc, pp);
    else if (m_gelu && ts_ok && e.pre) err = launch_tc2<true, true, bf16, EPI_GELU, 8>(ma, mb, args, grid, st, pc, pp);
    else if (m_gelu && ts_ok) err = launch_tc2<true, true, bf16, EPI_GELU_V, 8>(ma, mb, args, grid, st, pc, pp);
    else if (m_res && rs_ok && b_kmajor) err = launch_tc2<true, true, float, EPI_RES_TS>(ma, mb, args, grid, st, &mcf, &mrf);
    else if (m_res && rs_ok && !b_kmajor) err = launch_tc2<true, false, float, EPI_RES_TS>(ma, mb, args, grid, st, &mcf, &mrf);
    else if (m_res && b_kmajor) err = launch_tc2<true, true, float, EPI_RES>(ma, mb, args, grid, st);
    else if (m_res && !b_kmajor) err = launch_tc2<true, false, float, EPI_RES>(ma, mb, args, grid, st);
    else if (m_bias && a_kmajor && b_kmajor && ts_ok) err = launch_tc2<true, true, bf16, EPI_BIAS, 8>(ma, mb, args, grid, st, pc, pp);
    else if (m_bias && a_kmajor && !b_kmajor && ts_ok) err = launch_tc2<true, false, bf16, EPI_BIAS, 8>(ma, mb, args, grid, st, pc, pp);
    else if (sum_regs) err = launch_tc2<false, false, float, EPI_SUM>(ma, mb, args, grid, st);
    else if (m_bias && c_f32 && a_kmajor && !b_kmajor) err = launch_tc2<true, false, float, EPI_BIAS>(ma, mb, args, grid, st);
    else if (c_f32) err = launch_tc2_major<float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else err = launch_tc2_major<bf16>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
  } else if (dg_only) {
    if (BNsel == 256) err = launch_tc<256, true, false, bf16, EPI_DG>(ma, mb, args, grid, st);
    else if (BNsel == 128) err = launch_tc<128, true, false, bf16, EPI_DG>(ma, mb, args, grid, st);
    else err = launch_tc<64, true, false, bf16, EPI_DG>(ma, mb, args, grid, st);
  } else if (c_f32) {
    if (BNsel == 256) err = launch_tc_major<256, float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else if (BNsel == 128) err = launch_tc_major<128, float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else err = launch_tc_major<64, float>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
  } else {
    if (BNsel == 256) err = launch_tc_major<256, bf16>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else if (BNsel == 128) err = launch_tc_major<128, bf16>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
    else err = launch_tc_major<64, bf16>(a_kmajor, b_kmajor, ma, mb, args, grid, st);
  }
  if (err != cudaSuccess) return gram_set_error(ctx, "gemm launch failed: %s", cudaGetErrorString(err)), GRAM_ERR_CUDA;
  return GRAM_OK;
}
