// Attention over sequences of up to 256 rows (head width 64, bf16 operands, fp32 softmax) with warp-level MMA.
//
// One block owns one (sequence, head) and keeps what every row needs in shared memory (forward: K, V; backward: Q, K, V,
// dO), each row once from HBM.  A warp owns 16 rows at a time and walks the other side in chunks, with its scores,
// probabilities and results in registers:
//   forward        16 query rows, 64 keys a chunk, running maximum and sum
//   backward, dQ   16 query rows, 32 keys a chunk:    P = exp2(c S - lse), dS = P (dP - delta), dQ += dS K
//   backward, dK   16 key rows, 32 queries a chunk:   the transposed tiles, so that P^T and dS^T are the left operands of
//                  dV += P^T dO and dK += dS^T Q as they stand in registers
// The second walk computes S and dP again (14 S^2 dh flops instead of 10), which costs less than passing P and dS
// between warps would: no tile leaves a warp, there is one barrier after the loads, and several blocks fit an SM.
// Chunks stop at the sequence's last 16 rows (and at the diagonal of causal launches), so a text of 147 tokens costs
// 160 rows where 128-row tensor-memory tiles cost 256: 364 -> 152 us forward, 936 -> 516 us backward per layer of 54 000
// such rows.  What bounds them now is the shared-memory traffic of the fragments (two B fragments per 16 x 16 x 16 product).
#include "layers.h"
#include "warp_mma.cuh"

namespace {
using namespace wmma16;

constexpr int DH = 64, LD = DH + 8;
constexpr int FL_MAX_WARPS = 8;                  // most warps of a forward block
constexpr int FL_BWD_WARPS = 12;                 // and of a backward block
constexpr int STAGE_ELEMS = 16 * LD;             // a warp's private 16-row tile

struct FlashArgs {
  const bf16* qkv;
  bf16* out;                 // forward
  float* lse;                // [H, T] base-2 log-sum-exp of the scaled scores
  const bf16* dctx;          // backward
  const bf16* octx;
  bf16* dqkv;
  float* colpart;            // [.., 3d] column sums of dqkv, one row per sequence of the launch, or null
  int64_t T;
  int32_t S, d, H, rows_cap; // rows_cap: rows the shared-memory tiles hold
  float c, scale;            // scale * log2(e), 1 / sqrt(dh)
  const int32_t* seq_len;
  const int32_t* seq_off;
  const int32_t* seq_list;
};

struct FlashSeq {
  int64_t row0;
  int len, h;
  int64_t slot;              // running number of the sequence in this launch
};
__device__ __forceinline__ FlashSeq flash_seq(const FlashArgs& a) {
  FlashSeq x;
  x.slot = blockIdx.x / a.H;
  x.h = blockIdx.x % a.H;
  const int64_t s = a.seq_list ? a.seq_list[x.slot] : x.slot;
  x.row0 = a.seq_off ? (int64_t)a.seq_off[s] : s * a.S;
  x.len = min(a.seq_len ? a.seq_len[s] : a.S, a.rows_cap);
  return x;
}

// rows 0 .. len-1 of one head's slice -> shared memory, zeros up to the next multiple of 64 (below rows_cap)
__device__ __forceinline__ void flash_load(const bf16* __restrict__ src, int64_t ld, int len, int cap, bf16* dst) {
  const int pad = min((len + 63) & ~63, cap);
  for (int i = threadIdx.x; i < pad * 8; i += blockDim.x) {
    const int s = i >> 3, c = (i & 7) * 8;
    if (s < len)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst + s * LD + c)), "l"(src + (int64_t)s * ld + c)
                   : "memory");
    else
      *reinterpret_cast<uint4*>(dst + s * LD + c) = make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ void flash_loads_done() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

// a warp's 16 x 64 results (C layout) as bf16 through its private tile into whole 128-byte rows
__device__ __forceinline__ void flash_store(const float (&o)[DH / 8][4], bf16* stage, int rows, bf16* dst, int64_t ld, int lane) {
  const int g = lane >> 2, q = lane & 3;
  __syncwarp();
#pragma unroll
  for (int nt = 0; nt < DH / 8; ++nt) {
    *reinterpret_cast<uint32_t*>(stage + g * LD + nt * 8 + 2 * q) = pack2(o[nt][0], o[nt][1]);
    *reinterpret_cast<uint32_t*>(stage + (g + 8) * LD + nt * 8 + 2 * q) = pack2(o[nt][2], o[nt][3]);
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = i * 4 + (lane >> 3), c = (lane & 7) * 8;
    if (r < rows) *reinterpret_cast<uint4*>(dst + (int64_t)r * ld + c) = *reinterpret_cast<const uint4*>(stage + r * LD + c);
  }
}
// adds the columns 2 lane, 2 lane + 1 of the first `rows` rows of the private tile (bf16 as stored), rows ascending
__device__ __forceinline__ void flash_colsum(const bf16* stage, int rows, int lane, float2& sum) {
#pragma unroll 4
  for (int r = 0; r < rows; ++r) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(stage + r * LD + 2 * lane));
    sum.x += f.x;
    sum.y += f.y;
  }
}

template <bool CAUSAL>
__global__ void __launch_bounds__(FL_MAX_WARPS * 32, 2) attn_flash_fwd_kernel(FlashArgs a) {
  if (!chain_begin()) return;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  bf16* Ks = reinterpret_cast<bf16*>(smem_raw);
  bf16* Vs = Ks + a.rows_cap * LD;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, g = lane >> 2, q = lane & 3;
  bf16* stage = Vs + a.rows_cap * LD + warp * STAGE_ELEMS;
  const FlashSeq x = flash_seq(a);
  const bf16* base = a.qkv + x.row0 * 3 * (int64_t)a.d + x.h * DH;
  const int64_t ld3 = 3 * (int64_t)a.d;
  flash_load(base + a.d, ld3, x.len, a.rows_cap, Ks);
  flash_load(base + 2 * a.d, ld3, x.len, a.rows_cap, Vs);
  flash_loads_done();
  bf16* ob = a.out + x.row0 * (int64_t)a.d + x.h * DH;
  for (int r0 = warp * 16; r0 < x.len; r0 += nw * 16) {
    const int rows = min(16, x.len - r0);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {                        // this tile's queries through the private tile
      const int r = i * 4 + (lane >> 3), c = (lane & 7) * 8;
      *reinterpret_cast<uint4*>(stage + r * LD + c) =
          r < rows ? *reinterpret_cast<const uint4*>(base + (int64_t)(r0 + r) * ld3 + c) : make_uint4(0u, 0u, 0u, 0u);
    }
    __syncwarp();
    uint32_t qa[4][4];
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) load_a_rows(stage, LD, 0, kt * 16, lane, qa[kt][0], qa[kt][1], qa[kt][2], qa[kt][3]);
    float o[DH / 8][4];
#pragma unroll
    for (int nt = 0; nt < DH / 8; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    const int i0 = r0 + g, i1 = r0 + g + 8;
    const int kend = CAUSAL ? min(x.len, r0 + 16) : x.len;         // keys some row of the tile can see
    for (int k0 = 0; k0 < kend; k0 += 64) {
      float p[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) p[nt][0] = p[nt][1] = p[nt][2] = p[nt][3] = 0.f;
#pragma unroll
      for (int nt = 0; nt < 8; nt += 2) {
        if (k0 + nt * 8 < kend) {
#pragma unroll
          for (int kt = 0; kt < 4; ++kt) {
            uint32_t b0, b1, b2, b3;
            load_b_rows(Ks, LD, k0 + nt * 8, kt * 16, lane, b0, b1, b2, b3);
            mma16816(p[nt], qa[kt][0], qa[kt][1], qa[kt][2], qa[kt][3], b0, b1);
            mma16816(p[nt + 1], qa[kt][0], qa[kt][1], qa[kt][2], qa[kt][3], b2, b3);
          }
        }
      }
      if (k0 + 64 > x.len || (CAUSAL && k0 + 63 > r0)) {
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = k0 + nt * 8 + 2 * q + (e & 1);
            if (j >= x.len || (CAUSAL && j > (e < 2 ? i0 : i1))) p[nt][e] = -INFINITY;
          }
      }
      float n0 = m0, n1 = m1;
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        n0 = fmaxf(n0, fmaxf(p[nt][0], p[nt][1]));
        n1 = fmaxf(n1, fmaxf(p[nt][2], p[nt][3]));
      }
      n0 = quad_max(n0);
      n1 = quad_max(n1);
      const float c0 = n0 == -INFINITY ? 0.f : n0 * a.c, c1 = n1 == -INFINITY ? 0.f : n1 * a.c;
      const float f0 = fast_exp2(fmaf(m0, a.c, -c0)), f1 = fast_exp2(fmaf(m1, a.c, -c1));     // 0 before the first key
      m0 = n0;
      m1 = n1;
      l0 *= f0;
      l1 *= f1;
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        p[nt][0] = fast_exp2(fmaf(p[nt][0], a.c, -c0)); p[nt][1] = fast_exp2(fmaf(p[nt][1], a.c, -c0));
        p[nt][2] = fast_exp2(fmaf(p[nt][2], a.c, -c1)); p[nt][3] = fast_exp2(fmaf(p[nt][3], a.c, -c1));
        l0 += p[nt][0] + p[nt][1];
        l1 += p[nt][2] + p[nt][3];
        o[nt][0] *= f0; o[nt][1] *= f0; o[nt][2] *= f1; o[nt][3] *= f1;
      }
#pragma unroll
      for (int kt = 0; kt < 4; ++kt) {
        if (k0 + kt * 16 < kend) {
          const uint32_t a0 = pack2(p[2 * kt][0], p[2 * kt][1]), a1 = pack2(p[2 * kt][2], p[2 * kt][3]);
          const uint32_t a2 = pack2(p[2 * kt + 1][0], p[2 * kt + 1][1]), a3 = pack2(p[2 * kt + 1][2], p[2 * kt + 1][3]);
#pragma unroll
          for (int nt = 0; nt < DH / 8; nt += 2) {
            uint32_t b0, b1, b2, b3;
            load_b_trans(Vs, LD, k0 + kt * 16, nt * 8, lane, b0, b1, b2, b3);
            mma16816(o[nt], a0, a1, a2, a3, b0, b1);
            mma16816(o[nt + 1], a0, a1, a2, a3, b2, b3);
          }
        }
      }
    }
    l0 = quad_sum(l0);
    l1 = quad_sum(l1);
    const float v0 = l0 > 0.f ? 1.f / l0 : 0.f, v1 = l1 > 0.f ? 1.f / l1 : 0.f;
#pragma unroll
    for (int nt = 0; nt < DH / 8; ++nt) { o[nt][0] *= v0; o[nt][1] *= v0; o[nt][2] *= v1; o[nt][3] *= v1; }
    if (a.lse && q == 0) {
      float* lp = a.lse + (int64_t)x.h * a.T + x.row0 + r0;
      if (g < rows) lp[g] = m0 * a.c + __log2f(l0);
      if (g + 8 < rows) lp[g + 8] = m1 * a.c + __log2f(l1);
    }
    flash_store(o, stage, rows, ob + (int64_t)r0 * a.d, a.d, lane);
  }
}

// NWMAX: most warps a launch of this form has.  5: two blocks per SM; 12: one.
template <bool CAUSAL, int NWMAX>
__global__ void __launch_bounds__(NWMAX * 32, NWMAX <= 5 ? 2 : 1) attn_flash_bwd_kernel(FlashArgs a) {
  if (!chain_begin()) return;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  bf16* Qs = reinterpret_cast<bf16*>(smem_raw);
  bf16* Ks = Qs + a.rows_cap * LD;
  bf16* Vs = Ks + a.rows_cap * LD;
  bf16* dOs = Vs + a.rows_cap * LD;
  float* s_lse = reinterpret_cast<float*>(dOs + a.rows_cap * LD);
  float* s_delta = s_lse + a.rows_cap;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, g = lane >> 2, q = lane & 3;
  float* s_col = s_delta + a.rows_cap;                                  // [3][warps][64]
  bf16* stage = reinterpret_cast<bf16*>(s_col + 3 * FL_BWD_WARPS * DH) + warp * STAGE_ELEMS;
  const FlashSeq x = flash_seq(a);
  const int64_t ld3 = 3 * (int64_t)a.d;
  const bf16* base = a.qkv + x.row0 * ld3 + x.h * DH;
  const bf16* dob = a.dctx + x.row0 * (int64_t)a.d + x.h * DH;
  const bf16* ob = a.octx + x.row0 * (int64_t)a.d + x.h * DH;
  flash_load(base, ld3, x.len, a.rows_cap, Qs);
  flash_load(base + a.d, ld3, x.len, a.rows_cap, Ks);
  flash_load(base + 2 * a.d, ld3, x.len, a.rows_cap, Vs);
  flash_load(dob, a.d, x.len, a.rows_cap, dOs);
  // delta = dO . O per row, eight lanes a row; rows past the end: lse = +inf makes their probabilities zero
  for (int r = threadIdx.x >> 3; r < a.rows_cap; r += blockDim.x >> 3) {
    float v = 0.f;
    if (r < x.len) {
      const uint4 d4 = *reinterpret_cast<const uint4*>(dob + (int64_t)r * a.d + (lane & 7) * 8);
      const uint4 o4 = *reinterpret_cast<const uint4*>(ob + (int64_t)r * a.d + (lane & 7) * 8);
      const uint32_t dw[4] = {d4.x, d4.y, d4.z, d4.w}, ow[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&dw[i]));
        const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ow[i]));
        v += f.x * h.x + f.y * h.y;
      }
    }
    // the eight lanes of a row agree on r, so whole groups leave the loop together
    const uint32_t group = 0xFFu << (lane & 24);
    v += __shfl_xor_sync(group, v, 1);
    v += __shfl_xor_sync(group, v, 2);
    v += __shfl_xor_sync(group, v, 4);
    if ((lane & 7) == 0) {
      s_delta[r] = v;
      s_lse[r] = r < x.len ? a.lse[(int64_t)x.h * a.T + x.row0 + r] : INFINITY;
    }
  }
  flash_loads_done();
  bf16* dq = a.dqkv + x.row0 * ld3 + x.h * DH;
  float2 cs[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  // ---- 16 query rows at a time: dQ ----
  for (int r0 = warp * 16; r0 < x.len; r0 += nw * 16) {
    const int rows = min(16, x.len - r0);
    uint32_t qa[4][4], da[4][4];
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) {
      load_a_rows(Qs, LD, r0, kt * 16, lane, qa[kt][0], qa[kt][1], qa[kt][2], qa[kt][3]);
      load_a_rows(dOs, LD, r0, kt * 16, lane, da[kt][0], da[kt][1], da[kt][2], da[kt][3]);
    }
    const float e0 = s_lse[r0 + g], e1 = s_lse[r0 + g + 8], t0 = s_delta[r0 + g], t1 = s_delta[r0 + g + 8];
    float o[DH / 8][4];
#pragma unroll
    for (int nt = 0; nt < DH / 8; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
    const int kend = CAUSAL ? min(x.len, r0 + 16) : x.len;
    for (int k0 = 0; k0 < kend; k0 += 32) {
      float p[4][4], dp[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) p[nt][e] = dp[nt][e] = 0.f;
#pragma unroll
      for (int nt = 0; nt < 4; nt += 2) {
        if (k0 + nt * 8 < kend) {
#pragma unroll
          for (int kt = 0; kt < 4; ++kt) {
            uint32_t b0, b1, b2, b3;
            load_b_rows(Ks, LD, k0 + nt * 8, kt * 16, lane, b0, b1, b2, b3);
            mma16816(p[nt], qa[kt][0], qa[kt][1], qa[kt][2], qa[kt][3], b0, b1);
            mma16816(p[nt + 1], qa[kt][0], qa[kt][1], qa[kt][2], qa[kt][3], b2, b3);
            load_b_rows(Vs, LD, k0 + nt * 8, kt * 16, lane, b0, b1, b2, b3);
            mma16816(dp[nt], da[kt][0], da[kt][1], da[kt][2], da[kt][3], b0, b1);
            mma16816(dp[nt + 1], da[kt][0], da[kt][1], da[kt][2], da[kt][3], b2, b3);
          }
        }
      }
      const bool edge = k0 + 32 > x.len || (CAUSAL && k0 + 31 > r0);
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float pr = fast_exp2(fmaf(p[nt][e], a.c, -(e < 2 ? e0 : e1)));
          if (edge) {
            const int j = k0 + nt * 8 + 2 * q + (e & 1);
            if (j >= x.len || (CAUSAL && j > r0 + g + (e < 2 ? 0 : 8))) pr = 0.f;
          }
          dp[nt][e] = pr * (dp[nt][e] - (e < 2 ? t0 : t1)) * a.scale;
        }
#pragma unroll
      for (int kt = 0; kt < 2; ++kt) {
        if (k0 + kt * 16 < kend) {
          const uint32_t a0 = pack2(dp[2 * kt][0], dp[2 * kt][1]), a1 = pack2(dp[2 * kt][2], dp[2 * kt][3]);
          const uint32_t a2 = pack2(dp[2 * kt + 1][0], dp[2 * kt + 1][1]), a3 = pack2(dp[2 * kt + 1][2], dp[2 * kt + 1][3]);
#pragma unroll
          for (int nt = 0; nt < DH / 8; nt += 2) {
            uint32_t b0, b1, b2, b3;
            load_b_trans(Ks, LD, k0 + kt * 16, nt * 8, lane, b0, b1, b2, b3);
            mma16816(o[nt], a0, a1, a2, a3, b0, b1);
            mma16816(o[nt + 1], a0, a1, a2, a3, b2, b3);
          }
        }
      }
    }
    flash_store(o, stage, rows, dq + (int64_t)r0 * ld3, ld3, lane);
    if (a.colpart) flash_colsum(stage, rows, lane, cs[0]);
  }
  // ---- 16 key rows at a time: dK, dV ----
  for (int j0 = warp * 16; j0 < x.len; j0 += nw * 16) {
    const int rows = min(16, x.len - j0);
    uint32_t ka[4][4], va[4][4];
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) {
      load_a_rows(Ks, LD, j0, kt * 16, lane, ka[kt][0], ka[kt][1], ka[kt][2], ka[kt][3]);
      load_a_rows(Vs, LD, j0, kt * 16, lane, va[kt][0], va[kt][1], va[kt][2], va[kt][3]);
    }
    float dk[DH / 8][4], dv[DH / 8][4];
#pragma unroll
    for (int nt = 0; nt < DH / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) dk[nt][e] = dv[nt][e] = 0.f;
    const int qbeg = CAUSAL ? (j0 & ~31) : 0;            // earlier queries see none of these keys
    for (int q0 = qbeg; q0 < x.len; q0 += 32) {
      float p[4][4], dp[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) p[nt][e] = dp[nt][e] = 0.f;
#pragma unroll
      for (int nt = 0; nt < 4; nt += 2) {
        if (q0 + nt * 8 < x.len) {
#pragma unroll
          for (int kt = 0; kt < 4; ++kt) {
            uint32_t b0, b1, b2, b3;
            load_b_rows(Qs, LD, q0 + nt * 8, kt * 16, lane, b0, b1, b2, b3);
            mma16816(p[nt], ka[kt][0], ka[kt][1], ka[kt][2], ka[kt][3], b0, b1);
            mma16816(p[nt + 1], ka[kt][0], ka[kt][1], ka[kt][2], ka[kt][3], b2, b3);
            load_b_rows(dOs, LD, q0 + nt * 8, kt * 16, lane, b0, b1, b2, b3);
            mma16816(dp[nt], va[kt][0], va[kt][1], va[kt][2], va[kt][3], b0, b1);
            mma16816(dp[nt + 1], va[kt][0], va[kt][1], va[kt][2], va[kt][3], b2, b3);
          }
        }
      }
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const int i = q0 + nt * 8 + 2 * q;               // this thread's two queries
        const float2 le = *reinterpret_cast<const float2*>(s_lse + i), de = *reinterpret_cast<const float2*>(s_delta + i);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float pr = fast_exp2(fmaf(p[nt][e], a.c, -((e & 1) ? le.y : le.x)));           // queries past the end: lse = +inf
          if (CAUSAL && j0 + g + (e < 2 ? 0 : 8) > i + (e & 1)) pr = 0.f;
          p[nt][e] = pr;
          dp[nt][e] = pr * (dp[nt][e] - ((e & 1) ? de.y : de.x)) * a.scale;
        }
      }
#pragma unroll
      for (int kt = 0; kt < 2; ++kt) {
        if (q0 + kt * 16 < x.len) {
          const uint32_t a0 = pack2(p[2 * kt][0], p[2 * kt][1]), a1 = pack2(p[2 * kt][2], p[2 * kt][3]);
          const uint32_t a2 = pack2(p[2 * kt + 1][0], p[2 * kt + 1][1]), a3 = pack2(p[2 * kt + 1][2], p[2 * kt + 1][3]);
          const uint32_t s0 = pack2(dp[2 * kt][0], dp[2 * kt][1]), s1 = pack2(dp[2 * kt][2], dp[2 * kt][3]);
          const uint32_t s2 = pack2(dp[2 * kt + 1][0], dp[2 * kt + 1][1]), s3 = pack2(dp[2 * kt + 1][2], dp[2 * kt + 1][3]);
#pragma unroll
          for (int nt = 0; nt < DH / 8; nt += 2) {
            uint32_t b0, b1, b2, b3;
            load_b_trans(dOs, LD, q0 + kt * 16, nt * 8, lane, b0, b1, b2, b3);
            mma16816(dv[nt], a0, a1, a2, a3, b0, b1);
            mma16816(dv[nt + 1], a0, a1, a2, a3, b2, b3);
            load_b_trans(Qs, LD, q0 + kt * 16, nt * 8, lane, b0, b1, b2, b3);
            mma16816(dk[nt], s0, s1, s2, s3, b0, b1);
            mma16816(dk[nt + 1], s0, s1, s2, s3, b2, b3);
          }
        }
      }
    }
    flash_store(dk, stage, rows, dq + (int64_t)j0 * ld3 + a.d, ld3, lane);
    if (a.colpart) flash_colsum(stage, rows, lane, cs[1]);
    flash_store(dv, stage, rows, dq + (int64_t)j0 * ld3 + 2 * a.d, ld3, lane);
    if (a.colpart) flash_colsum(stage, rows, lane, cs[2]);
  }
  if (a.colpart) {                                       // the warps' column sums, added in warp order
#pragma unroll
    for (int w = 0; w < 3; ++w) *reinterpret_cast<float2*>(s_col + (w * FL_BWD_WARPS + warp) * DH + 2 * lane) = cs[w];
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * DH; i += blockDim.x) {
      const int which = i / DH, col = i - which * DH;
      float v = 0.f;
      for (int w = 0; w < nw; ++w) v += s_col[(which * FL_BWD_WARPS + w) * DH + col];
      a.colpart[x.slot * ld3 + (int64_t)which * a.d + x.h * DH + col] = v;
    }
  }
}

// warps per block: the 16-row tiles of the longest sequence in as few equal rounds as `most` warps allow
int flash_warps(int S, int most) {
  const int tiles = ceil_div(S, 16), rounds = ceil_div(tiles, most);
  return ceil_div(tiles, rounds);
}
size_t flash_fwd_smem(int cap, int warps) { return ((size_t)2 * cap * LD + (size_t)warps * STAGE_ELEMS) * 2; }
size_t flash_bwd_smem(int cap, int warps) {
  return ((size_t)4 * cap * LD + (size_t)warps * STAGE_ELEMS) * 2 + (size_t)(2 * cap + 3 * FL_BWD_WARPS * DH) * 4;
}
FlashArgs flash_args(const void* qkv, int64_t rows, int S, int d, int n_heads, const int32_t* seq_len, const int32_t* seq_off,
                     const int32_t* seq_list) {
  FlashArgs a = {};
  a.qkv = (const bf16*)qkv;
  a.T = rows;
  a.S = S; a.d = d; a.H = n_heads;
  a.rows_cap = (S + 31) & ~31;
  a.scale = 1.f / sqrtf((float)DH);
  a.c = a.scale * 1.4426950408889634f;
  a.seq_len = seq_len; a.seq_off = seq_off; a.seq_list = seq_list;
  return a;
}

}  // namespace

// Which sequences: those whose padding to 128-row tensor-memory tiles costs more than the faster MMA of those tiles gains.
// One layer of about 54 000 rows of width 768, every key visible, these kernels against the tcgen05 ones (attn_tc.cu), us:
//   rows       80    96    100   112   128   147   160   176   192   224   256
//   forward    125   144   152   141   133   149   142   173   168   179   172
//     tcgen05  144   121   127   117   81    342   285   292   247   218   188
//   backward   394   407   525   492   480   505   486   531   517
//     tcgen05  290   251   251   229   207   877   814   774   722   655   610
// (Causal histories, forward: 120 and 142 at 80 rows, 144 and 122 at 96, 144 and 130 at 100.  The tcgen05 kernels gained since the
// line was drawn at 96 rows; at 81 to 96 they are ahead in a layer of this size, while whole passes over 128 texts of 82, 90 and
// 96 tokens take the same 1336, 1394 and 1442 us either way.)
bool attention_flash_forward_supported(int S, int d, int n_heads) {
  return n_heads > 0 && d == n_heads * DH && ((S > 64 && S <= 96) || (S > 128 && S <= 256));
}
bool attention_flash_backward_supported(int S, int d, int n_heads) {
  return n_heads > 0 && d == n_heads * DH && S > 128 && S <= 192;
}

gram_status attention_forward_flash(gram_ctx* ctx, const void* qkv, void* out, float* lse, int64_t rows, int64_t n_seq, int S, int d,
                                    int n_heads, int causal, const int32_t* seq_len, const int32_t* seq_off, const int32_t* seq_list,
                                    cudaStream_t st) {
  if (n_seq == 0) return GRAM_OK;
  FlashArgs a = flash_args(qkv, rows, S, d, n_heads, seq_len, seq_off, seq_list);
  a.out = (bf16*)out;
  a.lse = lse;
  const int warps = flash_warps(S, FL_MAX_WARPS);
  const size_t smem = flash_fwd_smem(a.rows_cap, warps);
  auto kern = causal ? attn_flash_fwd_kernel<true> : attn_flash_fwd_kernel<false>;
  GRAM_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flash_fwd_smem(256, FL_MAX_WARPS)));
  launch_chain(kern, (unsigned)(n_seq * n_heads), warps * 32, smem, st, a);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

// colpart: one row of column sums per sequence of the launch, or null
gram_status attention_backward_flash(gram_ctx* ctx, const void* qkv, const void* dctx, const void* octx, const float* lse, void* dqkv,
                                     float* colpart, int64_t rows, int64_t n_seq, int S, int d, int n_heads, int causal,
                                     const int32_t* seq_len, const int32_t* seq_off, const int32_t* seq_list, cudaStream_t st) {
  if (n_seq == 0) return GRAM_OK;
  if (!lse || !octx) return gram_set_error(ctx, "attention backward: the forward pass's output and row statistics are missing"), GRAM_ERR_ARG;
  FlashArgs a = flash_args(qkv, rows, S, d, n_heads, seq_len, seq_off, seq_list);
  a.lse = const_cast<float*>(lse);
  a.dctx = (const bf16*)dctx;
  a.octx = (const bf16*)octx;
  a.dqkv = (bf16*)dqkv;
  a.colpart = colpart;
  // up to 160 rows two blocks of five warps fit an SM; above, one block with a warp per 16-row tile (168 registers a
  // thread either way; six warps in two rounds took 725 us at 192 rows, twelve take 525)
  const bool two = S <= 160;
  const int warps = flash_warps(S, two ? 5 : FL_BWD_WARPS);
  const size_t smem = flash_bwd_smem(a.rows_cap, warps);
  auto kern = two ? (causal ? attn_flash_bwd_kernel<true, 5> : attn_flash_bwd_kernel<false, 5>)
                  : (causal ? attn_flash_bwd_kernel<true, FL_BWD_WARPS> : attn_flash_bwd_kernel<false, FL_BWD_WARPS>);
  GRAM_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flash_bwd_smem(192, FL_BWD_WARPS)));
  launch_chain(kern, (unsigned)(n_seq * n_heads), warps * 32, smem, st, a);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}
