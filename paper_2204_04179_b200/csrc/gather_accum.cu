// Stage 3 (gather encodings into sequence positions) and stage 4 (sum the per-position
// gradients of each item, Eq. 6; Multi-step: add them into the per-item table, Section 4.2).
// Both are HBM-bound: 128-bit accesses, a warp per row, several rows in flight per warp.
#include "gram_internal.h"
#include "tc_common.cuh"

#include <type_traits>

namespace {

// ---------------------------------------------------------------------------
// gather: E[p, :] = src[index[p], :]
// Algorithmic bytes: P*row written + (distinct rows)*row read + 4P index.
// ---------------------------------------------------------------------------
template <int ROWS>   // rows a warp keeps in flight
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint4* __restrict__ src, int64_t n_src_rows,
                                                          const int32_t* __restrict__ index, int64_t P, int nvec,
                                                          uint4* __restrict__ dst, int32_t* status) {
  if (!chain_begin()) return;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p0 = warp * ROWS; p0 < P; p0 += nwarps * ROWS) {
    int64_t row[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      int64_t p = p0 + r;
      int32_t i = (p < P) ? index[p] : 0;
      if (i < 0 || i >= n_src_rows) {
        gram_device_fail(status, GRAM_ERR_ID_RANGE);
        i = 0;
      }
      row[r] = i;
    }
    for (int c = lane; c < nvec; c += 32) {
      uint4 v[ROWS];
#pragma unroll
      for (int r = 0; r < ROWS; ++r) v[r] = __ldg(src + row[r] * nvec + c);
#pragma unroll
      for (int r = 0; r < ROWS; ++r)
        if (p0 + r < P) __stcs(dst + (p0 + r) * nvec + c, v[r]);
    }
  }
}

// rows whose byte length is not a multiple of 16: element-wise copy of 2- or 4-byte elements
template <typename T>
__global__ void gather_scalar_kernel(const T* __restrict__ src, int64_t n_src_rows, const int32_t* __restrict__ index,
                                     int64_t P, int d, T* __restrict__ dst, int32_t* status) {
  if (!chain_begin()) return;
  const int64_t n = P * d;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = k / d;
    int c = (int)(k - p * d);
    int32_t i = index[p];
    if (i < 0 || i >= n_src_rows) {
      gram_device_fail(status, GRAM_ERR_ID_RANGE);
      i = 0;
    }
    dst[k] = src[(int64_t)i * d + c];
  }
}

// dst[p, :] (fp32) = src[index[p], :] (bf16): the Multi-step gather from a bf16 encoding cache, widened on the way so
// that the task module's fp32 input is written once.  A warp per row, 8 elements (16 bytes in, 32 out) per lane and step.
template <int ROWS>
__global__ void __launch_bounds__(256) gather_widen_kernel(const uint4* __restrict__ src, int64_t n_src_rows,
                                                           const int32_t* __restrict__ index, int64_t P, int nvec,
                                                           float4* __restrict__ dst, int32_t* status) {
  if (!chain_begin()) return;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p0 = warp * ROWS; p0 < P; p0 += nwarps * ROWS) {
    int64_t row[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      int64_t p = p0 + r;
      int32_t i = (p < P) ? index[p] : 0;
      if (i < 0 || i >= n_src_rows) {
        gram_device_fail(status, GRAM_ERR_ID_RANGE);
        i = 0;
      }
      row[r] = i;
    }
    for (int c = lane; c < nvec; c += 32) {
      uint4 v[ROWS];
#pragma unroll
      for (int r = 0; r < ROWS; ++r) v[r] = __ldg(src + row[r] * nvec + c);
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        if (p0 + r < P) {
          const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v[r].x));
          const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v[r].y));
          const float2 e = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v[r].z));
          const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v[r].w));
          float4* q = dst + ((p0 + r) * nvec + c) * 2;
          __stcs(q, make_float4(a.x, a.y, b.x, b.y));
          __stcs(q + 1, make_float4(e.x, e.y, f.x, f.y));
        }
      }
    }
  }
}

// out[r, :] = a[index[r], :] - b[index[r], :], or x[r, :] - that; a warp per row, 4 floats per lane and step
__global__ void __launch_bounds__(256) gather_diff_kernel(const float* __restrict__ a, const float* __restrict__ b,
                                                          int64_t n_src_rows, const int32_t* __restrict__ index, int64_t n,
                                                          int d, const float* __restrict__ x, float* __restrict__ out,
                                                          int32_t* status) {
  if (!chain_begin()) return;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const bool vec = (d & 3) == 0;
  for (int64_t r = warp; r < n; r += nwarps) {
    int32_t i = index[r];
    if (i < 0 || i >= n_src_rows) {
      gram_device_fail(status, GRAM_ERR_ID_RANGE);
      i = 0;
    }
    const float* pa = a + (int64_t)i * d;
    const float* pb = b + (int64_t)i * d;
    const float* px = x ? x + r * d : nullptr;
    float* po = out + r * d;
    if (vec) {
      for (int c = lane * 4; c < d; c += 128) {
        const float4 va = *reinterpret_cast<const float4*>(pa + c), vb = *reinterpret_cast<const float4*>(pb + c);
        float4 v = make_float4(va.x - vb.x, va.y - vb.y, va.z - vb.z, va.w - vb.w);
        if (px) {
          const float4 vx = *reinterpret_cast<const float4*>(px + c);
          v = make_float4(vx.x - v.x, vx.y - v.y, vx.z - v.z, vx.w - v.w);
        }
        *reinterpret_cast<float4*>(po + c) = v;
      }
    } else {
      for (int c = lane; c < d; c += 32) {
        const float v = pa[c] - pb[c];
        po[c] = px ? px[c] - v : v;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// segmented sum.  The sorted order j in [0, P) is cut into nchunks equal chunks of R rows; the
// columns into slabs of VPL*128 floats.  One warp owns one (chunk, slab): it walks its rows in
// order, adding into registers, and closes a sum whenever the item changes.
//   - an item whose rows all lie inside the chunk is written to its output row directly;
//   - the item that entered the chunk from the left leaves its part in partial[chunk][0];
//   - the item that leaves the chunk to the right leaves its part in partial[chunk][1].
// A second launch adds, for every item that spans chunks, partial[first][1] and the following
// chunks' partial[c][0] in a fixed association (eight interleaved ascending runs, then their sum).  The order of additions depends only
// on (P, U, seg_off), never on scheduling: repeated runs are bit-identical.
// Algorithmic bytes: 4*P*d read + 4*U*d written + 4P (perm) + 4(U+1) (seg_off).
// ---------------------------------------------------------------------------
// largest u in [0, U) with seg_off[u] <= j, found by the whole warp: every lane probes one of 32 evenly spaced
// entries per round, so U = 10^6 takes four dependent loads instead of twenty.  All 32 lanes must call it.
__device__ __forceinline__ int32_t find_segment(const int32_t* __restrict__ seg_off, int32_t U, int64_t j, int lane) {
  int32_t lo = 0, n = U;                       // the answer lies in [lo, lo + n) and seg_off[lo] <= j
  while (n > 1) {
    const int32_t step = (n + 31) >> 5;
    const int32_t idx = lo + lane * step;
    const bool ok = (lane * step < n) && (seg_off[idx] <= j);
    const unsigned m = __ballot_sync(0xffffffffu, ok) | 1u;
    const int k = 31 - __clz(m);
    n = min(step, n - k * step);
    lo += k * step;
  }
  return lo;
}

template <int VPL>
__device__ __forceinline__ void store_row(float* __restrict__ out, int64_t row, int d, int col0, int lane,
                                          const float4 (&acc)[VPL], bool add) {
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    int c = col0 + (v * 32 + lane) * 4;
    if (c < d) {
      float4* q = reinterpret_cast<float4*>(out + row * d + c);
      float4 a = acc[v];
      if (add) {
        float4 o = *q;
        a.x += o.x; a.y += o.y; a.z += o.z; a.w += o.w;
      }
      *q = a;
    }
  }
}

// The items of a chunk in ascending order: where each ends and the output row it goes to.
// AHEAD, for sums that are added to rows picked by `rows`: lane l holds those of item `base` + l, the next 32 are on their way, so an
// item costs shuffles.  With loads of its own, one after the other (its row, the row's old values, the end of the next item), a chunk of
// short items waited for each: 10^6 positions over 10^5 items into a table of 768 columns 882 us, 636 with the old values fetched when
// the item begins; 25 600 over 10^4 58 and 35.  Plain sums have the one load of the next end, and keep it: there the shuffles cost
// more (10^6 x 128 over 3 10^5 items 158 us, 174 ahead).  All lanes of a warp call.
template <bool AHEAD> struct SegItems {
  const int32_t* seg_off;
  const int32_t* rows;
  int32_t U, base, u, off, row, off_next, row_next;      // u: the current item
  int lane;
  __device__ __forceinline__ void fetch(int32_t first, int32_t& o, int32_t& r) const {
    const int32_t i = first + lane;
    o = i < U ? seg_off[i + 1] : INT32_MAX;
    r = i < U ? (rows ? rows[i] : i) : 0;
  }
  __device__ __forceinline__ SegItems(const int32_t* so, const int32_t* rw, int32_t n, int32_t first, int l)
      : seg_off(so), rows(rw), U(n), base(first), u(first), lane(l) {
    if (AHEAD) {
      fetch(first, off, row);
      fetch(first + 32, off_next, row_next);
    }
  }
  __device__ __forceinline__ void advance() {
    ++u;
    if (AHEAD && u - base == 32) {
      base = u;
      off = off_next;
      row = row_next;
      fetch(base + 32, off_next, row_next);
    }
  }
  __device__ __forceinline__ int32_t end() const { return AHEAD ? __shfl_sync(0xffffffffu, off, u - base) : seg_off[u + 1]; }
  __device__ __forceinline__ int32_t out_row() const { return AHEAD ? __shfl_sync(0xffffffffu, row, u - base) : (rows ? rows[u] : u); }
};
// what a row of sums is added to, fetched when its item begins
template <int VPL>
__device__ __forceinline__ void load_old(const float* __restrict__ out, int64_t row, int d, int col0, int lane, float4 (&old)[VPL]) {
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int c = col0 + (v * 32 + lane) * 4;
    old[v] = c < d ? *reinterpret_cast<const float4*>(out + row * d + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
template <int VPL>
__device__ __forceinline__ void add_old(float4 (&acc)[VPL], const float4 (&old)[VPL]) {
#pragma unroll
  for (int v = 0; v < VPL; ++v) { acc[v].x += old[v].x; acc[v].y += old[v].y; acc[v].z += old[v].z; acc[v].w += old[v].w; }
}

// ADD: out[row] += the sum
template <int VPL, int UNROLL, bool ADD>
__global__ void __launch_bounds__(256) segsum_chunks_kernel(const float* __restrict__ in, const int32_t* __restrict__ perm,
                                                            const int32_t* __restrict__ seg_off, int64_t P, int32_t U,
                                                            int d, int64_t R, int nchunks, int nslabs,
                                                            const int32_t* __restrict__ rows,
                                                            float* __restrict__ out, float* __restrict__ partial,
                                                            int2* __restrict__ span, int32_t* status,
                                                            const int32_t* __restrict__ d_U,
                                                            const int32_t* __restrict__ gate) {
  if (!chain_begin()) return;
  if (d_U) U = *d_U;            // the number of items may live on the device
  if (U <= 0) return;
  if (gate && *gate) return;    // an earlier kernel of the step reported an error: leave the accumulated rows alone
  const int lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= (int64_t)nchunks * nslabs) return;
  const int chunk = (int)(w / nslabs), slab = (int)(w - (int64_t)chunk * nslabs);
  const int col0 = slab * (VPL * 128);
  const int64_t c0 = (int64_t)chunk * R, c1 = min(c0 + R, P);
  if (c0 >= c1) return;

  // the current item's ends, in the width that the row loop is faster with: 300 000 x 256 65.8 us with 32 bits and 61.2 with 64, 1600 x 768 7.3
  // and 6.6; with half the columns a warp 300 000 x 64 42.0 and 43.2, 3200 x 64 6.4 and 6.6
  typedef typename std::conditional<VPL == 2, int64_t, int32_t>::type Bound;
  SegItems<ADD> it(seg_off, rows, U, find_segment(seg_off, U, c0, lane), lane);
  Bound seg_begin = seg_off[it.u], seg_end = it.end();
  float4 acc[VPL], old[ADD ? VPL : 1];
#pragma unroll
  for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (ADD) load_old<VPL>(out, it.out_row(), d, col0, lane, old);

  for (int64_t j0 = c0; j0 < c1; j0 += 32) {
    const int nrow = (int)min((int64_t)32, c1 - j0);
    int32_t my = (lane < nrow) ? perm[j0 + lane] : 0;
    if ((uint32_t)my >= (uint32_t)P) {       // a position outside the batch: record it, read row 0 instead
      gram_device_fail(status, GRAM_ERR_ID_RANGE);
      my = 0;
    }
    for (int b = 0; b < nrow; b += UNROLL) {
      float4 x[UNROLL][VPL];
#pragma unroll
      for (int r = 0; r < UNROLL; ++r) {
        const int32_t p = __shfl_sync(0xffffffffu, my, (b + r) & 31);
        const bool live = (b + r) < nrow;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          int c = col0 + (v * 32 + lane) * 4;
          x[r][v] = (live && c < d) ? __ldcs(reinterpret_cast<const float4*>(in + (int64_t)p * d + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
#pragma unroll
      for (int r = 0; r < UNROLL; ++r) {
        const int64_t j = j0 + b + r;
        if (j < c1) {
          while (j == seg_end && it.u + 1 < U) {   // the item is complete (its end lies inside this chunk)
            if (seg_begin >= c0) {
              if constexpr (ADD) add_old<VPL>(acc, old);
              store_row<VPL>(out, it.out_row(), d, col0, lane, acc, false);
            } else store_row<VPL>(partial, (int64_t)chunk * 2 + 0, d, col0, lane, acc, false);
            it.advance();
            seg_begin = seg_end;
            seg_end = it.end();
#pragma unroll
            for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (ADD) load_old<VPL>(out, it.out_row(), d, col0, lane, old);
          }
#pragma unroll
          for (int v = 0; v < VPL; ++v) {
            acc[v].x += x[r][v].x; acc[v].y += x[r][v].y; acc[v].z += x[r][v].z; acc[v].w += x[r][v].w;
          }
        }
      }
    }
  }
  // the item still open at the end of the chunk
  int2 sp = make_int2(-1, 0);
  if (seg_end <= c1) {             // it ends exactly at the chunk end
    if (seg_begin >= c0) {
      if constexpr (ADD) add_old<VPL>(acc, old);
      store_row<VPL>(out, it.out_row(), d, col0, lane, acc, false);
    } else store_row<VPL>(partial, (int64_t)chunk * 2 + 0, d, col0, lane, acc, false);
  } else {                         // it continues to the right
    store_row<VPL>(partial, (int64_t)chunk * 2 + (seg_begin >= c0 ? 1 : 0), d, col0, lane, acc, false);
    if (seg_begin >= c0) sp = make_int2(it.u, (int)((seg_end - 1) / R));      // it starts here: the fix-up adds its parts
  }
  if (slab == 0 && lane == 0) span[chunk] = sp;   // (item, last chunk it reaches), or -1: nothing to fix up from here
}

// The same walk for fp32 rows of 516 to 1024 columns with one warp per chunk (all columns): the rows arrive as bulk copies
// in a ring of `stages` slots per warp, so a warp has that many rows on their way while it adds, instead of none between
// two batches of register loads.  Sums, partial sums and spans as above, bit for bit (a chunk's rows are added in the same
// order).  Through registers / this way, us: 25 600 rows of 768 36 / 32, 150 000 107 / 104, 10^6 606 / 586; of 1024 41 / 41,
// 138 / 130.  Narrower rows (512: 75 / 80 at 150 000; 256: 45 / 50) and short calls (3000 rows: 12 / 15) stay with registers:
// a bulk copy of 2 KB or less costs its issue.
constexpr int SEG_WARPS = 8, SEG_STAGES_MAX = 8;
constexpr int kSegRingMin = 512;                 // columns, more than
constexpr int64_t kSegRingRows = 20000;          // positions, at least
constexpr int64_t kSegRingBytes = 110 * 1024;    // shared memory of a block: two per SM
template <int NQ, bool ADD>
__global__ void __launch_bounds__(32 * SEG_WARPS, 2) segsum_ring_kernel(const float* __restrict__ in, const int32_t* __restrict__ perm,
                                                                    const int32_t* __restrict__ seg_off, int64_t P, int32_t U, int d,
                                                                    int64_t R, int nchunks, int stages, int32_t ring_rows,
                                                                    const int32_t* __restrict__ rows,
                                                                    float* __restrict__ out, float* __restrict__ partial,
                                                                    int2* __restrict__ span, int32_t* status,
                                                                    const int32_t* __restrict__ d_U, const int32_t* __restrict__ gate) {
  if (!chain_begin()) return;
  extern __shared__ __align__(16) float seg_ring[];
  __shared__ __align__(8) uint64_t bars[SEG_WARPS * SEG_STAGES_MAX];
  __shared__ int abort_flag;
  if (d_U) U = *d_U;
  if (U <= 0) return;
  if (gate && *gate) return;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int chunk = blockIdx.x * SEG_WARPS + wib;
  float* ring = seg_ring + (size_t)wib * stages * d;
  const uint32_t bar0 = tc::smem_u32(bars + wib * SEG_STAGES_MAX), ring0 = tc::smem_u32(ring), row_bytes = (uint32_t)d * 4u;
  if (threadIdx.x == 0) abort_flag = 0;
  if (lane == 0) {
    for (int s = 0; s < stages; ++s) tc::mbar_init(bar0 + 8u * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int64_t c0 = (int64_t)chunk * R, c1 = min(c0 + R, P);
  if (chunk >= nchunks || c0 >= c1) return;
  auto fetch_perm = [&](int64_t j0) -> int32_t {             // positions j0 + lane of the sorted order
    int32_t p = 0;
    if (j0 + lane < c1) {
      p = perm[j0 + lane];
      if ((uint32_t)p >= (uint32_t)P) {                      // a position outside the batch: record it, read row 0 instead
        gram_device_fail(status, GRAM_ERR_ID_RANGE);
        p = 0;
      }
    }
    return p;
  };
  auto request = [&](int32_t p, int s) {
    tc::mbar_expect_tx(bar0 + 8u * s, row_bytes);
    tc::bulk_load(ring0 + (uint32_t)s * row_bytes, in + (int64_t)p * d, row_bytes, bar0 + 8u * s);
  };
  int32_t cur = fetch_perm(c0), nxt = fetch_perm(c0 + 32);
  for (int k = 0; k < stages; ++k) {                          // stages <= 8: inside the first window
    const int32_t p = __shfl_sync(0xffffffffu, cur, k);
    if (lane == 0 && c0 + k < c1) request(p, k);
  }
  SegItems<ADD> it(seg_off, rows, U, find_segment(seg_off, U, c0, lane), lane);
  int32_t seg_begin = seg_off[it.u], seg_end = it.end();
  float4 acc[NQ], old[ADD ? NQ : 1];
#pragma unroll
  for (int v = 0; v < NQ; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (ADD) load_old<NQ>(out, it.out_row(), d, 0, lane, old);
  int s = 0;
  uint32_t parity = 0;
  bool failed = false;
  for (int64_t j = c0; j < c1; ++j) {
    if (!__all_sync(0xffffffffu, ring_rows-- > 0 && tc::mbar_wait(bar0 + 8u * s, parity, (volatile int*)&abort_flag))) { failed = true; break; }
    float4 x[NQ];
    const float* row = ring + (size_t)s * d;
#pragma unroll
    for (int v = 0; v < NQ; ++v) {
      const int c = (v * 32 + lane) * 4;
      x[v] = c < d ? *reinterpret_cast<const float4*>(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int at = (int)((j - c0) & 31) + stages;             // the row `stages` places on, in this window or the next
    const int32_t pa = __shfl_sync(0xffffffffu, cur, at & 31), pb = __shfl_sync(0xffffffffu, nxt, at & 31);
    __syncwarp();                                              // every lane has read the slot
    if (lane == 0 && j + stages < c1) request(at < 32 ? pa : pb, s);
    if (((j - c0) & 31) == 31) {
      cur = nxt;
      nxt = fetch_perm(j + 33);
    }
    if (++s == stages) { s = 0; parity ^= 1u; }
    while (j == seg_end && it.u + 1 < U) {                     // the item is complete (its end lies inside this chunk)
      if (seg_begin >= c0) {
        if constexpr (ADD) add_old<NQ>(acc, old);
        store_row<NQ>(out, it.out_row(), d, 0, lane, acc, false);
      } else store_row<NQ>(partial, (int64_t)chunk * 2 + 0, d, 0, lane, acc, false);
      it.advance();
      seg_begin = seg_end;
      seg_end = it.end();
#pragma unroll
      for (int v = 0; v < NQ; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (ADD) load_old<NQ>(out, it.out_row(), d, 0, lane, old);
    }
#pragma unroll
    for (int v = 0; v < NQ; ++v) { acc[v].x += x[v].x; acc[v].y += x[v].y; acc[v].z += x[v].z; acc[v].w += x[v].w; }
  }
  if (failed) {
    if (lane == 0) {
      abort_flag = 1;
      span[chunk] = make_int2(-1, 0);                          // not what an earlier call left there: the fix-up reads it
      gram_device_fail(status, GRAM_ERR_TIMEOUT);
      const uint64_t t0 = clock64();                           // let the copies that were issued end (bounded)
      while (clock64() - t0 < tc::WAIT_LIMIT_CYCLES / 64) {}
    }
    __syncwarp();
    return;
  }
  int2 sp = make_int2(-1, 0);
  if (seg_end <= c1) {             // the item still open ends exactly at the chunk end
    if (seg_begin >= c0) {
      if constexpr (ADD) add_old<NQ>(acc, old);
      store_row<NQ>(out, it.out_row(), d, 0, lane, acc, false);
    } else store_row<NQ>(partial, (int64_t)chunk * 2 + 0, d, 0, lane, acc, false);
  } else {                         // it continues to the right
    store_row<NQ>(partial, (int64_t)chunk * 2 + (seg_begin >= c0 ? 1 : 0), d, 0, lane, acc, false);
    if (seg_begin >= c0) sp = make_int2(it.u, (int)((seg_end - 1) / R));
  }
  if (lane == 0) span[chunk] = sp;
}

// A warp per (chunk, slab): if an item starts in this chunk and runs past its end, add its parts.  Eight runs: run w adds the
// following chunks' parts number w, w + 8, ... (ascending), run 0 starts from this chunk's own part, and the eight sums are
// added in ascending w: a fixed association, whatever the schedule.  With up to eight parts a run is one part, so the warp
// simply adds them in order; an item that reaches farther is summed by the whole block, a run per warp.
// Nearly every chunk has an item that runs into the next one, and what that takes is the chain item, parts, store: with a block of
// eight warps for each of them 34 us at 10^6 positions of 768 columns, a twelfth of the blocks on the chip at a time; 14 this way.
// While a block for each of them fits the chip at once (eight blocks an SM) it has one all the same (PER = 1), and all eight warps take
// the item: one over more than nine parts then waits for no others.  us with a block each and with eight to a block: 912 positions of 64
// columns 2.28 and 2.85 (Zipf 1.1; 2.23 and 2.11 at 0.8, where no item is that long), 3200 x 64 2.50 and 3.10, 1600 x 768 3.06 and 3.51,
// 12 800 x 128 (800 pairs) 3.46 and 3.66, into a table 3.73 and 4.19; 6400 x 768 (1200 pairs) 4.13 and 3.81, 9000 x 768 4.98 and 4.11.
constexpr int FIX_RUNS = 8;
constexpr int64_t kFixAlone = 8 * kNumSMs;
template <int VPL, int PER>
__global__ void __launch_bounds__(32 * FIX_RUNS) segsum_fixup_kernel(const int32_t* __restrict__ seg_off, int64_t P, int32_t U,
                                                           int d, int64_t R, int nchunks, int nslabs,
                                                           const int32_t* __restrict__ rows, int add,
                                                           float* __restrict__ out, const float* __restrict__ partial,
                                                           const int2* __restrict__ span, const int32_t* __restrict__ d_U,
                                                           const int32_t* __restrict__ gate) {
  if (!chain_begin()) return;
  __shared__ float4 red[FIX_RUNS][VPL][32];
  __shared__ int2 far[FIX_RUNS];                     // (item, last chunk) of the warps whose item takes the block, else last = -1
  if (d_U) U = *d_U;
  if (U <= 0) return;
  if (gate && *gate) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int chunk0 = (int)(blockIdx.x / nslabs) * PER, slab = (int)(blockIdx.x % nslabs);
  const int col0 = slab * (VPL * 128);
  // part of item chunk c: the own part of the chunk it starts in (which = 1), what it left in a later one (which = 0)
  auto part = [&](int c, int which, float4 (&x)[VPL]) {
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int cc = col0 + (v * 32 + lane) * 4;
      x[v] = cc < d ? *reinterpret_cast<const float4*>(partial + ((int64_t)c * 2 + which) * d + cc) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto plus = [](float4 (&a)[VPL], const float4 (&x)[VPL]) {
#pragma unroll
    for (int v = 0; v < VPL; ++v) { a[v].x += x[v].x; a[v].y += x[v].y; a[v].z += x[v].z; a[v].w += x[v].w; }
  };
  constexpr bool alone = PER == 1;                   // all warps look at the same chunk
  const int chunk = chunk0 + (alone ? 0 : w);
  const int64_t c0 = (int64_t)chunk * R, c1 = min(c0 + R, P);
  int2 sp = make_int2(-1, -1);
  if (chunk < nchunks && c0 < c1 && c1 < P) sp = span[chunk];       // left by the first launch
  const bool mine = sp.x >= 0 && sp.x < U;           // else no item starts here and runs on (same for the whole warp)
  const int last = mine ? min(sp.y, nchunks - 1) : -1;
  const bool block_wide = mine && (alone || last - chunk > FIX_RUNS);
  if (!alone && mine && !block_wide) {
    float4 acc[VPL];
    part(chunk, 1, acc);
#pragma unroll
    for (int k0 = 0; k0 < FIX_RUNS; k0 += 4) {       // four parts on their way
      if (chunk + 1 + k0 > last) break;
      float4 x[4][VPL];
#pragma unroll
      for (int k = 0; k < 4; ++k) part(min(chunk + 1 + k0 + k, last), 0, x[k]);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (chunk + 1 + k0 + k <= last) plus(acc, x[k]);
    }
    store_row<VPL>(out, rows ? rows[sp.x] : sp.x, d, col0, lane, acc, add != 0);
  }
  if (!alone) {
    if (lane == 0) far[w] = make_int2(sp.x, block_wide ? last : -1);
    if (!__syncthreads_or(block_wide)) return;
  }
  for (int f = 0; f < PER; ++f) {
    const int2 it = alone ? make_int2(sp.x, block_wide ? last : -1) : far[f];
    if (it.y < 0) continue;                          // the same for the whole block
    const int first = chunk0 + f;
    float4 acc[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (w == 0) part(first, 1, acc);
    constexpr int AHEAD = alone ? 4 : 8;             // parts on their way per warp
    for (int c = first + 1 + w; c <= it.y; c += AHEAD * FIX_RUNS) {
      float4 x[AHEAD][VPL];
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) part(min(c + FIX_RUNS * k, it.y), 0, x[k]);
#pragma unroll
      for (int k = 0; k < AHEAD; ++k)
        if (c + FIX_RUNS * k <= it.y) plus(acc, x[k]);
    }
#pragma unroll
    for (int v = 0; v < VPL; ++v) red[w][v][lane] = acc[v];
    __syncthreads();
    if (w == 0) {
#pragma unroll
      for (int k = 1; k < FIX_RUNS; ++k) {
        float4 y[VPL];
#pragma unroll
        for (int v = 0; v < VPL; ++v) y[v] = red[k][v][lane];
        plus(acc, y);
      }
      store_row<VPL>(out, rows ? rows[it.x] : it.x, d, col0, lane, acc, add != 0);
    }
    __syncthreads();
  }
}

// d_U (may be null): the number of items lives on the device.  count (may be null): one word that counts the set
// bits (integer adds: the total does not depend on their order).  gated: nothing is marked once the status word is set.
__global__ void touched_mark_kernel(const int32_t* __restrict__ unique, int32_t U, const int32_t* __restrict__ d_U,
                                    int32_t n_items, uint32_t* __restrict__ bits, int32_t* __restrict__ count,
                                    int32_t* status, int gated) {
  if (!chain_begin()) return;
  if (d_U) U = *d_U;
  if (gated && *status) return;
  for (int32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < U; u += gridDim.x * blockDim.x) {
    const int32_t i = unique[u];
    if (i < 0 || i >= n_items) {
      gram_device_fail(status, GRAM_ERR_ID_RANGE);
      continue;
    }
    const uint32_t bit = 1u << (i & 31);
    const uint32_t old = atomicOr(&bits[i >> 5], bit);
    if (count && !(old & bit)) atomicAdd(count, 1);
  }
}

// ascending list of set bits, one block
__global__ void __launch_bounds__(1024) touched_list_kernel(const uint32_t* __restrict__ bits, int32_t n_items,
                                                            int32_t* __restrict__ list, int32_t* __restrict__ count) {
  if (!chain_begin()) return;
  __shared__ int32_t sw[33];
  const int nwords = (n_items + 31) >> 5;
  const int per = (nwords + 1023) / 1024;
  const int w0 = threadIdx.x * per, w1 = min(w0 + per, nwords);
  int32_t c = 0;
  for (int w = w0; w < w1; ++w) {
    uint32_t b = bits[w];
    if (w == nwords - 1 && (n_items & 31)) b &= (1u << (n_items & 31)) - 1u;
    c += __popc(b);
  }
  // exclusive scan over the 1024 threads
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t incl = c;
  for (int o = 1; o < 32; o <<= 1) {
    int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) sw[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int32_t x = sw[lane], xi = x;
    for (int o = 1; o < 32; o <<= 1) {
      int32_t t = __shfl_up_sync(0xffffffffu, xi, o);
      if (lane >= o) xi += t;
    }
    sw[lane] = xi - x;
    if (lane == 31) sw[32] = xi;
  }
  __syncthreads();
  int32_t pos = sw[warp] + incl - c;
  for (int w = w0; w < w1; ++w) {
    uint32_t b = bits[w];
    if (w == nwords - 1 && (n_items & 31)) b &= (1u << (n_items & 31)) - 1u;
    while (b) {
      int bit = __ffs(b) - 1;
      list[pos++] = w * 32 + bit;
      b &= b - 1;
    }
  }
  if (threadIdx.x == 0) *count = sw[32];
}

}  // namespace

gram_status gather_launch(gram_ctx* ctx, const void* d_src, int64_t n_src_rows, const int32_t* d_index, int64_t P,
                          int32_t d, int elem_bytes, void* d_E, cudaStream_t st) {
  if (P < 0 || d <= 0 || n_src_rows < 0 || (elem_bytes != 2 && elem_bytes != 4))
    return gram_set_error(ctx, "gram_gather: bad argument"), GRAM_ERR_ARG;
  if (P == 0) return GRAM_OK;
  if (!d_src || !d_index || !d_E || n_src_rows == 0)
    return gram_set_error(ctx, "gram_gather: null buffer"), GRAM_ERR_ARG;
  int32_t* status = gram_status_word(ctx);
  const int64_t row_bytes = (int64_t)d * elem_bytes;
  ProfScope prof(ctx, GRAM_K_GATHER, (double)row_bytes * (double)(P + (n_src_rows < P ? n_src_rows : P)) + 4.0 * P, 1, st);
  const bool vec_ok = (row_bytes % 16 == 0) && ((uintptr_t)d_src % 16 == 0) && ((uintptr_t)d_E % 16 == 0);
  if (vec_ok) {
    const int nvec = (int)(row_bytes / 16);
    constexpr int ROWS = 4;
    int64_t warps = ceil_div64(P, ROWS);
    int blocks = (int)ceil_div64(warps, 8);
    const int cap = kNumSMs * 8;
    if (blocks > cap) blocks = cap;
    launch_chain(gather_rows_kernel<ROWS>, blocks, 256, 0, st, (const uint4*)d_src, n_src_rows, d_index, P, nvec, (uint4*)d_E,
                                                     status);
  } else {
    int64_t n = P * d;
    int blocks = (int)ceil_div64(n, 256);
    if (blocks > kNumSMs * 16) blocks = kNumSMs * 16;
    if (elem_bytes == 4)
      launch_chain(gather_scalar_kernel<float>, blocks, 256, 0, st, (const float*)d_src, n_src_rows, d_index, P, d, (float*)d_E, status);
    else
      launch_chain(gather_scalar_kernel<bf16>, blocks, 256, 0, st, (const bf16*)d_src, n_src_rows, d_index, P, d, (bf16*)d_E, status);
  }
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

gram_status gather_widen_launch(gram_ctx* ctx, const void* d_src_bf16, int64_t n_src_rows, const int32_t* d_index, int64_t P,
                                int32_t d, float* d_E, cudaStream_t st) {
  if (P < 0 || d <= 0 || n_src_rows <= 0 || (d % 8) || ((uintptr_t)d_src_bf16 % 16) || ((uintptr_t)d_E % 16))
    return gram_set_error(ctx, "widening gather: bad argument (rows of a multiple of 8 elements, 16-byte aligned)"), GRAM_ERR_ARG;
  if (P == 0) return GRAM_OK;
  if (!d_src_bf16 || !d_index || !d_E) return gram_set_error(ctx, "widening gather: null buffer"), GRAM_ERR_ARG;
  ProfScope prof(ctx, GRAM_K_GATHER, 4.0 * (double)d * (double)P + 2.0 * (double)d * (double)(n_src_rows < P ? n_src_rows : P) + 4.0 * P, 1, st);
  constexpr int ROWS = 4;
  int blocks = (int)ceil_div64(ceil_div64(P, ROWS), 8);
  if (blocks > kNumSMs * 8) blocks = kNumSMs * 8;
  launch_chain(gather_widen_kernel<ROWS>, blocks, 256, 0, st, (const uint4*)d_src_bf16, n_src_rows, d_index, P, d / 8, (float4*)d_E,
                                                    gram_status_word(ctx));
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

gram_status gather_diff_launch(gram_ctx* ctx, const float* d_a, const float* d_b, int64_t n_src_rows, const int32_t* d_index,
                               int64_t n, int32_t d, const float* d_x, float* d_out, cudaStream_t st) {
  if (n < 0 || d <= 0 || n_src_rows <= 0 || (n > 0 && (!d_a || !d_b || !d_index || !d_out)))
    return gram_set_error(ctx, "gather of pseudo-targets: bad argument"), GRAM_ERR_ARG;
  if (n == 0) return GRAM_OK;
  ProfScope prof(ctx, GRAM_K_GATHER, (double)n * d * 4.0 * (d_x ? 4.0 : 3.0) + 4.0 * (double)n, 1, st);
  int blocks = (int)ceil_div64(n, 8);
  if (blocks > kNumSMs * 8) blocks = kNumSMs * 8;
  launch_chain(gather_diff_kernel, blocks, 256, 0, st, d_a, d_b, n_src_rows, d_index, n, d, d_x, d_out, gram_status_word(ctx));
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

template <int VPL>
static void segsum_run(const float* d_in, const int32_t* d_perm, const int32_t* d_seg_off, int64_t P, int32_t U, int32_t d,
                       int64_t R, int nchunks, const int32_t* d_rows, int add, float* d_out, float* partial, int2* span,
                       int32_t* status, const int32_t* d_U, cudaStream_t st, const int32_t* gate, int32_t ring_rows) {
  const int nslabs = ceil_div(d, VPL * 128);
  const int64_t warps = (int64_t)nchunks * nslabs;
  const int blocks = (int)ceil_div64(warps, 8);
  if (d > kSegRingMin && d <= 1024 && P >= kSegRingRows) {
    auto kern = d <= 768 ? (add ? segsum_ring_kernel<6, true> : segsum_ring_kernel<6, false>) : (add ? segsum_ring_kernel<8, true> : segsum_ring_kernel<8, false>);
    int stages = (int)(kSegRingBytes / ((int64_t)SEG_WARPS * d * 4));
    if (stages > SEG_STAGES_MAX) stages = SEG_STAGES_MAX;
    (void)cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSegRingBytes);
    launch_chain(kern, ceil_div(nchunks, SEG_WARPS), 32 * SEG_WARPS, (size_t)SEG_WARPS * stages * d * 4, st, d_in, d_perm,
                 d_seg_off, P, U, d, R, nchunks, stages, ring_rows, d_rows, d_out, partial, span, status, d_U, gate);
  } else {
    launch_chain(add ? segsum_chunks_kernel<VPL, 8, true> : segsum_chunks_kernel<VPL, 8, false>, blocks, 256, 0, st, d_in, d_perm, d_seg_off, P, U, d, R,
                 nchunks, nslabs, d_rows, d_out, partial, span, status, d_U, gate);
  }
  const int per_block = warps <= kFixAlone ? 1 : FIX_RUNS;
  if (nchunks > 1)
    launch_chain(per_block == 1 ? segsum_fixup_kernel<VPL, 1> : segsum_fixup_kernel<VPL, FIX_RUNS>, (unsigned)(ceil_div(nchunks, per_block) * nslabs),
                 32 * FIX_RUNS, 0, st, d_seg_off, P, U, d, R, nchunks, nslabs, d_rows, add, d_out, partial, span, d_U, gate);
}

gram_status accumulate_launch(gram_ctx* ctx, IndexWorkspace* ws, const float* d_in, const int32_t* d_perm,
                              const int32_t* d_seg_off, int64_t P, int32_t U, const int32_t* d_U, int32_t d,
                              const int32_t* d_rows, int add, float* d_out, cudaStream_t st, int gated) {
  if (P < 0 || U < 0 || d <= 0 || U > P) return gram_set_error(ctx, "gram_accumulate: bad argument"), GRAM_ERR_ARG;
  if (P == 0 || (U == 0 && !d_U)) return GRAM_OK;
  if (!d_in || !d_perm || !d_seg_off || !d_out) return gram_set_error(ctx, "gram_accumulate: null buffer"), GRAM_ERR_ARG;
  if (d % 4 != 0 || ((uintptr_t)d_in % 16) || ((uintptr_t)d_out % 16))
    return gram_set_error(ctx, "gram_accumulate: d must be a multiple of 4 and buffers 16-byte aligned"), GRAM_ERR_UNSUPPORTED;
  if (d > ws->d_max) return gram_set_error(ctx, "gram_accumulate: d=%d exceeds the context's d_max=%d", d, ws->d_max), GRAM_ERR_WORKSPACE;
  // chunks: at least 16 rows each, at most kAccMaxChunks
  int64_t nchunks = ceil_div64(P, 16);
  if (nchunks > kAccMaxChunks) nchunks = kAccMaxChunks;
  const int64_t R = ceil_div64(P, nchunks);
  nchunks = ceil_div64(P, R);
  int2* span = reinterpret_cast<int2*>(ws->partial + (size_t)kAccMaxChunks * 2 * (ws->d_max > 0 ? ws->d_max : 1));   // after the partial sums
  ProfScope prof(ctx, GRAM_K_ACCUMULATE, 4.0 * (double)P * d + 4.0 * (double)U * d + 4.0 * P + 4.0 * (U + 1),
                 nchunks > 1 ? 2 : 1, st);
  int32_t* sw = gram_status_word(ctx);
  const int32_t* gate = gated ? sw : nullptr;
  const int32_t ring_rows = gram_ring_rows(ctx);
  if (d >= 256) segsum_run<2>(d_in, d_perm, d_seg_off, P, U, d, R, (int)nchunks, d_rows, add, d_out, ws->partial, span, sw, d_U, st, gate, ring_rows);
  else segsum_run<1>(d_in, d_perm, d_seg_off, P, U, d, R, (int)nchunks, d_rows, add, d_out, ws->partial, span, sw, d_U, st, gate, ring_rows);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

gram_status touched_mark_launch(gram_ctx* ctx, const int32_t* d_unique, int32_t U, const int32_t* d_U, int32_t n_items,
                                uint32_t* d_bits, int32_t* d_count, int gated, cudaStream_t st) {
  if (U <= 0 && !d_U) return GRAM_OK;
  if (d_U) U = n_items;                              // upper bound for the launch shape
  ProfScope prof(ctx, GRAM_K_OTHER, 8.0 * U, 1, st);
  int blocks = ceil_div(U, 256);
  if (blocks > kNumSMs * 4) blocks = kNumSMs * 4;
  launch_chain(touched_mark_kernel, blocks, 256, 0, st, d_unique, U, d_U, n_items, d_bits, d_count, gram_status_word(ctx), gated);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

gram_status touched_list_launch(gram_ctx* ctx, const uint32_t* d_bits, int32_t n_items, int32_t* d_list,
                                int32_t* d_count, cudaStream_t st) {
  if (n_items <= 0 || !d_bits || !d_list || !d_count) return gram_set_error(ctx, "gram_touched_list: bad argument"), GRAM_ERR_ARG;
  ProfScope prof(ctx, GRAM_K_OTHER, (double)n_items / 8.0, 1, st);
  launch_chain(touched_list_kernel, 1, 1024, 0, st, d_bits, n_items, d_list, d_count);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

// ---------------------------------------------------------------------------------------------
// The segmented sum for callers that must not allocate.  Its chunk-boundary partial sums live in
// a fixed array that is part of the library image, so the call touches no allocator at all.
// ---------------------------------------------------------------------------------------------
namespace {
constexpr int kStaticChunks = 592;            // work units (4 per SM)
constexpr int kStaticMaxD = 1024;             // widest row the fixed scratch can serve
constexpr size_t kStaticPartialFloats = (size_t)kStaticChunks * 2 * kStaticMaxD;
// [0, kStaticPartialFloats): partial sums; then 64 floats whose first word is the device status word; then one
// (item, last chunk) pair per work unit
static __device__ __align__(256) float g_static_scratch[kStaticPartialFloats + 64 + 2 * kStaticChunks];

constexpr int kMaxDevices = 64;
float* g_static_ptr[kMaxDevices] = {};        // device address of the array, looked up once per device

void static_fail(char* h_err, size_t n, const char* msg) {
  if (h_err && n) snprintf(h_err, n, "%s", msg);
}
}  // namespace

extern "C" gram_status gram_accumulate_static(const float* d_dE, const int32_t* d_perm, const int32_t* d_seg_off,
                                               int64_t P, int32_t U, int32_t d, float* d_G, gram_stream stream,
                                               char* h_err, size_t err_len) {
  if (h_err && err_len) h_err[0] = 0;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (P < 0 || U < 0 || d <= 0 || U > P) return static_fail(h_err, err_len, "gram_accumulate_static: bad size"), GRAM_ERR_ARG;
  if (d > kStaticMaxD) {
    if (h_err && err_len) snprintf(h_err, err_len, "gram_accumulate_static: d=%d exceeds the fixed scratch's maximum of %d columns", d, kStaticMaxD);
    return GRAM_ERR_WORKSPACE;
  }
  if (P > INT32_MAX) return static_fail(h_err, err_len, "gram_accumulate_static: P exceeds 2^31-1 positions"), GRAM_ERR_WORKSPACE;
  if (P == 0 || U == 0) return GRAM_OK;
  if (!d_dE || !d_perm || !d_seg_off || !d_G) return static_fail(h_err, err_len, "gram_accumulate_static: null buffer"), GRAM_ERR_ARG;
  if (d % 4 != 0 || ((uintptr_t)d_dE % 16) || ((uintptr_t)d_G % 16))
    return static_fail(h_err, err_len, "gram_accumulate_static: d must be a multiple of 4 and buffers 16-byte aligned"), GRAM_ERR_UNSUPPORTED;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return static_fail(h_err, err_len, "gram_accumulate_static: cannot identify the current device"), GRAM_ERR_CUDA;
  if (!g_static_ptr[dev]) {
    // in host code the array's name is only a handle: ask the runtime for its address on this device
    float* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress((void**)&ptr, g_static_scratch);
    if (e != cudaSuccess || !ptr) {
      if (h_err && err_len) snprintf(h_err, err_len, "gram_accumulate_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      return GRAM_ERR_CUDA;
    }
    g_static_ptr[dev] = ptr;
  }
  float* partial = g_static_ptr[dev];
  int32_t* status = reinterpret_cast<int32_t*>(partial + kStaticPartialFloats);
  int2* span = reinterpret_cast<int2*>(partial + kStaticPartialFloats + 64);
  // the status word must start at zero; the partial sums and the (item, last chunk) pairs need no clearing
  // (each slot that is read in a call has been written earlier in the same call)
  if (cudaMemsetAsync(status, 0, sizeof(int32_t), st) != cudaSuccess)
    return static_fail(h_err, err_len, "gram_accumulate_static: clearing the status word failed"), GRAM_ERR_CUDA;
  int64_t nchunks = ceil_div64(P, 16);
  if (nchunks > kStaticChunks) nchunks = kStaticChunks;
  const int64_t R = ceil_div64(P, nchunks);
  nchunks = ceil_div64(P, R);
  if (d >= 256) segsum_run<2>(d_dE, d_perm, d_seg_off, P, U, d, R, (int)nchunks, nullptr, 0, d_G, partial, span, status, nullptr, st, nullptr, INT32_MAX);
  else segsum_run<1>(d_dE, d_perm, d_seg_off, P, U, d, R, (int)nchunks, nullptr, 0, d_G, partial, span, status, nullptr, st, nullptr, INT32_MAX);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    if (h_err && err_len) snprintf(h_err, err_len, "gram_accumulate_static: launch failed: %s", cudaGetErrorString(e));
    return GRAM_ERR_CUDA;
  }
  return GRAM_OK;
}
