// Stage 1 of the GRAM step: the unique-item set B_I of a mini-batch (Table 1) and the
// occurrence -> item map of Fig. 1, as a stable LSD radix sort of (item ID, position) over
// the low ceil(log2 n_items) key bits followed by a run-length pass.
//
// Small batches take one launch by one cluster of blocks (cluster_dedup_kernel).  Larger ones: one launch per radix pass
// of up to 10 bits (digit_plan): a block takes the next tile of 8192 keys (a ticket, so that
// every earlier tile is already running), ranks its keys within the tile, publishes the tile's
// digit counts and obtains the counts of all earlier tiles by looking back over their status
// words (the chained-scan idea of Merrill & Garland's decoupled look-back, as used by one-sweep
// radix sorts), then reorders the tile by digit in shared memory so that every digit leaves as
// one contiguous run.  Traffic per pass: 8P read + 8P written (the first pass generates the
// position payload instead of reading it); the digit totals of all passes come from one read of
// the keys before the first pass.  The run-length pass counts and then writes (two launches, no wait between blocks).
//
// Every wait on another tile is bounded: a tile that gives up records GRAM_ERR_TIMEOUT, releases
// its successors and writes nothing; every scattered write is bounds-checked.
#include "gram_internal.h"

namespace {

constexpr int RADIX = 256;                       // bins of the one-launch form's passes
constexpr int RADIX_MAX = 1024;                  // and of the widest pass of the other
constexpr int RS_THREADS = 512;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;   // keys per tile
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int kMaxPasses = 4;
constexpr int RLE_THREADS = 512;
constexpr int RLE_ITEMS = 16;
constexpr int RLE_TILE = RLE_THREADS * RLE_ITEMS;
constexpr int RLE_GROUP = 64;                    // tiles of the run-length pass whose counts are also kept as one sum
constexpr int TOT_THREADS = 512;

// status word of a (tile, digit): two flag bits above a 30-bit count
constexpr uint32_t LB_AGG = 1u << 30;      // the tile's own count
constexpr uint32_t LB_INCL = 2u << 30;     // the count of this tile and all earlier ones
constexpr uint32_t LB_MASK = LB_AGG - 1u;
constexpr int kSpinLimit = 1 << 20;        // polls of one predecessor before giving up (about a second)

// control block (32-bit words), cleared by one memset per call:
// tickets of the radix passes, digit totals [kMaxPasses][RADIX_MAX], then the status words of every pass and the counts of
// the run-length pass per tile and per group of tiles
constexpr int CTL_TICKET = 0, CTL_TOTALS = 8, CTL_WORDS = CTL_TOTALS + kMaxPasses * RADIX_MAX;

__device__ __forceinline__ uint32_t lb_load(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void lb_store(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A tile publishes its count for a slot as soon as it has it (lb_publish), reorders its keys in shared memory meanwhile, and
// then asks for the sum over all earlier tiles (lb_resolve), which replaces the published word by the inclusive one.  A word
// carries its flag and its count together, so no ordering between two stores is needed.  The words of LB_WINDOW predecessors
// are fetched at once (independent loads): eight, four with two slots per thread; 32 / 16 made a pass 10 % slower (registers).
// N: slots per thread, 1 or 2 (neighbouring, the first even: their words travel as one 64-bit access).
// false: a predecessor never published within the limit (the caller must then write nothing).
template <int N> struct LbWords { uint32_t v[N]; };
template <int N> __device__ __forceinline__ LbWords<N> lb_get(const uint32_t* p) {
  LbWords<N> r;
  if constexpr (N == 1) {
    r.v[0] = lb_load(p);
  } else {
    uint64_t x;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
    r.v[0] = (uint32_t)x;
    r.v[1] = (uint32_t)(x >> 32);
  }
  return r;
}
template <int N> __device__ __forceinline__ void lb_put(uint32_t* p, const LbWords<N>& w) {
  if constexpr (N == 1) lb_store(p, w.v[0]);
  else asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"((uint64_t)w.v[0] | ((uint64_t)w.v[N - 1] << 32)) : "memory");
}
template <int N> __device__ __forceinline__ void lb_publish(uint32_t* lb, int tile, int stride, int slot, const uint32_t (&own)[N]) {
  LbWords<N> w;
#pragma unroll
  for (int n = 0; n < N; ++n) w.v[n] = own[n] | (tile == 0 ? LB_INCL : LB_AGG);
  lb_put<N>(lb + (size_t)tile * stride + slot, w);
}
template <int N, int LB_WINDOW>
__device__ __forceinline__ bool lb_resolve(uint32_t* lb, int tile, int stride, int slot, const uint32_t (&own)[N], uint32_t (&excl)[N]) {
  LbWords<N> incl;
  bool done[N];
#pragma unroll
  for (int n = 0; n < N; ++n) { excl[n] = 0; done[n] = false; }
  if (tile == 0) return true;
  uint32_t* mine = lb + (size_t)tile * stride + slot;
  int spins = 0;
  int t = tile - 1;
  while (true) {
    LbWords<N> w[LB_WINDOW];
#pragma unroll
    for (int i = 0; i < LB_WINDOW; ++i) {
      if (t - i >= 0) {
        w[i] = lb_get<N>(lb + (size_t)(t - i) * stride + slot);
      } else {                              // before tile 0: nothing
#pragma unroll
        for (int n = 0; n < N; ++n) w[i].v[n] = LB_INCL;
      }
    }
    int used = 0;
    bool all = false;
#pragma unroll
    for (int i = 0; i < LB_WINDOW; ++i) {
      bool ready = used == i && !all;
#pragma unroll
      for (int n = 0; n < N; ++n) ready = ready && (w[i].v[n] & ~LB_MASK) != 0u;
      if (ready) {
        all = true;
#pragma unroll
        for (int n = 0; n < N; ++n) {
          if (!done[n]) {
            excl[n] += w[i].v[n] & LB_MASK;
            done[n] = (w[i].v[n] & LB_INCL) != 0u;
          }
          all = all && done[n];
        }
        used = i + 1;
      }
    }
    if (all) break;
    t -= used;
    if (used < LB_WINDOW) {                 // tile t has not published yet
      if (++spins > kSpinLimit) {
#pragma unroll
        for (int n = 0; n < N; ++n) incl.v[n] = LB_INCL;
        lb_put<N>(mine, incl);              // let the tiles after this one finish (their output is void as well)
        return false;
      }
      __nanosleep(40);
    }
  }
#pragma unroll
  for (int n = 0; n < N; ++n) incl.v[n] = ((excl[n] + own[n]) & LB_MASK) | LB_INCL;
  lb_put<N>(mine, incl);
  return true;
}

// ---- digit totals of every pass from one read of the keys; range check of the IDs -----------
// Shared-memory histograms in `copies` interleaved copies (a lane adds to copy lane % copies): the occurrences of a hot
// item inside a warp spread over the copies, which sit in different banks.  Eight copies, four with 1024 bins.
__global__ void __launch_bounds__(TOT_THREADS) digit_totals_kernel(const int32_t* __restrict__ keys, int64_t P, int passes, int bits,
                                                                   int copies, int32_t n_items, uint32_t* __restrict__ totals,
                                                                   int32_t* status) {
  if (!chain_begin()) return;
  extern __shared__ uint32_t tot_smem[];               // [passes][bins][copies]
  const int bins = 1 << bits;
  for (int i = threadIdx.x; i < passes * bins * copies; i += TOT_THREADS) tot_smem[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int copy = lane & (copies - 1);
  constexpr int UNROLL = 4;
  const int64_t stride = (int64_t)gridDim.x * TOT_THREADS * UNROLL;
  bool bad = false;
  // a warp reads UNROLL runs of 32 consecutive keys per iteration (independent loads)
  for (int64_t j0 = ((int64_t)blockIdx.x * TOT_THREADS + (threadIdx.x & ~31)) * UNROLL; j0 < P; j0 += stride) {
    int32_t k[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const int64_t j = j0 + u * 32 + lane;
      k[u] = (j < P) ? keys[j] : -1;
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      if (j0 + u * 32 + lane < P) {
        if (k[u] < 0 || k[u] >= n_items) { bad = true; k[u] = 0; }
        for (int p = 0; p < passes; ++p) atomicAdd(&tot_smem[(p * bins + ((k[u] >> (bits * p)) & (bins - 1))) * copies + copy], 1u);
      }
    }
  }
  if (bad) gram_device_fail(status, GRAM_ERR_ID_RANGE);
  __syncthreads();
  for (int i = threadIdx.x; i < passes * bins; i += TOT_THREADS) {
    uint32_t c = 0;
    for (int q = 0; q < copies; ++q) c += tot_smem[i * copies + q];
    if (c) atomicAdd(&totals[(i / bins) * RADIX_MAX + (i & (bins - 1))], c);
  }
}

// exclusive scan over the first 32 * WARPS threads of two values at once (the others pass zeros); all threads call
template <int WARPS>
__device__ __forceinline__ int2 scan_pair(int a, int b, int32_t (*sw)[16]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int ia = a, ib = b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ta = __shfl_up_sync(0xffffffffu, ia, o), tb = __shfl_up_sync(0xffffffffu, ib, o);
    if (lane >= o) { ia += ta; ib += tb; }
  }
  if (warp < WARPS && lane == 31) { sw[0][warp] = ia; sw[1][warp] = ib; }
  __syncthreads();
  int pa = 0, pb = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w)
    if (w < warp) { pa += sw[0][w]; pb += sw[1][w]; }
  return make_int2(pa + ia - a, pb + ib - b);
}

// How the lanes of a round with equal digits find each other.  One vote per digit bit costs about three instructions a bit; an
// OR of the lane's bit into the digit's word of the warp's own table costs the same for any width, but lanes of one digit
// follow each other there.  So one vote finds those with the first lane's digit, which is the digit of most lanes where one ID
// fills much of a batch, and only the others go to the table.  Whole calls over 10^7 positions, us, with a vote per bit /
// with the table alone / this way:
//   keys of        uniform          Zipf 1.1         Zipf 1.5         half of them one ID   one ID
//   16 bits (2x8)  220 / 206 / 212  210 / 207 / 196  205 / 212 / 183  212 / 215 / 197       197 / 217 / 155
//   18 bits (2x9)  269 / 257 / 261  241 / 238 / 226  231 / 236 / 210  248 / 251 / 233       223 / 246 / 181
//   20 bits (2x10) 292 / 276 / 280  257 / 249 / 238  242 / 245 / 215  263 / 262 / 242       231 / 246 / 182
// One pass of 7 bits: 123 with votes, 117 this way (two IDs alone, 16 lanes in line: 122 and 119); of 5 bits 115 and 107, but
// two IDs 113 and 118, so narrower passes keep the votes.  (The one-launch form below does the same at any width.)
constexpr int MATCH_BITS = 7;

template <int BINS> struct PassSmem {
  uint16_t cnt[RS_WARPS][BINS];    // keys of (warp, digit); later the warp's base inside the tile's digit run
  int32_t tile_excl[BINS];         // start of a digit's run inside the reordered tile
  int32_t gbase[BINS];             // global position of reordered element i of digit g is gbase[g] + i
  int32_t scan_w[2][16];
  int32_t tile, abort;
  union alignas(16) {              // cleared by 16-byte stores
    struct {
      int32_t keys[RS_TILE];
      int32_t vals[RS_TILE];
    };
    uint32_t match[RS_WARPS][BINS];  // before the reordering: lanes of the current round per (warp, digit); zeros between rounds
  };
};
static_assert(alignof(PassSmem<256>) == 16 && alignof(PassSmem<RADIX_MAX>) == 16, "the match tables start on 16 bytes");
static_assert(sizeof(uint32_t) * RS_WARPS * RADIX_MAX <= 2 * sizeof(int32_t) * RS_TILE, "the match tables fit the reordered tile");

// ---- one stable radix pass ------------------------------------------------------------------
// Warp w of a tile owns 32*RS_ITEMS consecutive keys and visits them 32 at a time, so that
// (tile, warp, round, lane) order is position order.  The rank of a key among equal digits:
// all earlier tiles + earlier warps of this tile + earlier rounds of this warp + earlier lanes.
// FULL: a tile without missing keys (all but the last one): no test per key.  The pass is bound by its shared-memory accesses
// (44 wavefronts per 32 keys, random words mostly; L1 72 % busy) and issues on 39 % of the cycles.
template <int NBITS, bool FULL>
__device__ __forceinline__ void radix_tile(PassSmem<(NBITS <= 8 ? 256 : 1024)>& s, const int32_t* __restrict__ kin,
                                           const int32_t* __restrict__ vin, int32_t tbase, int n_valid, uint32_t n_keys, int shift,
                                           int32_t n_items, int check_range, const uint32_t* __restrict__ totals, uint32_t* lb,
                                           int tile, int32_t* __restrict__ keys_out, int32_t* __restrict__ vals_out, int32_t* status) {
  constexpr int BINS = NBITS <= 8 ? 256 : 1024;
  constexpr int DPT = BINS / 512 > 0 ? BINS / 512 : 1;           // digits per thread in the digit-wise steps: one or two
  constexpr int DTHREADS = BINS / DPT;
  constexpr uint32_t MASK = (1u << NBITS) - 1u;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lbase = warp * (32 * RS_ITEMS) + lane;               // this lane's first key inside the tile
  kin += lbase;
  int32_t key[RS_ITEMS];
  int32_t pos[RS_ITEMS];
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) key[r] = (FULL || lbase + r * 32 < n_valid) ? kin[r * 32] : 0;
  if (check_range) {
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r)
      if ((uint32_t)key[r] >= (uint32_t)n_items) key[r] = 0;     // counted as 0 by the totals too
  }
  const uint32_t lt = (1u << lane) - 1u;
  uint16_t* my_cnt = s.cnt[warp];
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) {
    const bool valid = FULL || lbase + r * 32 < n_valid;
    const uint32_t dig = ((uint32_t)key[r] >> shift) & MASK;
    // lanes of this round with the same digit (a hardware match's latency grows with the number of distinct values)
    uint32_t peers;
    int32_t before = 0;
    if constexpr (NBITS >= MATCH_BITS) {
      const bool with_first = dig == __shfl_sync(0xffffffffu, dig, 0);       // the valid lanes are the first ones
      const uint32_t first_peers = __ballot_sync(0xffffffffu, valid && with_first);
      if (valid && !with_first) atomicOr(&s.match[warp][dig], 1u << lane);
      __syncwarp();
      peers = with_first ? first_peers : s.match[warp][dig];
    } else {
      peers = FULL ? 0xffffffffu : __ballot_sync(0xffffffffu, valid);
#pragma unroll
      for (int b = 0; b < NBITS; ++b) {
        const bool bit = (dig >> b) & 1u;
        const uint32_t vote = __ballot_sync(0xffffffffu, bit);
        peers &= vote ^ (bit ? 0u : 0xffffffffu);
      }
    }
    if (valid) before = my_cnt[dig];
    __syncwarp();
    const uint32_t earlier = peers & lt;
    pos[r] = before + __popc(earlier);
    if (valid && earlier == 0u) {
      my_cnt[dig] = (uint16_t)(before + __popc(peers));
      if constexpr (NBITS >= MATCH_BITS) s.match[warp][dig] = 0u;
    }
    __syncwarp();
  }
  __syncthreads();
  // digit-wise steps: thread t owns digit t, or digits 2t and 2t + 1 (their 16-bit counters as one word; a warp counts at
  // most 512 keys and a tile 8192, so the halves do not run over)
  uint32_t run = 0;
  int32_t tot[2] = {0, 0};
  if (tid < DTHREADS) {
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
      if (DPT == 1) {
        const uint32_t c = s.cnt[w][tid];
        s.cnt[w][tid] = (uint16_t)run;
        run += c;
      } else {
        uint32_t* p = reinterpret_cast<uint32_t*>(&s.cnt[w][0]) + tid;
        const uint32_t c = *p;
        *p = run;
        run += c;
      }
    }
    tot[0] = (int32_t)totals[tid * DPT];
    if (DPT == 2) tot[1] = (int32_t)totals[tid * DPT + 1];
  }
  const uint32_t count[2] = {DPT == 1 ? run : run & 0xFFFFu, DPT == 1 ? 0u : run >> 16};
  uint32_t own[DPT];
#pragma unroll
  for (int n = 0; n < DPT; ++n) own[n] = count[n];
  if (tid < DTHREADS) lb_publish<DPT>(lb, tile, BINS, tid * DPT, own);
  const int2 ex = scan_pair<DTHREADS / 32>((int)(count[0] + count[1]), tot[0] + tot[1], s.scan_w);
  if (tid < DTHREADS) {
    s.tile_excl[tid * DPT] = ex.x;
    if (DPT == 2) s.tile_excl[tid * DPT + 1] = ex.x + (int)count[0];
  }
  __syncthreads();
  // reorder the tile by digit in shared memory
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) {
    if (FULL || lbase + r * 32 < n_valid) {
      const uint32_t dig = ((uint32_t)key[r] >> shift) & MASK;
      pos[r] += s.tile_excl[dig] + my_cnt[dig];
      s.keys[pos[r]] = key[r];
    }
  }
  if (vin) {
    vin += lbase;
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) key[r] = (FULL || lbase + r * 32 < n_valid) ? vin[r * 32] : 0;
  } else {
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) key[r] = tbase + lbase + r * 32;
  }
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r)
    if (FULL || lbase + r * 32 < n_valid) s.vals[pos[r]] = key[r];
  if (tid < DTHREADS) {
    uint32_t before[DPT];
    if (!lb_resolve<DPT, DPT == 1 ? 8 : 4>(lb, tile, BINS, tid * DPT, own, before)) {
      s.abort = 1;
      gram_device_fail(status, GRAM_ERR_TIMEOUT);
    }
    s.gbase[tid * DPT] = ex.y + (int32_t)before[0] - ex.x;
    if (DPT == 2) s.gbase[tid * DPT + 1] = ex.y + tot[0] + (int32_t)before[DPT - 1] - (ex.x + (int)count[0]);
  }
  __syncthreads();
  if (s.abort) return;
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) {
    const int i = tid + r * RS_THREADS;
    if (FULL || i < n_valid) {
      const uint32_t k = (uint32_t)s.keys[i];
      const uint32_t dst = (uint32_t)(s.gbase[(k >> shift) & MASK] + i);
      if (dst < n_keys) {                    // always true unless an earlier tile gave up
        keys_out[dst] = (int32_t)k;
        vals_out[dst] = s.vals[i];
      }
    }
  }
}

template <int NBITS>
__global__ void __launch_bounds__(RS_THREADS, 2) radix_pass_kernel(const int32_t* __restrict__ keys_in,
                                                                   const int32_t* __restrict__ vals_in, int64_t P, int shift,
                                                                   int32_t n_items, int check_range,
                                                                   const uint32_t* __restrict__ totals, uint32_t* lb,
                                                                   int32_t* ticket, int32_t* __restrict__ keys_out,
                                                                   int32_t* __restrict__ vals_out, int32_t* status) {
  if (!chain_begin()) return;
  constexpr int BINS = NBITS <= 8 ? 256 : 1024;
  extern __shared__ __align__(16) unsigned char pass_smem_raw[];
  PassSmem<BINS>& s = *reinterpret_cast<PassSmem<BINS>*>(pass_smem_raw);
  if (threadIdx.x == 0) {
    s.tile = atomicAdd(ticket, 1);
    s.abort = 0;
  }
  for (int i = threadIdx.x; i < RS_WARPS * BINS / 2; i += RS_THREADS) reinterpret_cast<uint32_t*>(&s.cnt[0][0])[i] = 0u;
  if constexpr (NBITS >= MATCH_BITS) {
    for (int i = threadIdx.x; i < RS_WARPS * BINS / 4; i += RS_THREADS) reinterpret_cast<uint4*>(&s.match[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  const int tile = s.tile;
  const int64_t tbase = (int64_t)tile * RS_TILE, left = P - tbase;
  const int32_t* vin = vals_in ? vals_in + tbase : nullptr;
  if (left >= RS_TILE)
    radix_tile<NBITS, true>(s, keys_in + tbase, vin, (int32_t)tbase, RS_TILE, (uint32_t)P, shift, n_items, check_range, totals, lb, tile,
                            keys_out, vals_out, status);
  else
    radix_tile<NBITS, false>(s, keys_in + tbase, vin, (int32_t)tbase, (int)left, (uint32_t)P, shift, n_items, check_range, totals, lb,
                             tile, keys_out, vals_out, status);
}

typedef void (*RadixPassFn)(const int32_t*, const int32_t*, int64_t, int, int32_t, int, const uint32_t*, uint32_t*, int32_t*,
                            int32_t*, int32_t*, int32_t*);
// the instantiation for a pass whose digits have `nbits` bits
RadixPassFn radix_pass_fn(int nbits) {
  switch (nbits) {
    case 1: return radix_pass_kernel<1>;
    case 2: return radix_pass_kernel<2>;
    case 3: return radix_pass_kernel<3>;
    case 4: return radix_pass_kernel<4>;
    case 5: return radix_pass_kernel<5>;
    case 6: return radix_pass_kernel<6>;
    case 7: return radix_pass_kernel<7>;
    case 8: return radix_pass_kernel<8>;
    case 9: return radix_pass_kernel<9>;
    default: return radix_pass_kernel<10>;
  }
}
size_t radix_pass_smem(int nbits) { return nbits <= 8 ? sizeof(PassSmem<256>) : sizeof(PassSmem<1024>); }

// Passes of the sort over keys of `key_bits` bits: as few as 10-bit digits allow, the bits spread evenly.  Two passes over
// 1024 bins took 107 + 102 us at 10^7 positions of 20-bit keys (with votes), where three over 256 bins took 95 + 89 + 73.
struct DigitPlan {
  int passes, bits, bins;
};
DigitPlan digit_plan(int key_bits) {
  DigitPlan p;
  if (key_bits < 1) key_bits = 1;
  p.passes = (key_bits + 9) / 10;
  p.bits = (key_bits + p.passes - 1) / p.passes;
  p.bins = p.bits <= 8 ? 256 : 1024;
  return p;
}
int key_bits_of(int32_t n_items) {
  int bits = 0;
  while (((int64_t)1 << bits) < (int64_t)n_items) ++bits;
  return bits;
}

// exclusive scan of one value per thread over the block; returns the thread's base
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t thread_total, int32_t* sw /*[33]*/, int32_t* block_total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t incl = thread_total;
  for (int o = 1; o < 32; o <<= 1) {
    int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) sw[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int32_t w = (lane < (int)(blockDim.x >> 5)) ? sw[lane] : 0;
    int32_t wi = w;
    for (int o = 1; o < 32; o <<= 1) {
      int32_t t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    sw[lane] = wi - w;
    if (lane == 31) sw[32] = wi;
  }
  __syncthreads();
  int32_t r = sw[warp] + incl - thread_total;
  if (block_total) *block_total = sw[32];
  __syncthreads();
  return r;
}

// ---- run-length pass over the sorted keys: unique, seg_off, item -> rank table, U -------------
// Two launches without a wait between blocks: the items that start in each tile are counted, tile by tile and per group of
// RLE_GROUP tiles; then every tile adds up the groups and the tiles of its own group before it and writes its items.  The
// sorted keys are still in L2 for both (10^7 keys: 40 MB).  One launch with a look-back over the tiles took 44 us there
// (10 us per wave of resident tiles for the way back), the two take 19 + 25 us in isolation
// and 20 us less of the whole call, because the second no longer keeps SMs waiting.
// Warp w of a tile owns 32 * RLE_ITEMS consecutive keys and reads them 32 at a time, all loads in flight together.
__device__ __forceinline__ void rle_load(const int32_t* __restrict__ sk, int64_t P, int64_t base, int lane, int32_t (&k)[RLE_ITEMS],
                                         int32_t& before) {
#pragma unroll
  for (int i = 0; i < RLE_ITEMS; ++i) {
    const int64_t j = base + i * 32 + lane;
    k[i] = (j < P) ? sk[j] : -1;                                 // IDs are non-negative, so places past the end are no heads
  }
  before = (base > 0 && base <= P) ? sk[base - 1] : -1;
}
// lanes of round i whose key starts an item
__device__ __forceinline__ uint32_t rle_heads(const int32_t (&k)[RLE_ITEMS], int i, int32_t before, int lane) {
  int32_t prev = __shfl_up_sync(0xffffffffu, k[i], 1);
  const int32_t last = __shfl_sync(0xffffffffu, k[i > 0 ? i - 1 : 0], 31);
  if (lane == 0) prev = i > 0 ? last : before;
  return __ballot_sync(0xffffffffu, k[i] >= 0 && k[i] != prev);
}
__global__ void __launch_bounds__(RLE_THREADS) rle_count_kernel(const int32_t* __restrict__ sk, int64_t P, int32_t* __restrict__ tile_heads,
                                                               int32_t* __restrict__ group_heads) {
  if (!chain_begin()) return;
  __shared__ int32_t sum;
  if (threadIdx.x == 0) sum = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t k[RLE_ITEMS], before, n = 0;
  rle_load(sk, P, (int64_t)blockIdx.x * RLE_TILE + warp * (32 * RLE_ITEMS), lane, k, before);
#pragma unroll
  for (int i = 0; i < RLE_ITEMS; ++i) n += __popc(rle_heads(k, i, before, lane));
  if (lane == 0) atomicAdd(&sum, n);
  __syncthreads();
  if (threadIdx.x == 0) {
    tile_heads[blockIdx.x] = sum;
    atomicAdd(&group_heads[blockIdx.x / RLE_GROUP], sum);
  }
}
__global__ void __launch_bounds__(RLE_THREADS) rle_kernel(const int32_t* __restrict__ sk, int64_t P, int ntiles, int32_t cap,
                                                         int32_t n_items, const int32_t* __restrict__ tile_heads,
                                                         const int32_t* __restrict__ group_heads, int32_t* __restrict__ unique,
                                                         int32_t* __restrict__ seg_off, int32_t* __restrict__ rank_table,
                                                         int32_t* __restrict__ n_unique) {
  if (!chain_begin()) return;
  __shared__ int32_t sw[33];
  __shared__ int32_t s_before;
  if (threadIdx.x == 0) s_before = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = blockIdx.x, group = tile / RLE_GROUP;
  const int64_t base = (int64_t)tile * RLE_TILE + warp * (32 * RLE_ITEMS);
  int32_t k[RLE_ITEMS], before;
  rle_load(sk, P, base, lane, k, before);
  int32_t earlier = 0;                                           // items that start in earlier tiles
  for (int g = threadIdx.x; g < group; g += RLE_THREADS) earlier += group_heads[g];
  for (int t = group * RLE_GROUP + threadIdx.x; t < tile; t += RLE_THREADS) earlier += tile_heads[t];
  earlier = __reduce_add_sync(0xffffffffu, earlier);
  if (lane == 0 && earlier) atomicAdd(&s_before, earlier);       // integers: the order does not matter
  int32_t tot = 0;
#pragma unroll
  for (int i = 0; i < RLE_ITEMS; ++i) tot += __popc(rle_heads(k, i, before, lane));
  int32_t btot;
  int32_t ex = block_exclusive_scan(lane == 0 ? tot : 0, sw, &btot);
  ex = __shfl_sync(0xffffffffu, ex, 0) + s_before;
#pragma unroll
  for (int i = 0; i < RLE_ITEMS; ++i) {
    const uint32_t heads = rle_heads(k, i, before, lane);
    if (heads & (1u << lane)) {
      const int32_t u = ex + __popc(heads & ((1u << lane) - 1u));
      if (u < cap && (uint32_t)k[i] < (uint32_t)n_items) {       // always true unless a pass gave up
        unique[u] = k[i];
        seg_off[u] = (int32_t)(base + i * 32 + lane);
        rank_table[k[i]] = u;
      }
    }
    ex += __popc(heads);
  }
  if (tile == ntiles - 1 && threadIdx.x == 0) {
    const int32_t U = s_before + btot;
    *n_unique = U;
    if (U <= cap) seg_off[U] = (int32_t)P;
  }
}

__global__ void __launch_bounds__(256) inverse_kernel(const int32_t* __restrict__ ids, int64_t P, int32_t n_items,
                                                      const int32_t* __restrict__ rank_table, int32_t* __restrict__ inverse) {
  if (!chain_begin()) return;
  constexpr int UNROLL = 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * UNROLL;
  for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x * UNROLL + threadIdx.x; p0 < P; p0 += stride) {
    int32_t id[UNROLL], r[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const int64_t p = p0 + (int64_t)u * blockDim.x;
      id[u] = (p < P) ? ids[p] : -1;
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) r[u] = (id[u] >= 0 && id[u] < n_items) ? rank_table[id[u]] : -1;   // out of range: already recorded
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const int64_t p = p0 + (int64_t)u * blockDim.x;
      if (p < P) inverse[p] = r[u];
    }
  }
}

// ---- the whole dedup of a small batch in one launch -------------------------------------------
// Up to 16 x 4096 positions the sort is a chain of launches and look-backs that move next to nothing (25 600 positions
// over 10 000 items: 45 us, of which the traffic is 0.3; 12.5 us this way).  Here one cluster of up to 16 blocks holds all (ID, position)
// pairs in its shared memory: block r owns the sorted places r * TILE .., a radix pass ranks a block's pairs as above,
// the blocks read each other's digit counts, and every pair goes straight to its place in the owner's shared memory.
// The run-length pass and `inverse` follow in the same launch.  Between phases: cluster barriers, two a pass and one for the counts of
// items, which every block writes to all others so that none is read after it.  What bounds it is this chain of barriers and of
// looks into other blocks' memory: with a loop over the blocks' counts, votes for equal digits and a barrier at the end 15.4 us,
// 65 536 positions over 10^6 items 35.9 (30.5 now), 40 000 over 30 000 25.3 (21.4).  A position whose ID is out of range carries
// the sign bit along.
constexpr int CD_THREADS = 512;
constexpr int CD_WARPS = CD_THREADS / 32;
constexpr int kClusterMaxBlocks = 16;     // an opt-in above 8

__device__ __forceinline__ uint32_t cd_remote(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ int32_t cd_load(uint32_t a) {
  int32_t v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

// a word at the same place in every block of the cluster, all on their way together (a loop over the blocks waits some 200 cycles
// for each of them): v[i] is that of block `rank` + i, going round, so that the blocks do not all ask the same one; 0 from `blocks` on
__device__ __forceinline__ void cd_load_all(const void* p, int rank, int blocks, int32_t (&v)[kClusterMaxBlocks]) {
#pragma unroll
  for (int i = 0; i < kClusterMaxBlocks; ++i) {
    const int b = i >= blocks ? rank : (rank + i < blocks ? rank + i : rank + i - blocks);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %2, %3;\n\tmov.b32 %0, 0;\n\t@p ld.shared::cluster.s32 %0, [%1];\n\t}"
                 : "=&r"(v[i])
                 : "r"(cd_remote(p, (uint32_t)b)), "r"(i), "r"(blocks)
                 : "memory");
  }
}

template <int ROUNDS> struct ClusterSmem {
  int2 kv[CD_THREADS * ROUNDS];    // (ID, position) at this block's sorted places
  uint16_t cnt[CD_WARPS][RADIX];   // pairs of (warp, digit); later the warp's base inside the block's run of the digit
  int32_t count[RADIX];            // pairs of this block per digit (read by the others)
  int32_t gbase[RADIX];            // sorted place of this block's first pair of a digit
  int32_t scan_w[2][16];
  int32_t sw[33];
  alignas(16) uint32_t match[CD_WARPS][RADIX];   // lanes of the current round per (warp, digit); zeros between rounds
  int32_t heads[kClusterMaxBlocks];  // items that start in each block (written by that block)
};

template <int ROUNDS>
__global__ void __launch_bounds__(CD_THREADS) cluster_dedup_kernel(const int32_t* __restrict__ ids, int32_t P, int32_t n_items,
                                                                  int key_bits, int32_t* __restrict__ unique,
                                                                  int32_t* __restrict__ inverse, int32_t* __restrict__ perm,
                                                                  int32_t* __restrict__ seg_off, int32_t* __restrict__ n_unique,
                                                                  int32_t* status) {
  if (!chain_begin()) return;
  constexpr int TILE = CD_THREADS * ROUNDS;
  extern __shared__ __align__(16) unsigned char cd_smem_raw[];
  ClusterSmem<ROUNDS>& s = *reinterpret_cast<ClusterSmem<ROUNDS>*>(cd_smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x, blocks = gridDim.x;       // the grid is one cluster
  const int32_t base = rank * TILE;
  const int32_t n_valid = max(0, min(TILE, P - base));
  const int lbase = warp * (32 * ROUNDS) + lane;
  const uint32_t lt = (1u << lane) - 1u;
  uint16_t* my_cnt = s.cnt[warp];
  int32_t key[ROUNDS], val[ROUNDS], pos[ROUNDS];
  bool bad = false;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int i = lbase + r * 32;
    val[r] = base + i;
    key[r] = i < n_valid ? ids[base + i] : 0;
    if (key[r] < 0 || key[r] >= n_items) { bad = true; key[r] = 0; val[r] |= INT32_MIN; }
  }
  if (bad) gram_device_fail(status, GRAM_ERR_ID_RANGE);
  for (int i = tid; i < CD_WARPS * RADIX / 4; i += CD_THREADS) reinterpret_cast<uint4*>(&s.match[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int shift = 0; shift == 0 || shift < key_bits; shift += 8) {
    for (int i = tid; i < CD_WARPS * RADIX / 2; i += CD_THREADS) reinterpret_cast<uint32_t*>(&s.cnt[0][0])[i] = 0u;
    if (shift > 0) {
#pragma unroll
      for (int r = 0; r < ROUNDS; ++r) {
        const int2 x = s.kv[lbase + r * 32];
        key[r] = x.x;
        val[r] = x.y;
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {                   // stable rank among equal digits, as in radix_pass_kernel
      const bool valid = lbase + r * 32 < n_valid;
      const int dig = (key[r] >> shift) & 255;
      const bool with_first = dig == __shfl_sync(0xffffffffu, dig, 0);
      const uint32_t first_peers = __ballot_sync(0xffffffffu, valid && with_first);
      if (valid && !with_first) atomicOr(&s.match[warp][dig], 1u << lane);
      __syncwarp();
      const uint32_t peers = with_first ? first_peers : s.match[warp][dig];
      int32_t before = 0;
      if (valid) before = my_cnt[dig];
      __syncwarp();
      pos[r] = before + __popc(peers & lt);
      if (valid && (peers & lt) == 0u) {
        my_cnt[dig] = (uint16_t)(before + __popc(peers));
        s.match[warp][dig] = 0u;
      }
      __syncwarp();
    }
    __syncthreads();
    if (tid < RADIX) {
      int32_t run = 0;
#pragma unroll
      for (int w = 0; w < CD_WARPS; ++w) {
        const int32_t c = s.cnt[w][tid];
        s.cnt[w][tid] = (uint16_t)run;
        run += c;
      }
      s.count[tid] = run;
    }
    gram_cluster_sync();                                 // every block's pairs are in registers, its counts published
    int32_t total = 0, before_blocks = 0;
    if (tid < RADIX) {
      int32_t c[kClusterMaxBlocks];
      cd_load_all(&s.count[tid], rank, blocks, c);
#pragma unroll
      for (int i = 0; i < kClusterMaxBlocks; ++i) {
        total += c[i];
        if (rank + i >= blocks) before_blocks += c[i];     // block rank + i - blocks; zeros past the blocks
      }
    }
    const int2 ex = scan_pair<8>(total, 0, s.scan_w);
    if (tid < RADIX) s.gbase[tid] = ex.x + before_blocks;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
      if (lbase + r * 32 < n_valid) {
        const int dig = (key[r] >> shift) & 255;
        const int32_t dst = s.gbase[dig] + my_cnt[dig] + pos[r];        // 0 .. P - 1
        const uint32_t at = cd_remote(&s.kv[dst % TILE], (uint32_t)(dst / TILE));
        asm volatile("st.shared::cluster.v2.s32 [%0], {%1, %2};" ::"r"(at), "r"(key[r]), "r"(val[r]) : "memory");
      }
    }
    gram_cluster_sync();                                 // all pairs are at their places
  }
  // run lengths: thread t looks at ROUNDS consecutive places
  const int first = tid * ROUNDS;
  int32_t prev = -1;                                     // IDs are non-negative
  if (first > 0) prev = s.kv[first - 1].x;
  else if (rank > 0 && n_valid > 0) prev = cd_load(cd_remote(&s.kv[TILE - 1].x, (uint32_t)(rank - 1)));
  uint32_t heads = 0;
  int32_t tot = 0;
#pragma unroll
  for (int i = 0; i < ROUNDS; ++i) {
    const int2 x = s.kv[first + i];
    key[i] = x.x;
    val[i] = x.y;
    if (first + i < n_valid && key[i] != prev) { heads |= 1u << i; ++tot; }
    prev = key[i];
  }
  int32_t btot;
  int32_t ex = block_exclusive_scan(tot, s.sw, &btot);
  if (tid < blocks)
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cd_remote(&s.heads[rank], (uint32_t)tid)), "r"(btot) : "memory");
  gram_cluster_sync();                                   // the last look into another block's memory: blocks may leave after it
  int32_t U = 0;
  for (int b = 0; b < blocks; ++b) {
    if (b < rank) ex += s.heads[b];
    U += s.heads[b];
  }
#pragma unroll
  for (int i = 0; i < ROUNDS; ++i) {
    if (first + i < n_valid) {
      if (heads & (1u << i)) {
        unique[ex] = key[i];
        seg_off[ex] = base + first + i;
        ++ex;
      }
      const int32_t p = val[i] & INT32_MAX;
      perm[base + first + i] = p;
      inverse[p] = val[i] < 0 ? -1 : ex - 1;               // an ID out of range belongs to no item, as in inverse_kernel
    }
  }
  if (rank == 0 && tid == 0) {
    *n_unique = U;
    seg_off[U] = P;
  }
}

typedef void (*ClusterDedupFn)(const int32_t*, int32_t, int32_t, int, int32_t*, int32_t*, int32_t*, int32_t*, int32_t*, int32_t*);
struct ClusterDedup {
  ClusterDedupFn fn;
  int tile;
  size_t smem;
};
constexpr int kClusterForms = 4;
ClusterDedup cluster_dedup_form(int i) {
  switch (i) {
    case 0: return {cluster_dedup_kernel<1>, CD_THREADS, sizeof(ClusterSmem<1>)};
    case 1: return {cluster_dedup_kernel<2>, CD_THREADS * 2, sizeof(ClusterSmem<2>)};
    case 2: return {cluster_dedup_kernel<4>, CD_THREADS * 4, sizeof(ClusterSmem<4>)};
    default: return {cluster_dedup_kernel<8>, CD_THREADS * 8, sizeof(ClusterSmem<8>)};
  }
}

__global__ void dedup_empty_kernel(int32_t* seg_off, int32_t* n_unique) {
  if (!chain_begin()) return;
  seg_off[0] = 0;
  *n_unique = 0;
}

size_t rle_words(int64_t P) {
  const size_t t = (size_t)ceil_div64(P, RLE_TILE);
  return t + (t + RLE_GROUP - 1) / RLE_GROUP;
}
// 32-bit words of the control block for P positions over keys of up to max_key_bits bits (fewer bits may need more words)
size_t ctl_words(int64_t P, int max_key_bits) {
  const int64_t p = P > 0 ? P : 1;
  size_t per_tile = 0;
  for (int b = 1; b <= (max_key_bits > 1 ? max_key_bits : 1); ++b) {
    const DigitPlan d = digit_plan(b);
    const size_t w = (size_t)d.passes * d.bins;
    if (w > per_tile) per_tile = w;
  }
  const size_t words = per_tile * (size_t)ceil_div64(p, RS_TILE) + rle_words(p);
  return (size_t)CTL_WORDS + (words > 2 * RADIX ? words : 2 * RADIX);         // the self-test: two tiles of 256 bins
}
size_t totals_smem(const DigitPlan& d, int copies) { return (size_t)d.passes * (1 << d.bits) * copies * sizeof(uint32_t); }
int totals_copies(const DigitPlan& d) { return d.bins == 256 ? 8 : 4; }

}  // namespace

gram_status index_ws_alloc(gram_ctx* ctx, IndexWorkspace* ws, int64_t P_max, int32_t n_items_max, int32_t d_max) {
  ws->P_max = P_max;
  ws->n_items_max = n_items_max;
  ws->d_max = d_max;
  const size_t pb = (size_t)(P_max > 0 ? P_max : 1) * sizeof(int32_t);
  GRAM_CUDA(ctx, cudaMalloc(&ws->keys0, pb));
  GRAM_CUDA(ctx, cudaMalloc(&ws->keys1, pb));
  GRAM_CUDA(ctx, cudaMalloc(&ws->vals0, pb));
  GRAM_CUDA(ctx, cudaMalloc(&ws->vals1, pb));
  GRAM_CUDA(ctx, cudaMalloc(&ws->sort_ctl, ctl_words(P_max, key_bits_of(n_items_max > 0 ? n_items_max : 1)) * sizeof(uint32_t)));
  GRAM_CUDA(ctx, cudaMalloc(&ws->rank_table, (size_t)(n_items_max > 0 ? n_items_max : 1) * sizeof(int32_t)));
  GRAM_CUDA(ctx, cudaMalloc(&ws->partial, ((size_t)kAccMaxChunks * 2 * (d_max > 0 ? d_max : 1) + 2 * kAccMaxChunks) * sizeof(float)));
  int dev = 0;
  GRAM_CUDA(ctx, cudaGetDevice(&dev));
  static bool attributes_set[64] = {};                   // per device; setting them twice does no harm
  if (dev >= 64 || !attributes_set[dev]) {
    for (int b = 1; b <= 10; ++b)
      GRAM_CUDA(ctx, cudaFuncSetAttribute(radix_pass_fn(b), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)radix_pass_smem(b)));
    GRAM_CUDA(ctx, cudaFuncSetAttribute(digit_totals_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 3 * RADIX_MAX * 4 * (int)sizeof(uint32_t)));
    for (int i = 0; i < kClusterForms; ++i) {
      const ClusterDedup f = cluster_dedup_form(i);
      GRAM_CUDA(ctx, cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem));
      GRAM_CUDA(ctx, cudaFuncSetAttribute(f.fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    }
    if (dev < 64) attributes_set[dev] = true;
  }
  return GRAM_OK;
}

// The largest cluster of the widest one-launch form that can be placed now (a process may be limited to a part of the
// GPU's multiprocessors); the other kernels with clusters ask for less shared memory and fewer threads.
int32_t index_cluster_blocks() {
  const ClusterDedup f = cluster_dedup_form(kClusterForms - 1);
  for (int b = kClusterMaxBlocks; b > 1; b /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)b);
    cfg.blockDim = dim3(CD_THREADS);
    cfg.dynamicSmemBytes = f.smem;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)b;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, f.fn, &cfg) == cudaSuccess && n > 0) return b;
    (void)cudaGetLastError();
  }
  return 1;
}

void index_ws_free(IndexWorkspace* ws) {
  cudaFree(ws->keys0); cudaFree(ws->keys1); cudaFree(ws->vals0); cudaFree(ws->vals1);
  cudaFree(ws->sort_ctl); cudaFree(ws->rank_table); cudaFree(ws->partial);
  *ws = IndexWorkspace();
}

// A wait that nothing satisfies, to show that it ends: a radix pass is launched as tile 1 of a one-key input whose tile 0
// never runs, so its look-back finds no status word, gives up after kSpinLimit polls (about a second), records
// GRAM_ERR_TIMEOUT and writes nothing.
gram_status dedup_wait_selftest(gram_ctx* ctx, IndexWorkspace* ws, cudaStream_t st) {
  if (ws->P_max < 2) return gram_set_error(ctx, "the bounded-wait self-test needs a context with P_max >= 2"), GRAM_ERR_WORKSPACE;
  uint32_t* ctl = ws->sort_ctl;
  GRAM_CUDA(ctx, cudaMemsetAsync(ctl, 0, (size_t)(CTL_WORDS + 2 * RADIX) * sizeof(uint32_t), st));
  static const int32_t one = 1;
  GRAM_CUDA(ctx, cudaMemcpyAsync(reinterpret_cast<int32_t*>(ctl) + CTL_TICKET, &one, sizeof(one), cudaMemcpyHostToDevice, st));
  radix_pass_kernel<1><<<1, RS_THREADS, radix_pass_smem(1), st>>>(ws->keys0, nullptr, 1, 0, 1, 1, ctl + CTL_TOTALS, ctl + CTL_WORDS,
                                                                 reinterpret_cast<int32_t*>(ctl) + CTL_TICKET, ws->keys1, ws->vals1,
                                                                 gram_status_word(ctx));
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}

gram_status dedup_launch(gram_ctx* ctx, IndexWorkspace* ws, const int32_t* d_ids, int64_t P, int32_t n_items,
                         int32_t* d_unique, int32_t* d_inverse, int32_t* d_perm, int32_t* d_seg_off,
                         int32_t* d_n_unique, cudaStream_t st) {
  if (P < 0 || n_items <= 0 || !d_unique || !d_inverse || !d_perm || !d_seg_off || !d_n_unique || (P > 0 && !d_ids))
    return gram_set_error(ctx, "gram_dedup: bad argument"), GRAM_ERR_ARG;
  if (P > ws->P_max || n_items > ws->n_items_max)
    return gram_set_error(ctx, "gram_dedup: P=%lld n_items=%d exceed the context's P_max=%lld n_items=%d",
                          (long long)P, n_items, (long long)ws->P_max, ws->n_items_max), GRAM_ERR_WORKSPACE;
  if (P > (int64_t)LB_MASK)
    return gram_set_error(ctx, "gram_dedup: P=%lld is above the limit of 2^30 - 1 positions per call", (long long)P), GRAM_ERR_UNSUPPORTED;
  if (P == 0) {
    launch_chain(dedup_empty_kernel, 1, 1, 0, st, d_seg_off, d_n_unique);
    GRAM_LAUNCH_CHECK(ctx);
    return GRAM_OK;
  }
  const int key_bits = key_bits_of(n_items);
  const DigitPlan plan = digit_plan(key_bits);
  const int passes = plan.passes;
  // Up to 65 536 positions: the single launch, with the fewest positions per block.  Against the chain of launches, 10 000
  // items: 13 against 32 us at 25 600 positions, 21 / 32 at 65 536 (over 10^6 items 30 / 40); with twice the positions per block it took
  // 42 us at 131 072 where the chain takes 35: 16 SMs are then too few.  Where only smaller clusters can be placed, the line is lower.
  int form = 0;
  while (form < kClusterForms && P > (int64_t)gram_cluster_blocks(ctx) * cluster_dedup_form(form).tile) ++form;
  if (form < kClusterForms) {
    const ClusterDedup f = cluster_dedup_form(form);
    int blocks = 1;
    while ((int64_t)blocks * f.tile < P) blocks *= 2;
    ProfScope prof(ctx, GRAM_K_DEDUP, 12.0 * (double)P, 1, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(CD_THREADS);
    cfg.dynamicSmemBytes = f.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = chain_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    GRAM_CUDA(ctx, cudaLaunchKernelEx(&cfg, f.fn, d_ids, (int32_t)P, n_items, key_bits, d_unique, d_inverse, d_perm, d_seg_off, d_n_unique,
                                      gram_status_word(ctx)));
    return GRAM_OK;
  }
  const int ntiles = (int)ceil_div64(P, RS_TILE);
  const int rtiles = (int)ceil_div64(P, RLE_TILE);
  int32_t* status = gram_status_word(ctx);
  ProfScope prof(ctx, GRAM_K_DEDUP, (16.0 * passes + 20.0) * (double)P, passes + 4, st);

  uint32_t* ctl = ws->sort_ctl;
  const size_t lb_words = (size_t)passes * ntiles * plan.bins;
  GRAM_CUDA(ctx, cudaMemsetAsync(ctl, 0, ((size_t)CTL_WORDS + lb_words + rle_words(P)) * sizeof(uint32_t), st));
  uint32_t* totals = ctl + CTL_TOTALS;
  uint32_t* lb = ctl + CTL_WORDS;
  int tb = (int)ceil_div64(P, (int64_t)TOT_THREADS * 16);
  if (tb > kNumSMs * 4) tb = kNumSMs * 4;
  launch_chain(digit_totals_kernel, tb, TOT_THREADS, totals_smem(plan, totals_copies(plan)), st, d_ids, P, passes, plan.bits,
               totals_copies(plan), n_items, totals, status);

  const int32_t* kin = d_ids;
  const int32_t* vin = nullptr;
  int32_t* kbuf[2] = {ws->keys0, ws->keys1};
  int32_t* vbuf[2] = {ws->vals0, ws->vals1};
  for (int p = 0; p < passes; ++p) {
    int32_t* kout = kbuf[p & 1];
    int32_t* vout = (p == passes - 1) ? d_perm : vbuf[p & 1];
    launch_chain(radix_pass_fn(plan.bits), ntiles, RS_THREADS, radix_pass_smem(plan.bits), st, kin, vin, P, plan.bits * p, n_items, p == 0,
                 totals + p * RADIX_MAX, lb + (size_t)p * ntiles * plan.bins, reinterpret_cast<int32_t*>(ctl) + CTL_TICKET + p, kout, vout,
                 status);
    kin = kout;
    vin = vout;
  }
  GRAM_LAUNCH_CHECK(ctx);
  const int32_t cap = (int32_t)(P < (int64_t)n_items ? P : (int64_t)n_items);
  int32_t* tile_heads = reinterpret_cast<int32_t*>(lb + lb_words);
  int32_t* group_heads = tile_heads + rtiles;
  launch_chain(rle_count_kernel, rtiles, RLE_THREADS, 0, st, kin, P, tile_heads, group_heads);
  launch_chain(rle_kernel, rtiles, RLE_THREADS, 0, st, kin, P, rtiles, cap, n_items, tile_heads, group_heads, d_unique, d_seg_off,
               ws->rank_table, d_n_unique);
  int ib = (int)ceil_div64(P, 256 * 4);
  if (ib > kNumSMs * 16) ib = kNumSMs * 16;
  launch_chain(inverse_kernel, ib, 256, 0, st, d_ids, P, n_items, ws->rank_table, d_inverse);
  GRAM_LAUNCH_CHECK(ctx);
  return GRAM_OK;
}
