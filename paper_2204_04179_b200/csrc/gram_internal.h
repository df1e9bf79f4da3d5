// Internal declarations shared by the CUDA translation units of libgram.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include "gram.h"

typedef __nv_bfloat16 bf16;

// ---------------------------------------------------------------------------
// error plumbing
// ---------------------------------------------------------------------------
struct gram_ctx;
void gram_set_error(gram_ctx* ctx, const char* fmt, ...);

#define GRAM_CUDA(ctx, expr)                                                              \
  do {                                                                                    \
    cudaError_t e__ = (expr);                                                             \
    if (e__ != cudaSuccess) {                                                             \
      gram_set_error((ctx), "%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e__), __FILE__, __LINE__); \
      return GRAM_ERR_CUDA;                                                               \
    }                                                                                     \
  } while (0)

#define GRAM_TRY(expr)                        \
  do {                                        \
    gram_status s__ = (expr);                 \
    if (s__ != GRAM_OK) return s__;           \
  } while (0)

#define GRAM_LAUNCH_CHECK(ctx) GRAM_CUDA(ctx, cudaGetLastError())

// ---------------------------------------------------------------------------
// Launches.  A step is a chain of some hundred short kernels on one stream; with ordinary launches each waits for the one
// before it to drain, flush and retire and then pays its own start.  Every kernel here is launched with programmatic stream
// serialisation instead: its blocks are placed as soon as all blocks of the kernel before have ended, they set up what needs
// no memory of others, and chain_begin() then waits until that kernel's writes are visible.  (Ordinary launches -> this ->
// with an early trigger that lets blocks in while the kernel before still runs: the check's step 686 -> 532 -> 554 us, the
// task module at 25 600 rows 3.49 -> 3.40 -> 3.39 ms, encodings of 2048 ragged texts 2.86 -> 2.85 -> 2.92 ms: the blocks that
// wait on the SMs cost the large kernels more than they save, so there is no early trigger.)
// A kernel launched with launch_chain (or chain_attribute) must call chain_begin() before it touches global memory.
// It returns true; that the compiler cannot know it keeps loads that it takes to be of constant memory behind the wait.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool chain_begin() {
  uint32_t n;
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, %%nctaid.x;" : "=r"(n)::"memory");
  return n != 0u;
}
static inline cudaLaunchAttribute chain_attribute() {
  cudaLaunchAttribute a = {};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  return a;
}
// errors are left for the caller's GRAM_LAUNCH_CHECK
template <typename... P, typename... A>
static inline void launch_chain(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr = chain_attribute();
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

static inline int64_t ceil_div64(int64_t a, int64_t b) { return (a + b - 1) / b; }
static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// ---------------------------------------------------------------------------
// index / accumulation workspaces (dedup.cu, gather_accum.cu)
// ---------------------------------------------------------------------------
constexpr int kAccMaxChunks = 148 * 16;   // work units of the segmented sum
constexpr int kNumSMs = 148;

struct IndexWorkspace {
  int64_t P_max = 0;
  int32_t n_items_max = 0;
  int32_t d_max = 0;
  int32_t *keys0 = nullptr, *keys1 = nullptr, *vals0 = nullptr, *vals1 = nullptr;  // [P_max] radix ping-pong
  uint32_t* sort_ctl = nullptr;   // tile tickets, digit totals and per-tile status words of the sort (cleared per call)
  int32_t* rank_table = nullptr;  // [n_items_max] item ID -> index in unique
  float* partial = nullptr;       // [kAccMaxChunks * 2 * d_max] chunk-boundary partial sums, then kAccMaxChunks (item, last chunk) pairs
};

gram_status index_ws_alloc(gram_ctx* ctx, IndexWorkspace* ws, int64_t P_max, int32_t n_items_max, int32_t d_max);
void index_ws_free(IndexWorkspace* ws);
int32_t index_cluster_blocks();                      // asks the device; after index_ws_alloc

gram_status dedup_launch(gram_ctx* ctx, IndexWorkspace* ws, const int32_t* d_ids, int64_t P, int32_t n_items,
                         int32_t* d_unique, int32_t* d_inverse, int32_t* d_perm, int32_t* d_seg_off,
                         int32_t* d_n_unique, cudaStream_t st);

gram_status dedup_wait_selftest(gram_ctx* ctx, IndexWorkspace* ws, cudaStream_t st);

gram_status gather_launch(gram_ctx* ctx, const void* d_src, int64_t n_src_rows, const int32_t* d_index, int64_t P,
                          int32_t d, int elem_bytes, void* d_E, cudaStream_t st);

// out[r, :] = a[index[r], :] - b[index[r], :] (d_x == NULL), or d_x[r, :] - (a[index[r], :] - b[index[r], :]); fp32 rows.
// Multi-step with pseudo-targets: the first form is h~ = cache - table gathered into the positions (Eq. 6), the
// second the cotangent CE(c) - h~ of the pseudo-loss (Eq. 9).
gram_status gather_diff_launch(gram_ctx* ctx, const float* d_a, const float* d_b, int64_t n_src_rows, const int32_t* d_index,
                               int64_t n, int32_t d, const float* d_x, float* d_out, cudaStream_t st);

// d_E[p, :] (fp32) = d_src_bf16[d_index[p], :] (bf16 rows of d elements, d a multiple of 8): gather and widen in one pass
gram_status gather_widen_launch(gram_ctx* ctx, const void* d_src_bf16, int64_t n_src_rows, const int32_t* d_index, int64_t P,
                                int32_t d, float* d_E, cudaStream_t st);

// d_U (may be NULL): the number of segments is read from the device instead of U.
// d_rows (may be NULL): output row of segment u is d_rows[u] instead of u.  add != 0: out[row] += sum instead of out[row] = sum.  gated != 0: the kernels leave d_out alone
// when the context's status word already holds an error (a step that must not change state after a bad input).
gram_status accumulate_launch(gram_ctx* ctx, IndexWorkspace* ws, const float* d_in, const int32_t* d_perm,
                              const int32_t* d_seg_off, int64_t P, int32_t U, const int32_t* d_U, int32_t d,
                              const int32_t* d_rows, int add, float* d_out, cudaStream_t st, int gated = 0);

// sets bit d_unique[u] for u < U (U read from d_U when that is not NULL); d_count (may be NULL) counts the bits that
// were not set before; gated as above
gram_status touched_mark_launch(gram_ctx* ctx, const int32_t* d_unique, int32_t U, const int32_t* d_U, int32_t n_items,
                                uint32_t* d_bits, int32_t* d_count, int gated, cudaStream_t st);
gram_status touched_list_launch(gram_ctx* ctx, const uint32_t* d_bits, int32_t n_items, int32_t* d_list,
                                int32_t* d_count, cudaStream_t st);

// ---------------------------------------------------------------------------
// measurement: every launch wrapper opens a ProfScope.  It always counts the launches; when
// profiling is on it also brackets them with CUDA events on the launching stream and files the
// elapsed time and the algorithmic work (flops or bytes) under the kernel kind.
// ---------------------------------------------------------------------------
void gram_prof_open(gram_ctx* ctx, int kind, const char* tag, const char* tag2, double work, int launches, cudaStream_t st, int* slot);
void gram_prof_close(gram_ctx* ctx, int slot, cudaStream_t st);
struct ProfScope {
  gram_ctx* ctx;
  cudaStream_t st;
  int slot = -1;
  // tag: a string literal naming the call site (shown by gram_profile_dump); tag2: the other one of two equal shares of the work
  ProfScope(gram_ctx* c, int kind, double work, int launches, cudaStream_t s, const char* tag = nullptr, const char* tag2 = nullptr)
      : ctx(c), st(s) {
    gram_prof_open(c, kind, tag, tag2, work, launches, s, &slot);
  }
  ~ProfScope() { if (slot >= 0) gram_prof_close(ctx, slot, st); }
};

// All threads of a cluster meet.  The instructions take whole warps (.aligned): lanes that a test or a loop of their own sent
// different ways are brought together first.
__device__ __forceinline__ void gram_cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the device status word: kernels record the first error kind they meet
__device__ __forceinline__ void gram_device_fail(int32_t* status, int32_t code) { atomicCAS(status, 0, code); }
int32_t* gram_status_word(gram_ctx* ctx);
// the words that a step's host side reads lie together, the status word first: the number of unique items, the loss (fp32 bits), the
// number of touched items of the window
constexpr int STEP_STATUS = 0, STEP_UNIQUE = 1, STEP_LOSS = 2, STEP_TOUCHED = 3, kStepWords = 4;
int32_t gram_cluster_blocks(const gram_ctx* ctx);   // blocks of the largest cluster that can be placed: 16, 8, 4, 2 or 1
int32_t gram_ring_rows(const gram_ctx* ctx);   // rows a warp may take from a ring of bulk copies before it gives up; see gram_selftest_ring_rows
