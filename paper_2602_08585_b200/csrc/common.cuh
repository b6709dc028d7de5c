// Internal declarations shared by the translation units of liblukv.so.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include "lukv.h"

namespace lukv {

// Problem sizes derived once from lukv_params_t (validated by the API layer).
struct Dims {
  int S, L, H, G, d, T, w, kp, dtype, P;
  int N;        // heads per sequence
  int n;        // rankable positions per head
  int M;        // score rows per head = G*w
  int seg;      // tokens per curve segment s = T/(P-1)
  int nseg;     // curve segments with non-zero capacity = ceil(n/seg)
  float scale_log2;  // softmax scale * log2(e): logits are kept in the exp2 domain
  int n_sink;        // leading positions that rank first in the selection
  int floor_tok;     // tokens every head keeps at least: ceil(min_keep * n)
  // Sequences of different lengths in one call: seq_T[q] (HOST, S entries) is the context length of sequence q;
  // T, n and the tensor strides then describe the longest one.  nullptr: every sequence has length T.
  const int32_t* seq_T = nullptr;
  float min_keep = 0.f;  // as given (the per-sequence floors of a ragged call are derived from it)
  bool keydiff = false;  // stage (a) is the KeyDiff metric (keys only, no pooling)
  int64_t heads() const { return (int64_t)S * N; }
  int raw_stride() const { return (n + 3) & ~3; }  // floats between the rows of the un-pooled scores: 16-byte rows
  size_t esize() const { return dtype == LUKV_DTYPE_BF16 ? 2 : 4; }
};

// The hull of every curve as a list of its blocks of equal gain, steepest first: row i of `gain` and `start` ([curves]
// [P-1]) holds count[i] entries, `start` the first curve segment of the block.
struct HullLists {
  float* gain;
  unsigned short* start;
  int* count;
};
HullLists hull_lists(void* base, int64_t n_curves, int P);
size_t hull_lists_bytes(int64_t n_curves, int P);

// Workspace carve-up (all offsets 256-byte aligned).
struct Workspace {
  float* raw;        // [S*N][raw_stride]  un-pooled scores
  float* pooled;     // [S*N][raw_stride]  pooled scores (whole path, where the selection does not pool)
  float* stats;      // partials per row: (reference, sum-exp) [S*N][chunks][M][2] (FP32-pipe scorer) or the
                     // log-sum-exp [S*N][items][128 or 256] (tensor-core scorer); pieces and anchors (KeyDiff)
  float* tc_stats;   // those of the two-sweep tensor-core scorer: `stats`, or for small calls, whose work items are more and
                     // smaller, from `pooled` on, which is not written before they have been read
  HullLists hull;    // blocks of equal gain of every head's curve
  int* head_flags;   // tensor-core scorer: [S*N] items delivered per head and the status word, then the (lse, tag) rows
  size_t bytes;
};

int score_chunks(const Dims& dm);                       // key chunks per head of the SIMT scorer
size_t score_tc_stats_bytes(const Dims& dm);            // pass-1 partials of the two-sweep tensor-core scorer
bool score_tc_small(const Dims& dm);                    // a call in items of two tiles; its partials:
size_t score_tc_small_stats_bytes(const Dims& dm);
size_t score_tc_flag_bytes(const Dims& dm);             // zero-initialised block: [heads] counters, status, then the (lse, tag) rows
inline int* score_tc_status(const Dims& dm, const Workspace& ws) { return ws.head_flags + dm.heads(); }
size_t score_tc_lse_offset(const Dims& dm);             // offset of the (lse, tag) rows inside that block
void score_test_hooks(uint32_t* spin_limit, int* drop_item);  // environment hooks for the timeout tests
// Single-sweep tensor-core scorer: takes a shape if a head's work items fit kOnePassMaxItems CTAs.
constexpr int kOnePassMaxItems = 128;
bool score_onepass_eligible(const Dims& dm);
size_t score_onepass_stats_bytes(const Dims& dm);       // its per-(row, key tile) partials; 0 if not eligible
Workspace carve_workspace(const Dims& dm, void* base);  // base may be null (size query)

// Heads per sequence the greedy kernel can hold: 12 bytes of shared memory each, 227 KB per CTA
// less its static arrays.
constexpr int kGreedyMaxHeads = 18944;

// Most sequences a call with per-sequence context lengths takes: their lengths travel by value in the launch
// arguments of the kernels.
constexpr int kMaxRaggedSeqs = 64;
struct SeqLens {
  int T[kMaxRaggedSeqs];
};

// Rankable positions and minimum retention (tokens) of sequence q: the call's own when all sequences have one
// length, else from its length (the floor is ceil(min_keep * n) in fp64, as in the uniform case).
inline int seq_rankable(const Dims& dm, int q) { return dm.seq_T ? dm.seq_T[q] - dm.w : dm.n; }
inline int seq_floor_tokens(const Dims& dm, int q) {
  if (!dm.seq_T) return dm.floor_tok;
  const int n = dm.seq_T[q] - dm.w;
  const double fl = ceil((double)dm.min_keep * (double)n);
  return fl < 0.0 ? 0 : (fl > (double)n ? n : (int)fl);
}

// Launch bookkeeping: counts the kernels a call enqueues and, when a timeline is attached
// (profiling entry point only), records a CUDA event after each of them.
struct LaunchCtx {
  cudaStream_t st = nullptr;
  int launches = 0;
  cudaEvent_t* events = nullptr;  // [max_events + 1]; events[0] is recorded by the caller
  const char** names = nullptr;   // [max_events]
  int max_events = 0;
  void mark(const char* name) {
    if (events && launches < max_events) {
      names[launches] = name;
      cudaEventRecord(events[launches + 1], st);
    }
    ++launches;
  }
};

// Programmatic dependent launch: a kernel launched with launch_pdl(..., overlap = true) may start while the kernel before
// it on the stream still runs; it touches nothing that kernel (or any before it) reads or writes until pdl_wait, which
// returns once they are complete.  Both are no-ops in an ordinary launch.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Maximum over the warp.
__device__ __forceinline__ float warp_max(float v) {
  float d;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(d) : "f"(v));
  return d;
}
template <typename Kernel, typename... Args>
inline cudaError_t launch_pdl(Kernel kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool overlap,
                              const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}
#endif

// Multiprocessors of the current device (looked up once per device).
cudaError_t device_sms(int* sms);
// Lets a kernel use `bytes` of dynamic shared memory (the attribute is set once per kernel and device, to the most it can
// have).
cudaError_t allow_smem(const void* kernel, size_t bytes);

// Launchers.  Each returns cudaGetLastError() after its launches.
// The first sweep may run beside a kernel launched just before it (overlap); it ends after that kernel.
cudaError_t launch_score_simt(const Dims& dm, const void* q, const void* k, const Workspace& ws, bool overlap, LaunchCtx& lc);
// Tensor-core scorer (bf16).  A bounded wait that runs out stores LUKV_ERR_TIMEOUT to score_tc_status().
// spare_sms: SMs the persistent grid leaves to kernels that run beside it
bool score_tc_supported(const Dims& dm);
cudaError_t launch_score_tc(const Dims& dm, const void* q, const void* k, const Workspace& ws, int spare_sms, LaunchCtx& lc);
// The single-sweep kernel alone; cudaErrorNotSupported (nothing launched) if the device has too few SMs for the shape.
cudaError_t launch_score_onepass(const Dims& dm, const void* q, const void* k, const Workspace& ws, int spare_sms,
                                 LaunchCtx& lc);
// raw [heads][raw_stride] -> pooled [heads][stride]
cudaError_t launch_pool(const Dims& dm, const float* raw, float* pooled, int stride, LaunchCtx& lc);
// Allocation of up to 32 heads (544 curve points, 128 sequences) in one launch.  With `beside` it may run beside the kernel
// launched just before it, whose results it does not touch; it ends after that kernel.
bool allocate_small(const Dims& dm);
cudaError_t launch_allocate_small(const Dims& dm, const float* curves, const int64_t* budgets_host, int32_t* budgets,
                                  int32_t* offsets, bool beside, LaunchCtx& lc);
// Any size: the above where it applies, else hull and greedy.
cudaError_t launch_allocate(const Dims& dm, const float* curves, const int64_t* budgets_host, const HullLists& lists,
                            int32_t* budgets, int32_t* offsets, LaunchCtx& lc);
// The two halves.  launch_hull treats its input as n_curves independent curves;
// launch_greedy solves n_sets curve sets (lists of n_sets * N curves) for the same dm.S budgets and
// writes budgets [n_sets][S][N] and offsets [n_sets][S*N+1].  one_cta: by a single CTA (n_sets == 1).
cudaError_t launch_hull(const float* curves, const HullLists& out, int64_t n_curves, int P, LaunchCtx& lc);
cudaError_t launch_greedy(const Dims& dm, const HullLists& lists, const int64_t* budgets_host, int32_t* budgets,
                          int32_t* offsets, int n_sets, bool one_cta, LaunchCtx& lc);
// Offline profile (mean of the local ratios) and online lookup + budgeting.
cudaError_t launch_profile_mean(const int32_t* budgets, float* profile, int n_queries, int64_t count, int n,
                                LaunchCtx& lc);
constexpr int kLookupSeqPerLaunch = 32;
cudaError_t launch_profile_budgets(const float* profile, const int* row_lo, const int* row_hi, const double* frac,
                                   const Dims& dm, int32_t* budgets, int32_t* offsets, LaunchCtx& lc);
// Curves of a proxy ranking: scores, importance [heads][n] -> curves [heads][P].
size_t curves_smem_bytes(int n, int P);
cudaError_t launch_build_curves(const Dims& dm, const float* scores, const float* importance, float* curves,
                                LaunchCtx& lc);
// KeyDiff proxy scores (key-only metric): scores [heads][stride]; scratch of keydiff_scratch_bytes().  A bounded wait that
// runs out stores LUKV_ERR_TIMEOUT to dev_status, or to keydiff_status() when that is null.
size_t keydiff_scratch_bytes(const Dims& dm);
int* keydiff_status(const Dims& dm, float* scratch);
cudaError_t launch_keydiff(const Dims& dm, const void* k, float* scores, int stride, float* scratch, int32_t* dev_status,
                           int spare_sms, LaunchCtx& lc);
// Value norms || v_j W_O^(g) ||_2 of the oracle importance on the tensor cores (bf16): vnorm [heads][G][n].  Here and in
// the attention part a bounded wait that runs out stores LUKV_ERR_TIMEOUT to status.
// left (or null: all): [heads][G][128-position tiles][4] a bit per position to compute.
bool value_norm_tc_supported(const Dims& dm);
cudaError_t launch_value_norm_tc(const Dims& dm, int d_model, const void* v, const void* w_o, float* vnorm,
                                 const uint32_t* left, int32_t* status, LaunchCtx& lc);
// The same through the Gram matrix of the projection; positions for which it is not sound are left to the kernel above (left:
// as many bytes as the importance has at most, where the form pays).
bool value_norm_gram_pays(const Dims& dm, int d_model, const void* w_o);
cudaError_t launch_value_norm_gram(const Dims& dm, int d_model, const void* v, const void* w_o, float* vnorm,
                                   uint32_t* left, int32_t* status, LaunchCtx& lc);
// Attention part of the oracle importance on the tensor cores (bf16, up to 8 query heads per KV head): needs the value
// norms, leaves the un-normalised importance; part: importance_tc_part_bytes() of scratch.
bool importance_tc_supported(const Dims& dm, int k_max);
size_t importance_tc_part_bytes(const Dims& dm, int k_max);
cudaError_t launch_importance_tc(const Dims& dm, int k_max, const void* q_dec, const void* k, const void* k_dec,
                                 const float* vnorm, float* part, float* importance, int32_t* status, LaunchCtx& lc);
// Oracle importance of Sec. 4.1 from decode queries, the cache and the output projection.
size_t importance_workspace_bytes(const Dims& dm, int k_max);
cudaError_t launch_importance(const Dims& dm, int k_max, int d_model, const void* q_dec, const void* k, const void* v,
                              const void* k_dec, const void* w_o, bool normalize, float* importance, void* ws,
                              LaunchCtx& lc);
// Exact allocation (dynamic programme over the heads) at token resolution.
size_t exact_workspace_bytes(const Dims& dm, int64_t max_budget);
cudaError_t launch_exact_allocate(const Dims& dm, const float* curves, const int64_t* budgets_host, int32_t* budgets,
                                  int32_t* offsets, double* values, void* ws, LaunchCtx& lc);
// Selection from scores [heads][stride]; with `pool` the scores are max-pooled on the way in (select_pools() sizes).
// status: the scorer's status word, copied to dev_status (both may be null).  overlap: launched as the programmatic
// dependent of the kernel before it.
bool select_pools(const Dims& dm);
cudaError_t launch_select(const Dims& dm, const float* scores, int stride, bool pool, const int32_t* budgets,
                          const int32_t* offsets, int32_t* kept_idx, int64_t rows_cap, const int* status,
                          int32_t* dev_status, bool overlap, LaunchCtx& lc);
cudaError_t launch_gather(const Dims& dm, const int32_t* offsets, const int32_t* kept_idx, const void* k,
                          const void* v, void* k_out, void* v_out, int64_t rows_cap, bool overlap, LaunchCtx& lc);

}  // namespace lukv
