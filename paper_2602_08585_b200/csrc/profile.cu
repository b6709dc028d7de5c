// Offline profile and online lookup (paper Sec. 4.3).
//   profile_mean_kernel     Eq. "calibration_avg": the profile entry of (ratio, head) is the mean over
//                           the calibration queries of the optimal local ratio r* = 1 - b/n, where b is
//                           the head's budget in that query's solution of the relaxed problem.
//   profile_budget_kernel   "Lookup" and "Budgeting": r = profile row at the target ratio (linear
//                           interpolation between the two neighbouring grid rows), b = floor((1-r)*n).
//   offsets_scan_kernel     packed-row offsets of the resulting budgets.
//   profile_lookup_kernel   the two in one launch of one CTA, for calls of up to 8192 heads (launches and their
//                           gaps are the cost there: 6 us from the first start to the last end as two, 4 us as one).
// All ratio arithmetic is fp64 with explicit round-to-nearest operations (no contraction), because a
// floor follows it: the integer must not depend on how the compiler fuses the expression.
#include "common.cuh"

namespace lukv {
namespace {

constexpr int kProfileThreads = 256;

// budgets: [n_queries][count] with count = R*N; profile: [count].  Eight threads per entry share the divisions (an fp64
// division is a chain of some 700 clocks; 30 of them in one thread took 15 us at 25344 entries, 5.7 us now); the first of
// them adds the terms in query order.
constexpr int kMeanThreadsPer = 8;

__global__ void profile_mean_kernel(const int32_t* __restrict__ budgets, float* __restrict__ profile, int n_queries,
                                    long long count, int n) {
  __shared__ double term[kProfileThreads / kMeanThreadsPer][kMeanThreadsPer + 1];
  constexpr int kEntries = kProfileThreads / kMeanThreadsPer;
  // consecutive threads take consecutive entries: coalesced reads
  const int slot = threadIdx.x % kEntries, part = threadIdx.x / kEntries;
  const long long e = (long long)blockIdx.x * kEntries + slot;
  const double dn = (double)n;
  double acc = 0.0;
  for (int i0 = 0; i0 < n_queries; i0 += kMeanThreadsPer) {
    const int i = i0 + part;
    if (i < n_queries && e < count)
      term[slot][part] = __dsub_rn(1.0, __ddiv_rn((double)__ldg(budgets + (size_t)i * count + e), dn));
    __syncthreads();
    if (part == 0)
      for (int t = 0; t < kMeanThreadsPer && i0 + t < n_queries; ++t) acc = __dadd_rn(acc, term[slot][t]);
    __syncthreads();
  }
  if (part == 0 && e < count) profile[e] = __double2float_rn(__ddiv_rn(acc, (double)n_queries));
}

struct LookupArgs {
  int row_lo[kLookupSeqPerLaunch];   // grid row at or below the target ratio
  int row_hi[kLookupSeqPerLaunch];   // the next row (== row_lo at the last grid point)
  double frac[kLookupSeqPerLaunch];  // position of the target between the two rows, in [0,1)
  int n[kLookupSeqPerLaunch];        // rankable positions of the sequence
  int floor_tok[kLookupSeqPerLaunch];  // its minimum retention in tokens
  int seq0;
};

__device__ __forceinline__ int32_t lookup_budget(const float* __restrict__ profile, const LookupArgs& args, int i, int hid,
                                                 int N) {
  const int n = args.n[i], floor_tok = args.floor_tok[i];
  const double r0 = (double)profile[(size_t)args.row_lo[i] * N + hid];
  const double r1 = (double)profile[(size_t)args.row_hi[i] * N + hid];
  const double r = __dadd_rn(r0, __dmul_rn(__dsub_rn(r1, r0), args.frac[i]));
  double b = floor(__dmul_rn(__dsub_rn(1.0, r), (double)n));
  b = b < 0.0 ? 0.0 : (b > (double)n ? (double)n : b);
  return max((int32_t)b, floor_tok);  // minimum retention (App. E)
}

// blockIdx.y = sequence of this launch, x covers the heads.
__global__ void profile_budget_kernel(const float* __restrict__ profile, const __grid_constant__ LookupArgs args, int N,
                                      int32_t* __restrict__ budgets) {
  const int hid = blockIdx.x * kProfileThreads + threadIdx.x;
  if (hid >= N) return;
  budgets[(size_t)(args.seq0 + blockIdx.y) * N + hid] = lookup_budget(profile, args, blockIdx.y, hid, N);
}

constexpr int kScanThreads = 1024;

// Exclusive scan over the CTA in thread order.
__device__ __forceinline__ long long cta_scan(long long v) {
  __shared__ long long warp_sums[kScanThreads / 32];
  const int tid = threadIdx.x;
  long long incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const long long o = __shfl_up_sync(0xffffffffu, incl, off);
    if ((tid & 31) >= off) incl += o;
  }
  if ((tid & 31) == 31) warp_sums[tid >> 5] = incl;
  __syncthreads();
  long long run = incl - v;
  for (int wv = 0; wv < (tid >> 5); ++wv) run += warp_sums[wv];
  return run;
}

// offsets[0] = 0, offsets[u+1] = sum_{v<=u} (budgets[v] + w).  One CTA; each thread owns a
// contiguous run of heads.
__global__ void __launch_bounds__(kScanThreads) offsets_scan_kernel(const int32_t* __restrict__ budgets,
                                                                    int32_t* __restrict__ offsets, int count, int w) {
  const int tid = threadIdx.x;
  const int per = (count + kScanThreads - 1) / kScanThreads;
  const int u0 = min(count, tid * per), u1 = min(count, u0 + per);
  long long local = 0;
  for (int u = u0; u < u1; ++u) local += budgets[u] + w;
  long long run = cta_scan(local);
  if (tid == 0) offsets[0] = 0;
  for (int u = u0; u < u1; ++u) {
    run += budgets[u] + w;
    offsets[u + 1] = (int32_t)run;
  }
}

constexpr int kLookupPer = 8;  // heads per thread of the one-CTA form

__global__ void __launch_bounds__(kScanThreads) profile_lookup_kernel(const float* __restrict__ profile,
                                                                      const __grid_constant__ LookupArgs args, int N, int count,
                                                                      int w, int32_t* __restrict__ budgets,
                                                                      int32_t* __restrict__ offsets) {
  const int per = (count + kScanThreads - 1) / kScanThreads, u0 = threadIdx.x * per;
  int32_t b[kLookupPer];
  long long local = 0;
#pragma unroll
  for (int i = 0; i < kLookupPer; ++i) {
    const int u = u0 + i;
    b[i] = 0;
    if (i < per && u < count) {
      b[i] = lookup_budget(profile, args, u / N, u % N, N);
      local += b[i] + w;
    }
  }
  long long run = cta_scan(local);
  if (threadIdx.x == 0) offsets[0] = 0;
#pragma unroll
  for (int i = 0; i < kLookupPer; ++i)
    if (i < per && u0 + i < count) {
      run += b[i] + w;
      budgets[u0 + i] = b[i];
      offsets[u0 + i + 1] = (int32_t)run;
    }
}

}  // namespace

cudaError_t launch_profile_mean(const int32_t* budgets, float* profile, int n_queries, int64_t count, int n,
                                LaunchCtx& lc) {
  const long long per = kProfileThreads / kMeanThreadsPer;
  const unsigned blocks = (unsigned)((count + per - 1) / per);
  profile_mean_kernel<<<blocks, kProfileThreads, 0, lc.st>>>(budgets, profile, n_queries, (long long)count, n);
  lc.mark("profile_mean");
  return cudaGetLastError();
}

cudaError_t launch_profile_budgets(const float* profile, const int* row_lo, const int* row_hi, const double* frac,
                                   const Dims& dm, int32_t* budgets, int32_t* offsets, LaunchCtx& lc) {
  const int S = dm.S, N = dm.N, w = dm.w;
  for (int q0 = 0; q0 < S; q0 += kLookupSeqPerLaunch) {
    LookupArgs args;
    const int cnt = S - q0 < kLookupSeqPerLaunch ? S - q0 : kLookupSeqPerLaunch;
    for (int i = 0; i < kLookupSeqPerLaunch; ++i) {
      args.row_lo[i] = i < cnt ? row_lo[q0 + i] : 0;
      args.row_hi[i] = i < cnt ? row_hi[q0 + i] : 0;
      args.frac[i] = i < cnt ? frac[q0 + i] : 0.0;
      args.n[i] = i < cnt ? seq_rankable(dm, q0 + i) : 0;
      args.floor_tok[i] = i < cnt ? seq_floor_tokens(dm, q0 + i) : 0;
    }
    args.seq0 = q0;
    if (cnt == S && (long long)S * N <= kScanThreads * kLookupPer) {
      profile_lookup_kernel<<<1, kScanThreads, 0, lc.st>>>(profile, args, N, S * N, w, budgets, offsets);
      lc.mark("profile_lookup");
      return cudaGetLastError();
    }
    profile_budget_kernel<<<dim3((N + kProfileThreads - 1) / kProfileThreads, cnt), kProfileThreads, 0, lc.st>>>(
        profile, args, N, budgets);
    lc.mark("profile_budget");
  }
  offsets_scan_kernel<<<1, kScanThreads, 0, lc.st>>>(budgets, offsets, S * N, w);
  lc.mark("offsets_scan");
  return cudaGetLastError();
}

}  // namespace lukv
