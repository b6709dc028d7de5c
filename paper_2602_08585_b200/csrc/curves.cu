// Utility-versus-budget curves of a proxy metric (paper Sec. 3.2: M^pi(k) = the first k positions in the
// ranking of pi; Eq. "head_loss_def": the loss of a retained set is the oracle importance outside it).
// The curve point U(k) is the importance mass of the k highest-ranked positions.  One CTA per head:
//   rank    the order is: sinks first, score descending, lower position first among equals.  Up to 16384
//           positions (the calibration contexts this serves have a few thousand): the scores are dealt into
//           buckets that follow their order, and a position's rank is its bucket's offset plus the entries of the
//           bucket that go before it.  Longer heads: every position's rank by counting the positions ahead of it
//           (O(n^2) compares on keys held in shared memory).  Ranks are unique either way;
//   sum     the importance goes to its rank's slot; fp64 prefix sums over the slots (a thread adds consecutive
//           ones, then warp and CTA scans) give the curve points, each rounded once to fp32.
#include "common.cuh"

namespace lukv {
namespace {

constexpr int kCurveThreads = 1024;
constexpr int kCurvePer = 4;  // positions ranked together by a thread (one key load serves all of them)

__device__ __forceinline__ uint32_t curve_key(float x, int j, int n_sink) {
  if (j < n_sink) return 0xFFFFFFFFu;
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);  // order-preserving map float -> uint32
}

// Curve points from the importance in ranking order: one thread per curve segment adds its slots in fp64, in
// order; warp 0 then runs the sum over the segments.  Call with the whole CTA, after a barrier behind the writes of
// `sorted`.
__device__ __forceinline__ void curve_tail(const float* sorted, double* segsum, float* out, int n, int P, int seg,
                                           int tid, int nthreads) {
  const int nseg = P - 1;
  for (int k = tid; k < nseg; k += nthreads) {
    const long long lo = (long long)k * seg, hi = lo + seg;
    const int a = (int)(lo < n ? lo : n), b = (int)(hi < n ? hi : n);
    double acc = 0.0;
    for (int i = a; i < b; ++i) acc = __dadd_rn(acc, (double)sorted[i]);
    segsum[k] = acc;
  }
  __syncthreads();
  // running sum over the segments: warp 0, 32 consecutive segments per step
  if (tid < 32) {
    if (tid == 0) out[0] = 0.f;
    double carry = 0.0;
    for (int k0 = 0; k0 < nseg; k0 += 32) {
      const int k = k0 + tid;
      double v = k < nseg ? segsum[k] : 0.0;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, v, off);
        if (tid >= off) v = __dadd_rn(v, o);
      }
      v = __dadd_rn(v, carry);
      if (k < nseg) out[k + 1] = __double2float_rn(v);
      carry = __shfl_sync(0xffffffffu, v, 31);
    }
  }
}

__global__ void __launch_bounds__(kCurveThreads) build_curves_kernel(const float* __restrict__ scores,
                                                                     const float* __restrict__ importance,
                                                                     float* __restrict__ curves, int n, int P,
                                                                     int seg, int n_sink) {
  extern __shared__ __align__(16) unsigned char curve_smem[];
  const int npad = (n + 3) & ~3;
  uint32_t* keys = reinterpret_cast<uint32_t*>(curve_smem);             // [npad], padding = 0 (ranks last)
  float* sorted = reinterpret_cast<float*>(curve_smem) + npad;          // [npad] importance in ranking order
  double* segsum = reinterpret_cast<double*>(sorted + npad + (npad & 1));  // [P-1], 8-byte aligned
  const int u = blockIdx.x, tid = threadIdx.x;
  const float* sc = scores + (size_t)u * n;
  const float* im = importance + (size_t)u * n;
  for (int j = tid; j < npad; j += kCurveThreads) keys[j] = j < n ? curve_key(sc[j], j, n_sink) : 0u;
  __syncthreads();

  for (int j0 = tid * kCurvePer; j0 < n; j0 += kCurveThreads * kCurvePer) {
    uint32_t mine[kCurvePer];
    int rank[kCurvePer];
#pragma unroll
    for (int i = 0; i < kCurvePer; ++i) {
      mine[i] = j0 + i < n ? keys[j0 + i] : 0u;
      rank[i] = 0;
    }
    // positions ahead of j: a larger key, or an equal key at a lower position
    for (int c = 0; c < npad; c += 4) {
      const uint4 k4 = *reinterpret_cast<const uint4*>(keys + c);
      const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int i = 0; i < kCurvePer; ++i)
#pragma unroll
        for (int t = 0; t < 4; ++t)
          rank[i] += (kk[t] > mine[i]) || (kk[t] == mine[i] && c + t < j0 + i);
    }
#pragma unroll
    for (int i = 0; i < kCurvePer; ++i)
      if (j0 + i < n) sorted[rank[i]] = im[j0 + i];
  }
  __syncthreads();

  curve_tail(sorted, segsum, curves + (size_t)u * P, n, P, seg, tid, kCurveThreads);
}

constexpr int kSortMaxN = 16384;   // positions (rounded up to a power of two) the bucket kernel takes
constexpr int kBucketLimit = 64;   // entries of one bucket up to which ranking inside it beats sorting

// Where a bucket's word lies: threads that read 2 EPT consecutive ones, 16 bytes at a time, hit all banks.
__device__ __forceinline__ uint32_t bucket_place(uint32_t b) { return b ^ ((b >> 5 & 7) << 2); }

// npow2 / EPT threads; a thread owns EPT positions (tid + t * threads) while ranking and EPT consecutive ranks while
// summing.  A bucket is a stretch of 2^sh keys, at most 2 npow2 buckets cover the range of the head's keys; float keys are
// logarithmic, which spreads scores over orders of magnitude evenly: the fullest buckets of a log-normal distribution hold
// some five positions.  Inside a bucket the lower sh bits of the key and the inverted position, together at most 32 bits,
// decide the order in one comparison.  Should a bucket hold more than kBucketLimit entries (long runs of equal scores), the
// CTA sorts 64-bit keys instead (bitonic).
// Bound by shared-memory wavefronts (the random accesses to buckets and ranks) and issue slots.  30 queries x 256 heads x 3968
// positions: 1.94 ms for the bitonic sort of every head with sums by one warp; 285 us with four 16-bit buckets a position, whose
// reading by threads hit four times the same bank and took half the instructions, and all of a thread's positions compared as
// far as the fullest bucket of all; 221 so.  2560 heads of 2084 positions 84 and 57 us, 512 of 8968 119 and 62.
template <int EPT>
__global__ void __launch_bounds__(EPT == 8 ? 512 : 1024, EPT == 8 ? 3 : 1)
    build_curves_bucket_kernel(const float* __restrict__ scores, const float* __restrict__ importance,
                               float* __restrict__ curves, int n, int npow2, int P, int seg, int n_sink) {
  extern __shared__ __align__(16) unsigned char curve_smem[];
  uint32_t* local_key = reinterpret_cast<uint32_t*>(curve_smem);                  // [npow2], bucket by bucket
  uint32_t* words = local_key + npow2;                                           // [2 npow2], a bucket each, see bucket_place
  unsigned long long* comp = reinterpret_cast<unsigned long long*>(curve_smem);  // [npow2], when sorting
  float* sorted = reinterpret_cast<float*>(curve_smem);                           // [npow2], once the ranks are known
  __shared__ uint32_t red[2][32];
  __shared__ int scan[32], most_s[32];
  __shared__ double sums[32];
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, wv = tid >> 5, warps = nthr >> 5;
  const float* sc = scores + (size_t)blockIdx.x * n;
  const float* im = importance + (size_t)blockIdx.x * n;
  float* out = curves + (size_t)blockIdx.x * P;

  uint32_t key[EPT];
  float val[EPT];
  {
    float x[EPT];
#pragma unroll
    for (int t = 0; t < EPT; ++t) x[t] = __ldg(sc + min(tid + t * nthr, n - 1));  // no branches: all loads in flight
#pragma unroll
    for (int t = 0; t < EPT; ++t) val[t] = __ldg(im + min(tid + t * nthr, n - 1));
#pragma unroll
    for (int t = 0; t < EPT; ++t) key[t] = curve_key(x[t], tid + t * nthr, n_sink);
  }
#pragma unroll
  for (int i = 0; i < EPT / 2; ++i) reinterpret_cast<uint4*>(words)[tid + i * nthr] = make_uint4(0u, 0u, 0u, 0u);
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;  // range of the scored positions' keys
#pragma unroll
  for (int t = 0; t < EPT; ++t) {
    const int j = tid + t * nthr;
    if (j < n && j >= n_sink) {
      lo = min(lo, key[t]);
      hi = max(hi, key[t]);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    red[0][wv] = lo;
    red[1][wv] = hi;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, lane < warps ? red[0][lane] : 0xFFFFFFFFu);
  hi = __reduce_max_sync(0xffffffffu, lane < warps ? red[1][lane] : 0u);
  const int pos_bits = 31 - __clz(npow2);
  const int sh = max(0, 32 - __clz(hi > lo ? hi - lo : 0u) - pos_bits - 1);  // (hi - lo) >> sh is below 2 npow2
  const uint32_t top = hi > lo ? (hi - lo) >> sh : 0u, low_mask = (1u << sh) - 1u;
  uint32_t mine[EPT];
  uint32_t where[EPT];  // place of the bucket << 16 | slot in it; bucket 0 holds the largest keys
#pragma unroll
  for (int t = 0; t < EPT; ++t) {
    const int j = tid + t * nthr;
    where[t] = 0;
    if (j < n) {
      const bool sink = j < n_sink;  // before everything else: they have the lowest positions
      const uint32_t off = key[t] - lo;
      const uint32_t place = bucket_place(sink ? 0u : top - (off >> sh));
      mine[t] = ((sink ? low_mask : off & low_mask) << pos_bits) | (uint32_t)(npow2 - 1 - j);
      where[t] = (place << 16) | atomicAdd(words + place, 1u);
    }
  }
  __syncthreads();
  // exclusive offsets of the buckets; the fullest one
  auto own = [&](int i) { return reinterpret_cast<uint4*>(words + bucket_place((uint32_t)(tid * 2 * EPT + 4 * i))); };
  int local = 0, most = 0;  // a thread has 2 EPT buckets
#pragma unroll
  for (int i = 0; i < EPT / 2; ++i) {
    const uint4 c = *own(i);
    local += (int)((c.x + c.y) + (c.z + c.w));
    most = max(most, (int)max(max(c.x, c.y), max(c.z, c.w)));
  }
  int incl = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 31) scan[wv] = incl;
  if (lane == 0) most_s[wv] = most;
  __syncthreads();
  int run = __reduce_add_sync(0xffffffffu, lane < wv ? scan[lane] : 0) + incl - local;
  most = __reduce_max_sync(0xffffffffu, lane < warps ? most_s[lane] : 0);
  // a bucket's word: where its entries start << 16 | their number
  uint32_t at = (uint32_t)run;
#pragma unroll
  for (int i = 0; i < EPT / 2; ++i) {
    const uint4 c = *own(i);
    const uint32_t a1 = at + c.x, a2 = a1 + c.y, a3 = a2 + c.z;
    *own(i) = make_uint4(at << 16 | c.x, a1 << 16 | c.y, a2 << 16 | c.z, a3 << 16 | c.w);
    at = a3 + c.w;
  }
  __syncthreads();

  int rank[EPT];
  if (most <= kBucketLimit) {
#pragma unroll
    for (int t = 0; t < EPT; ++t)
      if (tid + t * nthr < n) {
        const uint32_t word = words[where[t] >> 16];
        local_key[(word >> 16) + (where[t] & 0xFFFFu)] = mine[t];
        where[t] = word;
      }
    __syncthreads();
    // Most buckets hold one entry: position by position, as far as the fullest of the warp's 32 buckets.
#pragma unroll
    for (int t = 0; t < EPT; ++t) {
      const int left = (int)(where[t] & 0xFFFFu), longest = __reduce_max_sync(0xffffffffu, left);
      const uint32_t* entries = local_key + (where[t] >> 16);
      rank[t] = (int)(where[t] >> 16);
      if (longest > 1) {
#pragma unroll 1
        for (int x = 0; x < longest; x += 2) {
          if (x < left) rank[t] += entries[x] > mine[t];
          if (x + 1 < left) rank[t] += entries[x + 1] > mine[t];
        }
      }
    }
  } else {
#pragma unroll
    for (int t = 0; t < EPT; ++t) {
      const int j = tid + t * nthr;
      comp[j] = j < n ? ((unsigned long long)curve_key(__ldg(sc + j), j, n_sink) << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)j)
                      : 0ull;
    }
    __syncthreads();
    const int pairs = npow2 >> 1;
    for (int k = 2; k <= npow2; k <<= 1) {
      for (int j = k >> 1, lj = 31 - __clz(j); j > 0; j >>= 1, --lj) {
        for (int t = tid; t < pairs; t += nthr) {
          const int a = ((t >> lj) << (lj + 1)) + (t & (j - 1)), b = a + j;
          const unsigned long long x = comp[a], y = comp[b];
          const bool descending = (a & k) == 0;
          if ((x < y) == descending) {
            comp[a] = y;
            comp[b] = x;
          }
        }
        __syncthreads();
      }
    }
#pragma unroll
    for (int t = 0; t < EPT; ++t) {
      const int r = tid + t * nthr;
      rank[t] = r;
      if (r < n) val[t] = __ldg(im + (0xFFFFFFFFu - (uint32_t)comp[r]));
    }
  }
  __syncthreads();  // comp is read: its place takes the importance in ranking order
#pragma unroll
  for (int t = 0; t < EPT; ++t)
    if (tid + t * nthr < n) sorted[rank[t]] = val[t];
    else sorted[tid + t * nthr] = 0.f;
  __syncthreads();

  // inclusive prefix sums in fp64, rounded once, in place
  float4* slots = reinterpret_cast<float4*>(sorted + tid * EPT);
  double acc[EPT];
#pragma unroll
  for (int q = 0; q < EPT / 4; ++q) {
    const float4 v = slots[q];
    acc[4 * q] = (double)v.x, acc[4 * q + 1] = (double)v.y, acc[4 * q + 2] = (double)v.z, acc[4 * q + 3] = (double)v.w;
  }
#pragma unroll
  for (int t = 1; t < EPT; ++t) acc[t] = __dadd_rn(acc[t - 1], acc[t]);
  double tot = acc[EPT - 1];
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const double o = __shfl_up_sync(0xffffffffu, tot, off);
    if (lane >= off) tot = __dadd_rn(tot, o);
  }
  if (lane == 31) sums[wv] = tot;
  double before = __shfl_up_sync(0xffffffffu, tot, 1);
  if (lane == 0) before = 0.0;
  __syncthreads();
  if (wv == 0) {
    double v = lane < warps ? sums[lane] : 0.0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const double o = __shfl_up_sync(0xffffffffu, v, off);
      if (lane >= off) v = __dadd_rn(v, o);
    }
    if (lane < warps) sums[lane] = v;
  }
  __syncthreads();
  if (wv > 0) before = __dadd_rn(before, sums[wv - 1]);
#pragma unroll
  for (int q = 0; q < EPT / 4; ++q)
    slots[q] = make_float4(__double2float_rn(__dadd_rn(before, acc[4 * q])), __double2float_rn(__dadd_rn(before, acc[4 * q + 1])),
                          __double2float_rn(__dadd_rn(before, acc[4 * q + 2])),
                          __double2float_rn(__dadd_rn(before, acc[4 * q + 3])));
  __syncthreads();
  for (int k = tid; k < P; k += nthr) out[k] = k == 0 ? 0.f : sorted[min(k * seg, n) - 1];
}

int curve_pow2(int n) {
  int p = 2;
  while (p < n) p <<= 1;
  return p;
}
// The bucket kernel runs with eight positions per thread, sixteen beyond 4096.
int bucket_pow2(int n) { return curve_pow2(n < 512 ? 512 : n); }
size_t curves_bucket_smem_bytes(int n) { return (size_t)bucket_pow2(n) * 12 + 16; }

}  // namespace

size_t curves_smem_bytes(int n, int P) {
  if (curve_pow2(n) <= kSortMaxN) return curves_bucket_smem_bytes(n);
  const size_t npad = ((size_t)n + 3) & ~(size_t)3;
  return (2 * npad + (npad & 1)) * 4 + (size_t)(P - 1) * 8;
}

cudaError_t launch_build_curves(const Dims& dm, const float* scores, const float* importance, float* curves,
                                LaunchCtx& lc) {
  const size_t smem = curves_smem_bytes(dm.n, dm.P);
  cudaError_t e;
  if (curve_pow2(dm.n) <= kSortMaxN) {
    const int np = bucket_pow2(dm.n);
    auto kern = np <= 4096 ? build_curves_bucket_kernel<8> : build_curves_bucket_kernel<16>;
    if ((e = allow_smem((const void*)kern, smem)) != cudaSuccess) return e;
    kern<<<(unsigned)dm.heads(), np <= 4096 ? np / 8 : np / 16, smem, lc.st>>>(
        scores, importance, curves, dm.n, np, dm.P, dm.seg, dm.n_sink);
    lc.mark("build_curves_bucket");
    return cudaGetLastError();
  }
  if ((e = allow_smem((const void*)build_curves_kernel, smem)) != cudaSuccess) return e;
  build_curves_kernel<<<(unsigned)dm.heads(), kCurveThreads, smem, lc.st>>>(scores, importance, curves, dm.n, dm.P,
                                                                            dm.seg, dm.n_sink);
  lc.mark("build_curves");
  return cudaGetLastError();
}

}  // namespace lukv
