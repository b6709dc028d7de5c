// Stages (c) and (d): per-head variable-k top-k selection and the packed gather.
//   select_kernel  one CTA per head, or a thread-block cluster of 2, 4 or 8 CTAs per head that merge their
//                  histograms and counts through distributed shared memory (long contexts): max-pools the
//                  scores on the way in, finds the b-th largest over the order-preserving integer image of
//                  the scores by a histogram of the head's own key range and a ranking of the few keys in
//                  the bin that holds it, and emits the kept positions in ascending order: everything above
//                  the threshold plus the first (lowest-position) ties.  This realises M^pi(b) of Sec. 3.2 /
//                  the "Eviction" step of Sec. 4.3 without a full sort.
//   select_stream_kernel  the same for contexts beyond eight CTAs' registers: one CTA per head that re-reads
//                  its keys in every round.
//   gather_kernel  copies the kept K/V rows into the packed cache, 16 bytes per lane.
#include <cooperative_groups.h>

#include "common.cuh"

namespace lukv {
namespace {

namespace cg = cooperative_groups;

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;

// Order-preserving map float -> uint32 (larger float <=> larger key).
__device__ __forceinline__ uint32_t score_key(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Key of position j: attention sinks (the first n_sink positions, App. E) get the largest key, so
// they rank before every scored position; among themselves the lower position wins like any tie.
__device__ __forceinline__ uint32_t key_at(const float* src, int j, int n_sink) {
  return j < n_sink ? 0xFFFFFFFFu : score_key(src[j]);
}

struct SelectArgs {
  const float* scores;      // [heads][stride], un-pooled when half > 0
  const int32_t* budgets;
  const int32_t* offsets;
  int32_t* kept_idx;
  long long rows_cap;
  int stride;               // floats between the rows of two heads
  int n, w;                 // rankable positions (of the longest sequence), window
  int half;                 // max-pool over [j - half, j + half], 0..4
  int vec;                  // rows start on 16-byte boundaries and are readable up to a multiple of 4 floats
  int n_sink;
  int heads_per_seq;        // > 0: sequences of different lengths, sl.T
  const int* status;        // the scorer's status word, copied to dev_status (null: 0)
  int32_t* dev_status;      // may be null
  SeqLens sl;
};

constexpr int kSelBins = 2048;
constexpr int kSelCands = 512;  // keys of one bin that are ranked directly

// One CTA per head (CLUSTER false) or one cluster of CTAs per head (CLUSTER true; CTA r of the cluster owns the
// positions [r*P, (r+1)*P), P = 4 V positions per thread).  A thread keeps 4 V pooled keys in registers: vector e of a
// warp's V holds four consecutive positions per lane, so loads are coalesced and position order is (CTA, warp, e, lane,
// element).
// The threshold: bins are stretches of the head's own key range [smallest, largest], so the first histogram already
// spreads the keys (a float key is logarithmic: scores over orders of magnitude fill the bins evenly, and a bin holds some
// n / 700 keys at the densest), and the keys of the bin that holds the b-th largest are ranked among themselves; a bin
// with more than kSelCands keys is split again.
// Bound by instruction issue and the latency of its phases: 256 heads x 32736 positions in two waves of CTAs took 13 us for
// a pooling pass and 43 us with three histograms of fixed 11-, 11- and 10-bit digits, 49 us pooled in place; 112 heads x
// 131040 positions in clusters of four 20 + 128 us, 99 us now.
template <int V, bool CLUSTER>
__global__ void __launch_bounds__(kSelThreads, 1) select_kernel(const __grid_constant__ SelectArgs a) {
  __shared__ int hist[kSelBins];
  __shared__ uint32_t red[2][kSelWarps];
  __shared__ int scan_gt[kSelWarps], scan_eq[kSelWarps];
  __shared__ int sel[3];                            // bin, keys still wanted in it, keys in it
  __shared__ uint32_t cand[kSelCands], cand_all[CLUSTER ? kSelCands : 1];
  __shared__ int cand_n, cta_tot[2];                // cta_tot: keys of this CTA above / equal to the threshold
  __shared__ uint32_t found[2];                     // threshold, ties to keep
  cg::cluster_group cluster = cg::this_cluster();
  const int csize = CLUSTER ? (int)cluster.num_blocks() : 1, crank = CLUSTER ? (int)cluster.block_rank() : 0;
  const int nthr = blockDim.x, warps = nthr >> 5;
  const int u = (int)blockIdx.x / csize, tid = threadIdx.x, lane = tid & 31, wv = tid >> 5;
  auto sync = [&] {
    if (CLUSTER) cluster.sync(); else __syncthreads();
  };
  pdl_launch_dependents();
  pdl_wait();
  if (a.dev_status && blockIdx.x == 0 && tid == 0) *a.dev_status = a.status ? *a.status : 0;
  const int b = a.budgets[u];
  const long long off = a.offsets[u];
  const int n = a.heads_per_seq > 0 ? a.sl.T[u / a.heads_per_seq] - a.w : a.n;
  const float* src = a.scores + (size_t)u * a.stride;
  int32_t* out = a.kept_idx + off;
  const long long room = a.rows_cap - off;  // rows of this head that fit in the output

  // window rows follow the selected ones
  if (crank == 0)
    for (int t = tid; t < a.w; t += nthr)
      if (b + t < room) out[b + t] = n + t;
  if (b <= 0) return;  // the whole cluster leaves

  // ---- keys of this thread's positions: key 0 is no position, sinks get the largest key
  const int quad0 = (crank * warps + wv) * V * 32 + lane;  // first group of four positions
  uint32_t key[4 * V];
  {
    auto load4 = [&](int quad, float (&x)[4]) {  // -inf outside [0, n)
      const int j = 4 * quad;
      if (a.vec) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(src) + min(max(quad, 0), (n - 1) >> 2));
        x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __ldg(src + min(max(j + i, 0), n - 1));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if ((unsigned)(j + i) >= (unsigned)n) x[i] = -INFINITY;
    };
    float mid[V][4], before[4], behind[4];
#pragma unroll
    for (int e = 0; e < V; ++e) load4(quad0 + 32 * e, mid[e]);
    if (a.half > 0) {  // the groups next to the warp's own; those in between come from the neighbouring lanes
      load4(quad0 - lane - 1, before);
      load4(quad0 - lane + 32 * V, behind);
    }
#pragma unroll
    for (int e = 0; e < V; ++e) {
      float y[4] = {mid[e][0], mid[e][1], mid[e][2], mid[e][3]};
      if (a.half > 0) {
        float x[12];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          x[4 + i] = y[i];
          // lane 31 stands in for the lane before lane 0, lane 0 for the one behind lane 31
          const float l = __shfl_sync(0xffffffffu, lane == 31 && e > 0 ? mid[e > 0 ? e - 1 : 0][i] : y[i], (lane + 31) & 31);
          const float r = __shfl_sync(0xffffffffu, lane == 0 && e + 1 < V ? mid[e + 1 < V ? e + 1 : 0][i] : y[i], (lane + 1) & 31);
          x[i] = lane == 0 && e == 0 ? before[i] : l;
          x[8 + i] = lane == 31 && e == V - 1 ? behind[i] : r;
        }
#pragma unroll
        for (int d = 1; d <= 4; ++d)
          if (d <= a.half)
#pragma unroll
            for (int i = 0; i < 4; ++i) y[i] = fmaxf(y[i], fmaxf(x[4 + i - d], x[4 + i + d]));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = 4 * (quad0 + 32 * e) + i;
        // scored positions keep off the two marks, whatever the score (a NaN may be either): a head emits b rows
        key[4 * e + i] = j >= n ? 0u : j < a.n_sink ? 0xFFFFFFFFu : min(max(score_key(y[i]), 1u), 0xFFFFFFFEu);
      }
    }
  }

  // ---- b-th largest key
  uint32_t thr = 0xFFFFFFFFu;
  int k_eq = b;  // ties at the threshold to keep
  const int sinks = min(a.n_sink, n);
  if (b > sinks) {
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int i = 0; i < 4 * V; ++i)
      if (key[i] - 1u < 0xFFFFFFFEu) {  // neither no position nor a sink
        lo = min(lo, key[i]);
        hi = max(hi, key[i]);
      }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      red[0][wv] = lo;
      red[1][wv] = hi;
    }
    sync();
    lo = 0xFFFFFFFFu, hi = 0u;
    for (int c = 0; c < csize; ++c) {
      const uint32_t* r0 = CLUSTER ? cluster.map_shared_rank(&red[0][0], c) : &red[0][0];
      if (lane < warps) {
        lo = min(lo, r0[lane]);
        hi = max(hi, r0[kSelWarps + lane]);
      }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    int want = b - sinks;
#pragma unroll 1
    for (;;) {
      const int sh = max(0, 32 - __clz(hi - lo) - 11);  // (hi - lo) >> sh is below kSelBins
      for (int i = tid; i < kSelBins; i += nthr) hist[i] = 0;
      if (tid == 0) {
        cand_n = 0;
        sel[0] = 0, sel[1] = want, sel[2] = 0;
        found[0] = 0xFFFFFFFFu, found[1] = 0u;
      }
      __syncthreads();
      const uint32_t width = hi - lo;
#pragma unroll
      for (int i = 0; i < 4 * V; ++i)
        if (key[i] - lo <= width) atomicAdd(&hist[(key[i] - lo) >> sh], 1);
      sync();  // every histogram of the head is complete
      // a thread owns `per` bins, added over the CTAs of the head (every CTA computes the same); sums from the top
      const int per = kSelBins / nthr;  // 2, 4 or 8
      int mine = 0;
      for (int i = 0; i < per; ++i)
        for (int c = 0; c < csize; ++c) mine += (CLUSTER ? cluster.map_shared_rank(hist, c) : hist)[tid * per + i];
      int incl = mine;  // sum over the lanes >= this one
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += x;
      }
      if (lane == 0) scan_gt[wv] = incl;
      __syncthreads();
      const int higher = __reduce_add_sync(0xffffffffu, lane > wv && lane < warps ? scan_gt[lane] : 0) + incl - mine;
      if (higher < want && want <= higher + mine) {  // exactly one thread: the bin is among its own
        int run = higher;
        for (int i = per - 1; i >= 0; --i) {
          int c = 0;
          for (int r = 0; r < csize; ++r) c += (CLUSTER ? cluster.map_shared_rank(hist, r) : hist)[tid * per + i];
          if (want <= run + c) {
            sel[0] = tid * per + i;
            sel[1] = want - run;
            sel[2] = c;
            break;
          }
          run += c;
        }
      }
      sync();  // the histograms may be cleared again
      lo += (uint32_t)sel[0] << sh;
      hi = lo + min(hi - lo, (1u << sh) - 1u);
      want = sel[1];
      const int cnt = sel[2];
      if (sh == 0) {
        thr = lo;
        k_eq = want;
        break;
      }
      if (cnt <= kSelCands) {
        const uint32_t span = hi - lo;
        uint32_t in = 0;
#pragma unroll
        for (int i = 0; i < 4 * V; ++i) in |= key[i] - lo <= span ? 1u << i : 0u;
        if (in) {  // few threads
          int at = atomicAdd(&cand_n, __popc(in));
#pragma unroll
          for (int i = 0; i < 4 * V; ++i)
            if ((in >> i) & 1u) cand[at++] = key[i];
        }
        sync();
        const uint32_t* list = cand;
        if (CLUSTER) {
          int at = 0;
          for (int c = 0; c < csize; ++c) {
            const int m = *cluster.map_shared_rank(&cand_n, c);
            const uint32_t* from = cluster.map_shared_rank(cand, c);
            for (int i = tid; i < m; i += nthr) cand_all[at + i] = from[i];
            at += m;
          }
          list = cand_all;
          __syncthreads();
        }
        // eight lanes per candidate count the larger and the equal ones
        for (int i0 = 0; i0 < cnt; i0 += nthr >> 3) {
          const int i = i0 + (tid >> 3);
          const uint32_t me = i < cnt ? list[i] : 0u;
          uint32_t c = 0;
          for (int x = tid & 7; x < cnt; x += 8) {
            const uint32_t o = list[x];
            c += (o > me ? 1u : 0u) + (o == me ? 0x10000u : 0u);
          }
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
          const int larger = (int)(c & 0xFFFFu), equal = (int)(c >> 16);
          if (i < cnt && larger < want && want <= larger + equal) {  // one key; all that hold it write the same
            found[0] = me;
            found[1] = (uint32_t)(want - larger);
          }
        }
        __syncthreads();
        thr = found[0];
        k_eq = (int)found[1];
        break;
      }
      __syncthreads();  // every thread has read sel: the next split writes it
    }
  }

  // ---- keys above and equal to the threshold, one bit each; per-warp totals, then an exclusive scan over warps
  uint32_t kept = 0, tied = 0;
#pragma unroll
  for (int i = 0; i < 4 * V; ++i) {
    kept |= key[i] > thr ? 1u << i : 0u;
    tied |= key[i] == thr ? 1u << i : 0u;
  }
  const uint32_t both = __reduce_add_sync(0xffffffffu, __popc(kept) | (__popc(tied) << 16));  // at most 1024 of each
  if (lane == 0) {
    scan_gt[wv] = (int)(both & 0xFFFFu);
    scan_eq[wv] = (int)(both >> 16);
  }
  __syncthreads();
  int run_gt = __reduce_add_sync(0xffffffffu, lane < wv ? scan_gt[lane] : 0);
  int run_eq = __reduce_add_sync(0xffffffffu, lane < wv ? scan_eq[lane] : 0);
  if (CLUSTER) {
    // the CTAs before this one along the positions come first
    if (wv == 0) {
      const int g = __reduce_add_sync(0xffffffffu, lane < warps ? scan_gt[lane] : 0);
      const int q = __reduce_add_sync(0xffffffffu, lane < warps ? scan_eq[lane] : 0);
      if (lane == 0) {
        cta_tot[0] = g;
        cta_tot[1] = q;
      }
    }
    cluster.sync();
    for (int c = 0; c < crank; ++c) {
      const int* tot = cluster.map_shared_rank(cta_tot, c);
      run_gt += tot[0];
      run_eq += tot[1];
    }
    cluster.sync();  // no CTA of the cluster exits while another may still read its shared memory
  }

  // ---- emit in ascending position: all keys > thr, and the first k_eq keys == thr
  const int room_b = (int)min(room, (long long)b);
  int run = run_gt + min(run_eq, k_eq);
  // counts per vector of a lane, four vectors to a word (a warp's vector holds at most 128 positions: no carries)
  auto counts = [&](uint32_t bits, int half) {
    uint32_t c = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) c |= (uint32_t)__popc((bits >> (16 * half + 4 * e)) & 0xFu) << (8 * e);
    return c;
  };
  auto scan = [&](uint32_t c) {  // inclusive over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, c, o);
      if (lane >= o) c += x;
    }
    return c;
  };
  constexpr int kWords = (V + 3) / 4;
  if (__any_sync(0xffffffffu, tied != 0)) {  // of the ties the first k_eq
#pragma unroll
    for (int h = 0; h < kWords; ++h) {
      const uint32_t mine = counts(tied, h), incl = scan(mine), total = __shfl_sync(0xffffffffu, incl, 31);
      const uint32_t excl = incl - mine;
#pragma unroll
      for (int e = 0; e < (V < 4 ? V : 4); ++e) {
        int left = k_eq - run_eq - (int)((excl >> (8 * e)) & 0xFFu);  // ties that may still be kept
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t bit = 1u << (16 * h + 4 * e + i);
          if (tied & bit) {
            if (left > 0) kept |= bit;
            --left;
          }
        }
        run_eq += (int)((total >> (8 * e)) & 0xFFu);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < kWords; ++h) {
    const uint32_t mine = counts(kept, h), incl = scan(mine), total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - mine;
#pragma unroll
    for (int e = 0; e < (V < 4 ? V : 4); ++e) {
      int pos = run + (int)((excl >> (8 * e)) & 0xFFu);
      const int j = 4 * (quad0 + 32 * (4 * h + e));
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool keep = (kept >> (16 * h + 4 * e + i)) & 1u;
        if (keep && pos < room_b) out[pos] = j + i;
        pos += keep;
      }
      run += (int)((total >> (8 * e)) & 0xFFu);
    }
  }
}

// Beyond 262144 positions: one CTA per head that re-reads its keys in each of the five sweeps.  Warp wv owns `span`
// consecutive positions (a multiple of 32) and lane l of it the positions e*32 + l of those.  Three histograms of 11, 11 and
// 10 bits of the key, most significant first.
__global__ void __launch_bounds__(kSelThreads, 1) select_stream_kernel(const __grid_constant__ SelectArgs a, int span) {
  __shared__ int hist[2048];
  __shared__ int scan_gt[kSelWarps], scan_eq[kSelWarps];
  __shared__ int sel_digit, sel_want;
  const int u = (int)blockIdx.x, tid = threadIdx.x, lane = tid & 31, wv = tid >> 5;
  pdl_launch_dependents();
  pdl_wait();
  if (a.dev_status && blockIdx.x == 0 && tid == 0) *a.dev_status = a.status ? *a.status : 0;
  const int b = a.budgets[u];
  const long long off = a.offsets[u];
  const int n = a.heads_per_seq > 0 ? a.sl.T[u / a.heads_per_seq] - a.w : a.n;
  const int n_sink = a.n_sink;
  const float* src = a.scores + (size_t)u * a.stride;
  int32_t* out = a.kept_idx + off;
  const long long room = a.rows_cap - off;  // rows of this head that fit in the output

  // window rows follow the selected ones
  for (int t = tid; t < a.w; t += kSelThreads)
    if (b + t < room) out[b + t] = n + t;
  if (b <= 0) return;

  const int base = wv * span + lane;
  const int iters = span >> 5;
  // b-th largest key: the largest thr with count(key >= thr) >= b, found digit by digit (11, 11 and
  // 10 bits, most significant first): the keys that match the digits fixed so far are counted into
  // a shared-memory histogram of the next digit, and the bin in which the count of larger keys
  // reaches the remaining budget is the next digit of thr.  Positions beyond n take no part.
  uint32_t thr = 0;
  {
    int want = b;  // keys still to be found among those that match the fixed digits
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
      const int bins = pass == 2 ? 1024 : 2048;
      const uint32_t above = pass == 0 ? 0u : (thr >> (shift + (pass == 1 ? 11 : 10)));  // the fixed digits
      for (int i = tid; i < bins; i += kSelThreads) hist[i] = 0;
      __syncthreads();
      auto count = [&](uint32_t key, int j) {
        if (j < n && (pass == 0 || (key >> (shift + (pass == 1 ? 11 : 10))) == above))
          atomicAdd(&hist[(key >> shift) & (uint32_t)(bins - 1)], 1);
      };
      for (int e = 0; e < iters; ++e) {
        const int j = base + 32 * e;
        count(j < n ? key_at(src, j, n_sink) : 0u, j);
      }
      __syncthreads();
      // thread t owns the bins [t*per, t*per+per); suffix sums over the threads, from the top
      const int per = bins / kSelThreads;  // 2 or 1
      const int merged0 = hist[tid * per], merged1 = per == 2 ? hist[tid * per + 1] : 0;
      const int mine = merged0 + merged1;
      int incl = mine;  // sum over the lanes >= this one
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_down_sync(0xffffffffu, incl, off);
        if (lane + off < 32) incl += o;
      }
      if (lane == 0) scan_gt[wv] = incl;  // warp totals (scan_gt is free until the emit phase)
      __syncthreads();
      int higher = 0;  // keys in bins above this thread's bins
      for (int x = wv + 1; x < kSelWarps; ++x) higher += scan_gt[x];
      higher += incl - mine;
      if (higher < want && want <= higher + mine) {  // exactly one thread: the digit is in its bins
        int run = higher;
        for (int i = per - 1; i >= 0; --i) {
          const int c = i ? merged1 : merged0;
          if (want <= run + c) {
            sel_digit = tid * per + i;
            sel_want = want - run;
            break;
          }
          run += c;
        }
      }
      __syncthreads();  // the histogram may be cleared again
      thr |= (uint32_t)sel_digit << shift;
      want = sel_want;
    }
  }

  // per-warp totals of keys above / equal to the threshold, then an exclusive scan over warps
  int my_gt = 0, my_eq = 0;
  for (int e = 0; e < iters; ++e) {
    const int j = base + 32 * e;
    const uint32_t key = j < n ? key_at(src, j, n_sink) : 0u;
    my_gt += key > thr;
    my_eq += key == thr;
  }
  my_gt = __reduce_add_sync(0xffffffffu, my_gt);
  my_eq = __reduce_add_sync(0xffffffffu, my_eq);
  if (lane == 0) {
    scan_gt[wv] = my_gt;
    scan_eq[wv] = my_eq;
  }
  __syncthreads();
  int run_gt = 0, run_eq = 0, total_gt = 0;
  for (int x = 0; x < kSelWarps; ++x) {
    if (x < wv) {
      run_gt += scan_gt[x];
      run_eq += scan_eq[x];
    }
    total_gt += scan_gt[x];
  }
  const int k_eq = b - total_gt;  // ties to keep (>= 1)

  // emit in ascending position: all keys > thr, and the first k_eq keys == thr
  const uint32_t lt_mask = (1u << lane) - 1u;
  auto emit = [&](uint32_t key, int j) {
    const bool gt = key > thr, eq = key == thr;
    const uint32_t m_gt = __ballot_sync(0xffffffffu, gt), m_eq = __ballot_sync(0xffffffffu, eq);
    const int before_gt = run_gt + __popc(m_gt & lt_mask);
    const int before_eq = run_eq + __popc(m_eq & lt_mask);
    if (gt || (eq && before_eq < k_eq)) {
      const int pos = before_gt + min(before_eq, k_eq);
      if (pos < room) out[pos] = j;
    }
    run_gt += __popc(m_gt);
    run_eq += __popc(m_eq);
  };
  for (int e = 0; e < iters; ++e) {
    const int j = base + 32 * e;
    emit(j < n ? key_at(src, j, n_sink) : 0u, j);
  }
}

// ---- gather --------------------------------------------------------------------------

constexpr int kGatherThreads = 256;

// LPR lanes copy one row of 16*LPR bytes.  A warp takes 32 consecutive packed rows (FULL), or one round of copies where
// that fills the chip better: every lane resolves one row (source head by binary search over the offsets, from shared memory
// when they fit; source position from kept_idx), then the warp copies the rows 32/LPR at a time, four batches in flight.
// Bound by HBM when there are many rows: 0.95 of the measured copy rate at 1.7 M rows.
constexpr int kGatherSmemHeads = 2047;

template <int LPR, bool FULL>
__global__ void __launch_bounds__(kGatherThreads, 4) gather_kernel(const int32_t* __restrict__ offsets,
                                                                const int32_t* __restrict__ kept_idx,
                                                                const uint4* __restrict__ k, const uint4* __restrict__ v,
                                                                uint4* __restrict__ k_out, uint4* __restrict__ v_out,
                                                                long long rows_cap, int nheads, int T) {
  __shared__ int32_t off_s[kGatherSmemHeads + 1];
  pdl_wait();
  const bool in_smem = nheads <= kGatherSmemHeads;
  if (in_smem) {
    for (int i = threadIdx.x; i <= nheads; i += kGatherThreads) off_s[i] = offsets[i];
    __syncthreads();
  }
  auto offset = [&](int u) { return (long long)(in_smem ? off_s[u] : __ldg(offsets + u)); };
  // packed rows of these heads (a caller may pass a slice of a larger call's offsets), clipped to what the output can hold
  const long long row_begin = offset(0), total_rows = min(offset(nheads), rows_cap);
  constexpr int kRowsPerBatch = 32 / LPR;
  constexpr int kInFlight = LPR < 4 ? LPR : 4;
  constexpr int span = FULL ? 32 : kRowsPerBatch * kInFlight;
  const int lane = threadIdx.x & 31;
  const long long warp_global = ((long long)blockIdx.x * kGatherThreads + threadIdx.x) >> 5;
  const long long warps_total = ((long long)gridDim.x * kGatherThreads) >> 5;
  const int sub = lane / LPR, part = lane % LPR;
  for (long long base = row_begin + warp_global * span; base < total_rows; base += warps_total * span) {
    const long long r = base + lane;
    long long src_row = -1;
    if (lane < span && r < total_rows) {
      int lo = 0, hi = nheads;  // largest u with offsets[u] <= r
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (offset(mid) <= r) lo = mid; else hi = mid;
      }
      // positions come from the selection kernel; clamping them keeps the copy inside the head even if
      // the scores were not finite (their ranking is then meaningless, but nothing is read out of bounds)
      const int pos = min(max(kept_idx[r], 0), T - 1);
      src_row = (long long)lo * T + pos;
    }
#pragma unroll
    for (int b0 = 0; b0 * kRowsPerBatch < span; b0 += kInFlight) {
      uint4 kv[kInFlight], vv[kInFlight];
      long long srow[kInFlight];
#pragma unroll
      for (int i = 0; i < kInFlight; ++i) {
        const int row_in_span = (b0 + i) * kRowsPerBatch + sub;
        srow[i] = __shfl_sync(0xffffffffu, src_row, row_in_span);
        if (srow[i] >= 0) {
          kv[i] = __ldg(k + srow[i] * LPR + part);
          vv[i] = __ldg(v + srow[i] * LPR + part);
        }
      }
#pragma unroll
      for (int i = 0; i < kInFlight; ++i) {
        const int row_in_span = (b0 + i) * kRowsPerBatch + sub;
        if (srow[i] >= 0) {
          __stcs(k_out + (base + row_in_span) * LPR + part, kv[i]);
          __stcs(v_out + (base + row_in_span) * LPR + part, vv[i]);
        }
      }
    }
  }
}

template <int LPR>
cudaError_t launch_gather_t(const Dims& dm, const int32_t* offsets, const int32_t* kept_idx, const void* k, const void* v,
                            void* k_out, void* v_out, long long rows_cap, bool overlap, cudaStream_t st) {
  // the row count is only known on the device; size the grid for the capacity, or for what these heads can hold where that
  // is less (the kernel gets the capacity itself: a slice of a larger call's offsets starts beyond these heads' own rows)
  const long long rows_max = (long long)dm.heads() * dm.T, rows_grid = rows_cap < rows_max ? rows_cap : rows_max;
  // one round of copies per warp (4 to 16 rows) unless that makes more warps than the chip holds
  constexpr int kOneRound = (32 / LPR) * (LPR < 4 ? LPR : 4);
  const bool full = rows_grid > 148LL * 64 * kOneRound;
  const int span = full ? 32 : kOneRound;
  const long long spans = (rows_grid + span - 1) / span + 1;
  long long blocks = (spans + kGatherThreads / 32 - 1) / (kGatherThreads / 32);
  const long long max_blocks = 148LL * 8 * 4;  // a few waves of resident CTAs; the loop covers the rest
  if (blocks > max_blocks) blocks = max_blocks;
  if (blocks < 1) blocks = 1;
  return launch_pdl(full ? gather_kernel<LPR, true> : gather_kernel<LPR, false>, dim3((unsigned)blocks), dim3(kGatherThreads), 0, st, overlap && !full, offsets, kept_idx,
                    (const uint4*)k, (const uint4*)v, (uint4*)k_out, (uint4*)v_out, rows_cap, (int)dm.heads(), dm.T);
}

}  // namespace

cudaError_t launch_select(const Dims& dm, const float* scores, int stride, bool pool, const int32_t* budgets,
                          const int32_t* offsets, int32_t* kept_idx, int64_t rows_cap, const int* status,
                          int32_t* dev_status, bool overlap, LaunchCtx& lc) {
  const unsigned heads = (unsigned)dm.heads();
  const int n = dm.n;
  SelectArgs a = {};
  a.scores = scores;
  a.budgets = budgets;
  a.offsets = offsets;
  a.kept_idx = kept_idx;
  a.rows_cap = rows_cap;
  a.stride = stride;
  a.n = n;
  a.w = dm.w;
  a.half = pool ? dm.kp / 2 : 0;
  a.vec = stride % 4 == 0 && (reinterpret_cast<uintptr_t>(scores) & 15u) == 0;
  a.n_sink = dm.n_sink;
  a.heads_per_seq = dm.seq_T ? dm.N : 0;
  a.status = status;
  a.dev_status = dev_status;
  if (dm.seq_T)
    for (int q = 0; q < dm.S; ++q) a.sl.T[q] = dm.seq_T[q];
  // Keys per thread (in registers) and CTAs per head.  Up to 32768 positions: one CTA of 256 to 1024 threads with 4 to 32
  // keys per thread (a cluster's barriers cost more than they save there).  Up to 262144: the smallest cluster (2, 4 or 8
  // CTAs) that covers the head with 32 keys per thread; small clusters are placed and synchronised faster than large
  // ones.  Beyond: one CTA that re-reads its keys from memory in every round.
  cudaError_t e;
  if (n <= 32 * kSelThreads) {
    const int threads = n <= 1024 ? 256 : n <= 2048 ? 512 : kSelThreads;
    auto kern = n <= 4 * kSelThreads ? select_kernel<1, false> : n <= 8 * kSelThreads ? select_kernel<2, false>
                : n <= 16 * kSelThreads ? select_kernel<4, false> : select_kernel<8, false>;
    e = launch_pdl(kern, dim3(heads), dim3(threads), 0, lc.st, overlap, a);
  } else if (n <= 8 * 32 * kSelThreads) {
    const int csize = n <= 2 * 32 * kSelThreads ? 2 : n <= 4 * 32 * kSelThreads ? 4 : 8;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(heads * csize);
    cfg.blockDim = dim3(kSelThreads);
    cfg.stream = lc.st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, select_kernel<8, true>, a);
  } else {
    const int per_warp = (n + kSelWarps - 1) / kSelWarps;
    e = launch_pdl(select_stream_kernel, dim3(heads), dim3(kSelThreads), 0, lc.st, overlap, a, (per_warp + 31) & ~31);
  }
  if (e != cudaSuccess) return e;
  lc.mark("select");
  return cudaGetLastError();
}

bool select_pools(const Dims& dm) { return dm.kp / 2 <= 4 && dm.n <= 8 * 32 * kSelThreads; }

cudaError_t launch_gather(const Dims& dm, const int32_t* offsets, const int32_t* kept_idx, const void* k,
                          const void* v, void* k_out, void* v_out, int64_t rows_cap, bool overlap, LaunchCtx& lc) {
  if (rows_cap <= 0) return cudaSuccess;
  const int lpr = (int)(dm.d * dm.esize() / 16);
  cudaError_t e;
  switch (lpr) {
    case 8: e = launch_gather_t<8>(dm, offsets, kept_idx, k, v, k_out, v_out, rows_cap, overlap, lc.st); break;
    case 16: e = launch_gather_t<16>(dm, offsets, kept_idx, k, v, k_out, v_out, rows_cap, overlap, lc.st); break;
    default: e = launch_gather_t<32>(dm, offsets, kept_idx, k, v, k_out, v_out, rows_cap, overlap, lc.st); break;
  }
  if (e != cudaSuccess) return e;
  lc.mark("gather");
  return cudaGetLastError();
}

}  // namespace lukv
