// KeyDiff proxy scores (the second metric the paper evaluates, pi_2 of Sec. 5.1; recent window 1 in App. E).  The
// paper only names the metric; the formula is the one of the method's own publication:
//   u_j = k_j / max(||k_j||, eps),  a = mean of u_j over all T cached keys of the head,
//   score_j = - <k_j, a> / (max(||k_j||, eps) * max(||a||, eps)),  eps = 1e-8, for the n = T-w rankable positions.
// A key-only scan with no contraction: bound by HBM and by L2.  The anchor needs every key of the head before any score, so
// K is read twice; the kernel walks the heads in groups, every CTA alternating between the first read of one group and the
// second read of an earlier one, which L2 then serves for the most part.
#include <cstdlib>

#include "tc_ptx.cuh"

namespace lukv {
namespace {

constexpr int kKdConsumerWarps = 8;
constexpr int kKdConsumers = kKdConsumerWarps * 32;
constexpr int kKdThreads = kKdConsumers + 64;  // + the warp whose first lane issues the bulk copies, + the helper warp
constexpr int kKdStageRows = 64;               // key rows per shared-memory stage (32 of 512 bytes)
constexpr int kKdSliceRows = 8;                // granularity of a slice: what a warp takes at a time
constexpr int kKdRingBytes = 96 * 1024;        // ring of stages per CTA; two CTAs per SM
constexpr int kKdMaxGrid = 512;                // CTAs of the persistent grid
constexpr int kKdMaxGroup = 512;               // heads per group, at most
constexpr int kKdLag = 2;                      // groups between the two reads of a group (LUKV_KEYDIFF_LAG: up to kKdMaxLag)
constexpr int kKdMaxLag = 8;
constexpr int kKdLanesPerRow = 4;
constexpr int kKdFoldDepth = 12;               // pieces a lane has in flight when an anchor is made
constexpr float kKdEps = 1e-8f;

// 16 bytes of a key row as packed pairs of fp32 (two lanes of one FMA-pipe instruction).
template <typename TIn>
struct Vec16;
template <>
struct Vec16<__nv_bfloat16> {
  static constexpr int kElems = 8;
  __device__ static void pairs(const uint4& raw, uint64_t (&x)[4]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
  }
};
template <>
struct Vec16<float> {
  static constexpr int kElems = 4;
  __device__ static void pairs(const uint4& raw, uint64_t (&x)[2]) {
    x[0] = pack2(__uint_as_float(raw.x), __uint_as_float(raw.y));
    x[1] = pack2(__uint_as_float(raw.z), __uint_as_float(raw.w));
  }
};

struct KdArgs {
  const unsigned char* k;  // [heads][T][d]
  float* scores;           // [heads][stride]
  float* pieces;           // [groups * CTAs + heads][d]: partial sums of unit keys
  uint32_t* anchors;       // [heads][d]   mean unit key, bits inverted; 0 until it is there (the inverse of no number)
  int* head_count;         // [heads]      pieces delivered.  Starts at 0.
  int32_t* dev_status;     // may be null
  int T, n, stride, heads, group, lag;
  int fold_shift;          // an anchor is made in 1 << fold_shift parts
  uint32_t per, per_tail;  // rows of a slice, in the groups of `group` heads and in a smaller last one
  uint32_t spin_limit;
  int drop_head;           // test hook: this head's anchor is never published (-1: none)
};

// C consecutive words, always from memory at GPU scope (polls data another CTA writes).
template <int C>
__device__ __forceinline__ void ld_relaxed_words(const uint32_t* p, uint32_t (&v)[C]) {
  if (C == 4)
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[C - 2]), "=r"(v[C - 1]) : "l"(p) : "memory");
  else
    asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "l"(p) : "memory");
}
// Counts one in; what this thread has seen written is ordered before.
__device__ __forceinline__ void red_release_inc(int* p) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The slice of a group's rows (heads x T, one head after the other; fewer than 2^31) that a CTA owns: equal slices, whole
// stages.
struct KdSlice {
  uint32_t h0, slice, per, lo, hi;
};
__device__ __forceinline__ KdSlice kd_slice(const KdArgs& a, int g) {
  KdSlice s;
  s.h0 = g * a.group;
  const bool tail = s.h0 + a.group > a.heads;  // the last group may hold fewer heads
  const uint32_t rows = (tail ? a.heads - s.h0 : a.group) * (uint32_t)a.T;
  s.per = tail ? a.per_tail : a.per;
  s.slice = (blockIdx.x + (uint32_t)g) % gridDim.x;
  s.lo = min(rows, s.slice * s.per);
  s.hi = min(rows, s.lo + s.per);
  return s;
}

// A CTA's pieces in order: the part of its slice that lies in one head, group by group.
struct KdWalk {
  int g;                   // group
  uint32_t ul, u;          // head of the group, head
  int j_begin, j_end;      // rows of the head
  KdSlice sl;
  uint32_t at;
};
__device__ __forceinline__ KdWalk kd_begin() {
  KdWalk w;
  w.g = -1;
  w.at = w.sl.hi = 0;
  return w;
}
__device__ __forceinline__ bool kd_next(const KdArgs& a, int G, KdWalk& w) {  // false: no piece is left
  while (w.at >= w.sl.hi) {
    if (++w.g >= G) return false;
    w.sl = kd_slice(a, w.g);
    w.at = w.sl.lo;
  }
  w.ul = w.at / (uint32_t)a.T;
  w.u = w.sl.h0 + w.ul;
  const uint32_t row0 = w.ul * (uint32_t)a.T;
  w.j_begin = (int)(w.at - row0);
  w.j_end = (int)min((uint32_t)a.T, w.sl.hi - row0);
  w.at = row0 + w.j_end;
  return true;
}
// Whether the walk's next piece is one of group g (the walk goes through the groups in order).
__device__ __forceinline__ bool kd_next_in(const KdArgs& a, int G, int g, KdWalk& w) {
  if (w.at >= w.sl.hi) {
    if (w.g >= g) return false;
    w.g = g;
    w.sl = kd_slice(a, g);
    w.at = w.sl.lo;
    if (w.at >= w.sl.hi) return false;
  }
  return kd_next(a, G, w);
}
// Slices that hold a piece of the ul-th head of a group.
__device__ __forceinline__ void kd_head_slices(const KdArgs& a, uint32_t ul, uint32_t per, uint32_t& first, uint32_t& last) {
  first = ul * (uint32_t)a.T / per;
  last = ((ul + 1) * (uint32_t)a.T - 1) / per;
}

// A lane's share of one key row out of a stage: V loads of 16 bytes (zeros for a row the stage does not hold).
// Lane l of the four that share the row reads the 16-byte parts 4i + l; odd rows take i in rotated order so that
// the two rows of a quarter-warp fall into different banks.
template <int V>
__device__ __forceinline__ void kd_load_row(const unsigned char* row, bool present, int l, int odd_row, uint4 (&raw)[V]) {
#pragma unroll
  for (int i = 0; i < V; ++i) raw[i] = *reinterpret_cast<const uint4*>(row + (4 * ((i + odd_row) % V) + l) * 16);
  if (!present)
#pragma unroll
    for (int i = 0; i < V; ++i) raw[i] = make_uint4(0u, 0u, 0u, 0u);
}

// One persistent cooperative kernel (cooperative only so that all CTAs are resident: they wait for one another's
// partial sums).  Every group is cut into one slice per CTA.  A CTA's "sum" step of a group adds the unit keys of its
// slice, one partial sum ("piece") per head the slice touches; its "score" step, `lag` groups later, re-reads the slice
// (from L2, mostly) and scores it against the anchors.  Even CTAs run sum(g), score(g-lag), sum(g+1), ...; odd CTAs score
// first, so that at any time half of the grid reads HBM and half reads L2.  The slices move on by one CTA per group: a
// slice that lies in two heads costs 20 % more, and all would wait for the CTA that had it every time (256 heads of 32768
// keys: 583 us instead of 601).  Piece ids: slice s's piece of head u in group g is g * CTAs + s + u, unique and
// ascending along the rows.
// Rows arrive in a ring of shared-memory stages filled by bulk copies that one producer lane issues as far ahead
// as the ring allows, across the two kinds of step.
// Everything that needs a round trip to global memory is the helper warp's: it adds up a piece that the consumers left in
// shared memory and delivers it, makes the anchors (or quarters of them, fold_shift) that fall to this CTA once all
// pieces are there, and fetches the anchors of the next score steps.  It takes whichever of the three can go on.  A quarter
// of an anchor out of 60 pieces is two round trips to L2 (all columns by one warp, 16 pieces at a time: 11; 583 -> 564 us).
// What bounds it: HBM for the first reads and the second reads that miss L2 (5.2 TB/s of the two at 564 us) beside the
// arithmetic, two passes of eight packed pairs per 16 bytes (all keys out of L2: 406 us).
template <typename TIn, int D>
__global__ void __launch_bounds__(kKdThreads, 2) keydiff_kernel(const KdArgs a) {
  constexpr int E = Vec16<TIn>::kElems;
  constexpr int kRowBytes = D * (int)sizeof(TIn);
  constexpr int kRows = kRowBytes > 256 ? kKdStageRows / 2 : kKdStageRows;  // rows per stage
  constexpr int kBatches = kRows / 32;                                      // eight rows of a warp at a time
  constexpr int kStageBytes = kRows * kRowBytes;
  constexpr int kStages = kKdRingBytes / kStageBytes;
  constexpr int V = kRowBytes / (16 * kKdLanesPerRow);  // 16-byte loads per lane and row
  constexpr int C = D / 32;                             // columns per lane of the helper
  constexpr int H = E / 2;                              // pairs per 16 bytes
  static_assert(V >= 2 && V % 2 == 0 && kStages >= 2 && kStages % 2 == 0 && (C == 2 || C == 4), "shape");
  extern __shared__ __align__(128) unsigned char ring[];
  __shared__ __align__(8) uint64_t bars[2 * kStages + 6];
  __shared__ __align__(16) float red[2 * kKdConsumerWarps][D];
  __shared__ __align__(16) float anchor_s[2][D];
  __shared__ float inv_s[2];
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = (a.heads + a.group - 1) / a.group;
  const bool odd_cta = blockIdx.x & 1;
  auto full = [&](uint32_t s) { return smem_u32(&bars[s]); };
  auto empty = [&](uint32_t s) { return smem_u32(&bars[kStages + s]); };
  const uint32_t red_full = smem_u32(&bars[2 * kStages]), red_empty = smem_u32(&bars[2 * kStages + 1]);
  auto anc_full = [&](uint32_t s) { return smem_u32(&bars[2 * kStages + 2 + s]); };
  auto anc_empty = [&](uint32_t s) { return smem_u32(&bars[2 * kStages + 4 + s]); };
  if (threadIdx.x == 0) {
    abort_s = 0;
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), kKdConsumerWarps / 2);
    }
    mbar_init(red_full, kKdConsumerWarps);
    mbar_init(red_empty, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(anc_full(s), 1);
      mbar_init(anc_empty(s), kKdConsumerWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp == kKdConsumerWarps) {
    // ---- producer: the same walk over steps, pieces and stages as the consumers
    if (lane != 0) return;
    uint32_t cnt = 0;
    bool ok = true;
    KdWalk sum = kd_begin(), score = kd_begin();
    const uint64_t keep = l2_policy_evict_last(), drop = l2_policy_evict_first();
    for (int it = 0; it < G + a.lag && ok; ++it) {
      for (int half = 0; half < 2 && ok; ++half) {
        const bool sum_step = (half == 0) != odd_cta;
        const int g = sum_step ? it : it - a.lag;
        if (g < 0 || g >= G) continue;
        KdWalk& w = sum_step ? sum : score;
        while (ok && kd_next_in(a, G, g, w)) {
          const int j_end = sum_step ? w.j_end : min(w.j_end, a.n);
          const unsigned char* base = a.k + (size_t)w.u * a.T * kRowBytes;
          for (int j = w.j_begin; j < j_end; j += kRows, ++cnt) {
            const uint32_t s = cnt % kStages, use = cnt / kStages;
            ok = mbar_wait(empty(s), (use & 1) ^ 1, abort_flag, a.dev_status, a.spin_limit);
            if (!ok) break;
            const uint32_t bytes = (uint32_t)min(kRows, j_end - j) * kRowBytes;
            mbar_expect_tx(full(s), bytes);
            bulk_load_hint(smem_u32(ring + (size_t)s * kStageBytes), base + (size_t)j * kRowBytes, bytes, full(s),
                           sum_step ? keep : drop);
          }
        }
      }
    }
    if (!ok) {
      // giving up: no copy of this CTA may still be in flight when it exits
      for (uint32_t back = 1; back <= (uint32_t)kStages && back <= cnt; ++back) {
        const uint32_t c = cnt - back, s = c % kStages, use = c / kStages;
        for (uint32_t i = 0; i < a.spin_limit && !mbar_try_wait(full(s), use & 1); ++i) __nanosleep(64);
      }
    }
    return;
  }

  if (warp == kKdConsumerWarps + 1) {
    // ---- helper
    KdWalk out = kd_begin(), in = kd_begin();
    bool more_out = kd_next(a, G, out), more_in = kd_next(a, G, in);
    // next anchor to make, or part of its columns: the fold-th, head fold_u of fold_n pieces
    uint32_t fold = blockIdx.x, fold_first = 0;
    int fold_u = 0, fold_n = 0;
    const int fold_lanes = D / 4 >> a.fold_shift;  // lanes (of four columns each) per piece
    auto fold_head = [&] {
      fold_u = (int)(fold >> a.fold_shift);
      if (fold_u >= a.heads) return;
      const KdSlice sl = kd_slice(a, fold_u / a.group);
      uint32_t first, last;
      kd_head_slices(a, fold_u - sl.h0, sl.per, first, last);
      fold_n = (int)(last - first) + 1;
      fold_first = (uint32_t)(fold_u / a.group) * gridDim.x + first + fold_u;
    };
    fold_head();
    uint32_t outs = 0, ins = 0, idle = 0;
    auto asked = [&](bool mine) {  // lane 0 looks for all; what it has seen is ordered before what they read
      const bool yes = __shfl_sync(0xffffffffu, (int)mine, 0) != 0;
      __syncwarp();
      return yes;
    };
    while ((more_out || more_in || fold_u < a.heads) && !*abort_flag) {
      bool progress = false;
      if (more_out && asked(lane == 0 && mbar_test_wait(red_full, outs & 1))) {
        float v[C];
#pragma unroll
        for (int c = 0; c < C; ++c) v[c] = 0.f;
#pragma unroll
        for (int p = 0; p < 2 * kKdConsumerWarps; ++p)
#pragma unroll
          for (int c = 0; c < C; ++c) v[c] += red[p][lane * C + c];
        __syncwarp();
        if (lane == 0) mbar_arrive(red_empty, 1);
        float* piece = a.pieces + ((size_t)out.g * gridDim.x + out.sl.slice + out.u) * D;
#pragma unroll
        for (int c = 0; c < C; ++c) __stcg(piece + lane * C + c, v[c]);
        __syncwarp();
        if (lane == 0) red_release_inc(a.head_count + out.u);
        ++outs;
        more_out = kd_next(a, G, out);
        progress = true;
      }
      // (asked for once this CTA has delivered its own pieces of that group)
      if (fold_u < a.heads && (!more_out || out.g > fold_u / a.group) &&
          asked(lane == 0 && ld_acquire(a.head_count + fold_u) == fold_n)) {
        // anchor = the sum of the pieces / T: 32 / fold_lanes pieces side by side, kKdFoldDepth loads in flight
        const int pp = 32 / fold_lanes;
        const uint32_t col = (fold & ((1u << a.fold_shift) - 1)) * (4 * fold_lanes) + (lane % fold_lanes) * 4;
        const float* src = a.pieces + (size_t)fold_first * D + col;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        for (int p0 = lane / fold_lanes; p0 < fold_n; p0 += kKdFoldDepth * pp) {
          float4 x[kKdFoldDepth];
#pragma unroll
          for (int i = 0; i < kKdFoldDepth; ++i)
            x[i] = p0 + i * pp < fold_n ? __ldcg(reinterpret_cast<const float4*>(src + (size_t)(p0 + i * pp) * D))
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int i = 0; i < kKdFoldDepth; ++i) v[0] += x[i].x, v[1] += x[i].y, v[2] += x[i].z, v[3] += x[i].w;
        }
        for (int off = fold_lanes; off < 32; off <<= 1)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], off);
        if (fold_u != a.drop_head && lane < fold_lanes)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            __stcg(a.anchors + (size_t)fold_u * D + col + c, ~__float_as_uint(v[c] / (float)a.T));
        fold += gridDim.x;
        fold_head();
        progress = true;
      }
      if (more_in) {
        const uint32_t s = ins & 1;
        if (asked(lane == 0 && mbar_test_wait(anc_empty(s), ((ins >> 1) & 1) ^ 1))) {
          uint32_t x[C];
          ld_relaxed_words<C>(a.anchors + (size_t)in.u * D + lane * C, x);
          bool here = true;
#pragma unroll
          for (int c = 0; c < C; ++c) here = here && x[c] != 0u;
          if (__all_sync(0xffffffffu, here)) {
            float n2 = 0.f;
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const float v = __uint_as_float(~x[c]);
              anchor_s[s][lane * C + c] = v;
              n2 = fmaf(v, v, n2);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, off);
            if (lane == 0) inv_s[s] = 1.f / fmaxf(sqrtf(n2), kKdEps);
            __syncwarp();
            if (lane == 0) mbar_arrive(anc_full(s), 1);
            ++ins;
            more_in = kd_next(a, G, in);
            progress = true;
          }
        }
      }
      if (progress) {
        idle = 0;
      } else {
        if (++idle > a.spin_limit) {
          if (lane == 0) raise_abort(abort_flag, a.dev_status);
          break;
        }
        if (idle > 4) __nanosleep(100);
      }
    }
    return;
  }

  // ---- consumers.  Nothing below leaves a loop early: once the abort flag is up every wait returns at once, and the walk
  // ends after arithmetic on whatever the stages hold.
  // Warps 0-3 take the even stages of the ring, warps 4-7 the odd ones.
  const int l = lane & (kKdLanesPerRow - 1), r = lane >> 2, odd_row = r & 1;
  const int row0 = (warp & 3) * (8 * kBatches) + r;
  const uint32_t turn = warp >> 2;
  uint32_t stage = 0, phase = 0, sums = 0, scores = 0;
  KdWalk sum = kd_begin(), score = kd_begin();
  auto wait = [&](uint32_t bar, uint32_t parity) { mbar_wait(bar, parity, abort_flag, a.dev_status, a.spin_limit); };
  // body(raw data of this lane's part of a row, row of the head, whether it is one) for this warp's rows in [j0, j1)
  auto rows = [&](int j0, int j1, auto&& body) {
    for (int j = j0; j < j1; j += kRows) {
      if ((stage & 1) == turn) {
        wait(full(stage), phase);
        const unsigned char* at = ring + (size_t)stage * kStageBytes + (size_t)row0 * kRowBytes;
#pragma unroll
        for (int b = 0; b < kBatches; ++b) {
          uint4 raw[V];
          kd_load_row<V>(at + b * 8 * kRowBytes, j + row0 + 8 * b < j1, l, odd_row, raw);
          if (b == kBatches - 1) {
            __syncwarp();
            if (lane == 0) mbar_arrive(empty(stage), 1);  // the rows are in registers
          }
          body(raw, j + row0 + 8 * b, j + row0 + 8 * b < j1);
        }
      }
      if (++stage == kStages) {
        stage = 0;
        phase ^= 1;
      }
    }
  };
  auto quad_sum = [&](float v) {  // over the four lanes that share a row
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
  };
  for (int it = 0; it < G + a.lag; ++it) {
    for (int half = 0; half < 2; ++half) {
      const bool sum_step = (half == 0) != odd_cta;
      const int g = sum_step ? it : it - a.lag;
      if (g < 0 || g >= G) continue;
      KdWalk& w = sum_step ? sum : score;
      while (kd_next_in(a, G, g, w)) {
        if (sum_step) {
          uint64_t acc[V][H];
#pragma unroll
          for (int i = 0; i < V; ++i)
#pragma unroll
            for (int e = 0; e < H; ++e) acc[i][e] = 0ull;
          rows(w.j_begin, w.j_end, [&](const uint4 (&raw)[V], int, bool) {
            uint64_t x[V][H], s0 = 0ull, s1 = 0ull;
#pragma unroll
            for (int i = 0; i < V; ++i) {
              Vec16<TIn>::pairs(raw[i], x[i]);
#pragma unroll
              for (int e = 0; e < H; e += 2) {
                s0 = ffma2(x[i][e], x[i][e], s0);
                s1 = ffma2(x[i][e + 1], x[i][e + 1], s1);
              }
            }
            const float inv = 1.f / fmaxf(sqrtf(quad_sum(sum4(s0, s1))), kKdEps);  // an absent row is zero and adds nothing
            const uint64_t inv2 = pack2(inv, inv);
#pragma unroll
            for (int i = 0; i < V; ++i)
#pragma unroll
              for (int e = 0; e < H; ++e) acc[i][e] = ffma2(x[i][e], inv2, acc[i][e]);
          });
          wait(red_empty, (sums & 1) ^ 1);
          // rows of equal parity a warp holds side by side; the helper adds warps and parities in a fixed order
#pragma unroll
          for (int i = 0; i < V; ++i)
#pragma unroll
            for (int e = 0; e < H; ++e) {
              float u, v;
              unpack2(acc[i][e], u, v);
              u += __shfl_xor_sync(0xffffffffu, u, 8);
              v += __shfl_xor_sync(0xffffffffu, v, 8);
              u += __shfl_xor_sync(0xffffffffu, u, 16);
              v += __shfl_xor_sync(0xffffffffu, v, 16);
              if (r < 2)
                *reinterpret_cast<float2*>(&red[warp * 2 + odd_row][(4 * ((i + odd_row) % V) + l) * E + 2 * e]) =
                    make_float2(u, v);
            }
          __syncwarp();
          if (lane == 0) mbar_arrive(red_full, 1);
          ++sums;
        } else {
          const uint32_t slot = scores & 1;
          wait(anc_full(slot), (scores >> 1) & 1);
          uint64_t av[V][H];
#pragma unroll
          for (int i = 0; i < V; ++i)
#pragma unroll
            for (int e = 0; e < H; ++e)
              av[i][e] = *reinterpret_cast<const uint64_t*>(&anchor_s[slot][(4 * ((i + odd_row) % V) + l) * E + 2 * e]);
          const float inv_an = inv_s[slot];
          __syncwarp();
          if (lane == 0) mbar_arrive(anc_empty(slot), 1);
          ++scores;
          float* out = a.scores + (size_t)w.u * a.stride;
          rows(w.j_begin, min(w.j_end, a.n), [&](const uint4 (&raw)[V], int j, bool present) {
            uint64_t s0 = 0ull, s1 = 0ull, d0 = 0ull, d1 = 0ull;
#pragma unroll
            for (int i = 0; i < V; ++i) {
              uint64_t x[H];
              Vec16<TIn>::pairs(raw[i], x);
#pragma unroll
              for (int e = 0; e < H; e += 2) {
                s0 = ffma2(x[e], x[e], s0);
                s1 = ffma2(x[e + 1], x[e + 1], s1);
                d0 = ffma2(x[e], av[i][e], d0);
                d1 = ffma2(x[e + 1], av[i][e + 1], d1);
              }
            }
            const float ss = quad_sum(sum4(s0, s1)), dot = quad_sum(sum4(d0, d1));
            if (l == 0 && present) out[j] = -dot * inv_an / fmaxf(sqrtf(ss), kKdEps);
          });
        }
      }
    }
  }
}

// Heads per group.  A group's second read comes out of L2 as far as the groups between the two reads fit there.  At
// kKdLag = 2, 256 heads of 32768 bf16 keys (2.1 GB) take 564 us with groups of 40 to 47 MB, 580 at 35, 711 at 26 (the
// anchors of a group are ready about 8 us after its last key) and 624 at 64 MB; with one group of all heads, which reads
// K twice from HBM, 645 us.  64 % of the second reads of 42 MB groups hit.  So: the number of heads nearest to 44 MB;
// all heads (at most kKdMaxGroup) where that is not within 34..54 MB (one
// head of 33.5 MB: 348 us against 328) or where there would be fewer than six groups (six: 88 us against 91; three: 54 against 52).
// LUKV_KEYDIFF_GROUP_MB sets the group's size in MB of keys.
int keydiff_group(const Dims& dm) {
  const char* env = getenv("LUKV_KEYDIFF_GROUP_MB");
  const int env_mb = env ? atoi(env) : 0;
  const size_t heads = (size_t)dm.heads(), cap = heads < (size_t)kKdMaxGroup ? heads : (size_t)kKdMaxGroup;
  const size_t head = (size_t)dm.T * dm.d * dm.esize(), mb = (size_t)1 << 20;
  if (env_mb >= 1 && env_mb <= 4096) {
    const size_t g = (size_t)env_mb * mb / head;
    return (int)(g < 1 ? 1 : g > cap ? cap : g);
  }
  const size_t g = (44 * mb + head / 2) / head;
  return (int)(g >= 1 && g * 6 <= heads && g <= cap && g * head >= 34 * mb && g * head <= 54 * mb ? g : cap);
}

size_t kd_align(size_t x) { return (x + 255) & ~(size_t)255; }
size_t kd_pieces_bytes(const Dims& dm) {
  const size_t group = (size_t)keydiff_group(dm), groups = ((size_t)dm.heads() + group - 1) / group;
  return kd_align((groups * kKdMaxGrid + (size_t)dm.heads()) * dm.d * sizeof(float));
}
size_t kd_anchor_bytes(const Dims& dm) { return kd_align((size_t)dm.heads() * dm.d * sizeof(float)); }
size_t kd_head_bytes(const Dims& dm) { return kd_align(((size_t)dm.heads() + 1) * sizeof(float)); }
size_t kd_count_offset(const Dims& dm) { return kd_pieces_bytes(dm) + kd_anchor_bytes(dm); }

}  // namespace

int* keydiff_status(const Dims& dm, float* scratch) {
  return reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(scratch) + kd_count_offset(dm)) + dm.heads();
}

namespace {

template <typename TIn, int D>
cudaError_t launch_keydiff_t(const Dims& dm, const void* k, float* scores, int stride, float* scratch, int32_t* dev_status,
                             int spare_sms, LaunchCtx& lc) {
  auto kern = keydiff_kernel<TIn, D>;
  int sms = 0, per_sm = 0;
  cudaError_t e;
  if ((e = device_sms(&sms)) != cudaSuccess || (e = allow_smem((const void*)kern, kKdRingBytes)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kKdThreads, kKdRingBytes)) != cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorLaunchOutOfResources;
  if (spare_sms > 0 && sms > 8 * spare_sms) sms -= spare_sms;  // kernels of another stream keep these
  KdArgs a;
  unsigned char* sc = reinterpret_cast<unsigned char*>(scratch);
  a.k = static_cast<const unsigned char*>(k);
  a.scores = scores;
  a.pieces = reinterpret_cast<float*>(sc);
  a.anchors = reinterpret_cast<uint32_t*>(sc + kd_pieces_bytes(dm));
  a.head_count = reinterpret_cast<int*>(sc + kd_count_offset(dm));
  a.dev_status = dev_status ? dev_status : keydiff_status(dm, scratch);
  a.T = dm.T, a.n = dm.n, a.stride = stride, a.heads = (int)dm.heads(), a.group = keydiff_group(dm);
  a.lag = env_int("LUKV_KEYDIFF_LAG", 1, kKdMaxLag, kKdLag);
  score_test_hooks(&a.spin_limit, &a.drop_head);
  if ((e = cudaMemsetAsync(a.anchors, 0, kd_anchor_bytes(dm) + kd_head_bytes(dm), lc.st)) != cudaSuccess) return e;
  // a slice is at least one stage: small problems get a smaller grid
  const long long slices = ((long long)a.group * dm.T + kKdStageRows - 1) / kKdStageRows;
  long long grid = (long long)sms * (per_sm > 2 ? 2 : per_sm);
  grid = grid > kKdMaxGrid ? kKdMaxGrid : grid;
  grid = grid > slices ? slices : grid;
  auto slice_rows = [&](long long heads) {
    const long long per = (heads * dm.T + grid - 1) / grid;
    return (uint32_t)((per + kKdSliceRows - 1) / kKdSliceRows * kKdSliceRows);
  };
  a.per = slice_rows(a.group);
  a.per_tail = a.heads % a.group ? slice_rows(a.heads % a.group) : a.per;
  // pieces of a head beyond what one warp can have in flight at once: their columns go to four CTAs
  a.fold_shift = dm.T / (long long)a.per > kKdFoldDepth ? 2 : 0;
  void* params[] = {(void*)&a};
  e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(kKdThreads), params, kKdRingBytes,
                                  lc.st);
  lc.mark("keydiff");
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// scratch of the KeyDiff scorer: pieces, anchors, the per-head counters and the status word
size_t keydiff_scratch_bytes(const Dims& dm) {
  return kd_pieces_bytes(dm) + kd_anchor_bytes(dm) + kd_head_bytes(dm);
}

cudaError_t launch_keydiff(const Dims& dm, const void* k, float* scores, int stride, float* scratch, int32_t* dev_status,
                           int spare_sms, LaunchCtx& lc) {
  if (dm.dtype == LUKV_DTYPE_BF16)
    return dm.d == 128 ? launch_keydiff_t<__nv_bfloat16, 128>(dm, k, scores, stride, scratch, dev_status, spare_sms, lc)
                       : launch_keydiff_t<__nv_bfloat16, 64>(dm, k, scores, stride, scratch, dev_status, spare_sms, lc);
  return dm.d == 128 ? launch_keydiff_t<float, 128>(dm, k, scores, stride, scratch, dev_status, spare_sms, lc)
                     : launch_keydiff_t<float, 64>(dm, k, scores, stride, scratch, dev_status, spare_sms, lc);
}

}  // namespace lukv
