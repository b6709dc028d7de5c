// Stage (b): global head-level budget allocation (paper Sec. 4.2, App. A.2).
//   hull_kernel    projection of every head's curve increments onto a non-increasing,
//                  non-negative sequence (Eq. "marginal_gain": what pooling adjacent violators gives);
//                  slopes compared as fp64 quotients, gains fp64 with explicit round-to-nearest
//                  operations, rounded once to fp32.  The result is a short list per head: the
//                  blocks of equal gain, steepest first.
//   greedy_kernel  the marginal-utility greedy, computed as a weighted selection: the greedy
//                  consumes curve segments in the order (gain desc, k asc, hid asc); the
//                  kernel finds the gain at which the budget runs out (capacities in bins of the
//                  gain, then a ranking; or bisection over its bits), then the segment index
//                  and the head among the segments of exactly that gain.
#include <algorithm>

#include "common.cuh"

namespace lukv {
namespace {

// ---- hull ----------------------------------------------------------------------------

// Where the blocks of one curve go.
struct HullOut {
  float* gain;
  unsigned short* start;
};

// mean of block 1 <= mean of block 2, where a block's mean is (its curve rise) / (its length) and
// the rises are differences of two fp32 curve values: decided exactly as the comparison of the two
// correctly rounded fp64 quotients.  Cheapest first:
//   fp32 cross products, when they are further apart than fp32 rounding can explain;
//   their exact values in two words, when both rises are exact in fp32 (neighbouring points of a long curve differ by a few
//   units in the last place, and ties are common): 24 + 13 bits, which fp64 quotients tell apart if they differ;
//   fp64 cross products, when they are clearly apart;
//   the fp64 quotients themselves.
// (the last two out of line: they are rare, and an fp64 operation costs a warp some 50 clocks)
// Block 1 rises from u_l1 to u_r1 over len1 points, block 2 from u_l2 to u_r2 over len2.
__device__ __noinline__ bool mean_le_f64(float u_l1, float u_r1, int len1, float u_l2, float u_r2, int len2) {
  const double a = __dsub_rn((double)u_r1, (double)u_l1), b = (double)len1;
  const double c = __dsub_rn((double)u_r2, (double)u_l2), d = (double)len2;
  const double p1 = __dmul_rn(a, d), p2 = __dmul_rn(c, b);
  const double diff = __dsub_rn(p1, p2);
  const double tol = fmax(fabs(p1), fabs(p2)) * 9.094947017729282e-13;  // 2^-40
  if (diff < -tol) return true;
  if (diff > tol) return false;
  return __ddiv_rn(a, b) <= __ddiv_rn(c, d);
}
// Whether d = fl(a - b) is a - b exactly: a sufficient condition (Sterbenz: the one at most twice the other).
__device__ __forceinline__ bool exact_diff(float a, float b, float d) { return fabsf(d) <= fminf(fabsf(a), fabsf(b)); }
// d1 / n1 <= d2 / n2 for exact rises d and lengths n below 2^13: exact cross products in two words.
__device__ __forceinline__ bool exact_le(float d1, float n1, float d2, float n2) {
  const float q1 = d1 * n2, q2 = d2 * n1;
  return (q1 < q2) | ((q1 == q2) & (fmaf(d1, n2, -q1) <= fmaf(d2, n1, -q2)));  // no branches
}
// Rises to or from a curve value of this magnitude, times a length, stay in fp32's range.
__device__ __forceinline__ bool exact_range(float u) { return fabsf(u) <= 1e34f; }
__device__ __forceinline__ bool mean_le(float u_l1, float u_r1, int len1, float u_l2, float u_r2, int len2) {
  const float d1 = u_r1 - u_l1, d2 = u_r2 - u_l2, n1 = (float)len1, n2 = (float)len2;
  const float q1 = d1 * n2, q2 = d2 * n1;
  const float diff = q1 - q2;
  // each product carries two roundings of 2^-24, the difference one; false if a product overflowed
  if (fabsf(diff) > 5e-7f * fmaxf(fabsf(q1), fabsf(q2))) return diff < 0.f;
  if (exact_range(u_l1) && exact_range(u_l2) && exact_diff(u_r1, u_l1, d1) && exact_diff(u_r2, u_l2, d2))
    return exact_le(d1, n1, d2, n2);
  return mean_le_f64(u_l1, u_r1, len1, u_l2, u_r2, len2);
}

// The vertices among cnt points (values us, places is, ascending; the first and the last are ends) in the warp's shared
// memory: a point on or below the chord of its neighbours is dropped, all of them tested at once.  One pass, in place; returns
// how many are left.
__device__ __forceinline__ int hull_pass(float* us, unsigned short* is, int cnt, int lane) {
  const uint32_t lt_mask = (1u << lane) - 1u;
  __syncwarp();
  int out = 0;
#pragma unroll 1
  for (int base = 0; base < cnt; base += 32) {
    // in place: the writes of a turn end before the points that the next one reads, but for the last, unless nothing
    // was dropped yet, when they write what is there
    const int i = base + lane, ii = min(i, cnt - 1), il = max(ii - 1, 0), ir = min(ii + 1, cnt - 1);
    const float um = us[ii], ul = us[il], ur = us[ir];
    const int km = is[ii], kl = is[il], kr = is[ir];
    // 2^23 + k as a float: differences of two are the lengths
    auto place = [](int k) { return __int_as_float(0x4B000000 | k); };
    const float d1 = um - ul, d2 = ur - um;
    bool keep;
    if (__all_sync(0xffffffffu, exact_range(um) & exact_diff(um, ul, d1) & exact_diff(ur, um, d2)))
      keep = !exact_le(d1, place(km) - place(kl), d2, place(kr) - place(km));
    else
      keep = !mean_le(ul, um, km - kl, um, ur, kr - km);
    keep = (i < cnt) & ((i == 0) | (i == cnt - 1) | keep);
    const uint32_t kept = __ballot_sync(0xffffffffu, keep);
    if (keep) {
      const int at = out + __popc(kept & lt_mask);
      us[at] = um;
      is[at] = (unsigned short)km;
    }
    out += __popc(kept);
    __syncwarp();
  }
  return out;
}
// Passes until one drops none; returns how many points are left, or -1 if that took more than max_passes.
__device__ __forceinline__ int hull_passes(float* us, unsigned short* is, int cnt, int max_passes, int lane) {
#pragma unroll 1
  for (int pass = 0; pass < max_passes; ++pass) {
    const int out = hull_pass(us, is, cnt, lane);
    if (out == cnt) return cnt;
    cnt = out;
  }
  return -1;
}
// The blocks between cnt vertices; the part without a positive slope is one block of gain 0.  The output may be the place
// of the vertices.  Returns the number of blocks.
__device__ __forceinline__ int hull_emit(const float* us, const unsigned short* is, int cnt, float* gain, unsigned short* start,
                                         int lane) {
  for (int base = 0; base < cnt - 1; base += 32) {
    const int i = base + lane;
    const bool block = i < cnt - 1;
    const float u = block ? us[i] : 0.f, u_next = block ? us[i + 1] : 0.f;
    const int k = block ? is[i] : 0, k_next = block ? is[i + 1] : 0;
    const bool rises = block && u_next > u;
    const int rising = __popc(__ballot_sync(0xffffffffu, rises));  // every lane has read
    if (block && lane <= rising) {
      double mean = 0.0;
      if (rises) mean = __ddiv_rn(__dsub_rn((double)u_next, (double)u), (double)(k_next - k));
      gain[i] = __double2float_rn(mean);
      start[i] = (unsigned short)k;
    }
    if (rising < 32) return min(base + rising + 1, cnt - 1);  // the rest has no positive slope
  }
  return cnt - 1;
}

// The blocks of cnt points, however many passes it takes (all but the last drop a point).
__device__ __noinline__ int hull_rest(float* us, unsigned short* is, int cnt, float* gain, unsigned short* start, int lane) {
  cnt = hull_passes(us, is, cnt, cnt, lane);
  return hull_emit(us, is, cnt, gain, start, lane);
}

// A vertex walk: the blocks that pooling adjacent violators ends up with are the edges of the least concave majorant of
// the points (k, U[k]); from a vertex i the next one is the point j > i with the steepest slope from i, the last of them
// if several share it.  Slopes are compared in fp32; points whose slopes fp32 cannot tell apart are compared by their
// correctly rounded fp64 quotients.  Once no slope is positive the rest is one block of gain 0.
// One warp per curve; returns the number of blocks.

// The last point among the candidates of the warp (j < 0: none in this lane) with the largest fp64 quotient.
__device__ __noinline__ int hull_resolve(float uj, int j, float ui, int i) {
  double q = j >= 0 ? __ddiv_rn(__dsub_rn((double)uj, (double)ui), (double)(j - i)) : -INFINITY;
#pragma unroll 1
  for (int off = 16; off > 0; off >>= 1) {
    const double qo = __shfl_xor_sync(0xffffffffu, q, off);
    const int jo = __shfl_xor_sync(0xffffffffu, j, off);
    if (qo > q || (qo == q && jo > j)) {
      q = qo;
      j = jo;
    }
  }
  return j;
}
// Steps of the walk after which the rest of a curve goes to hull_passes.
constexpr int kHullWalk = 16;
// The blocks found so far: lane l holds block l, its start and the curve there, until kHullWalk are complete or the walk
// ends.  A gain is an fp64 division, a chain of some 700 clocks: all of them at a time, off the walk's chain.
struct HullBlocks {
  int count = 0, start = 0;
  float u = 0.f;
  // the block that starts at point i (value ui) and ends at point `end` (value u_end); gain 0 when `flat`
  __device__ __forceinline__ void add(int i, float ui, int end, float u_end, bool flat, bool last, int lane,
                                      const HullOut& out) {
    if (lane == count) {
      start = i;
      u = ui;
    }
    if (++count < kHullWalk && !last) return;
    int r = __shfl_down_sync(0xffffffffu, start, 1);
    float ur = __shfl_down_sync(0xffffffffu, u, 1);
    if (lane == count - 1) {
      r = end;
      ur = u_end;
    }
    if (lane < count) {
      double mean = __ddiv_rn(__dsub_rn((double)ur, (double)u), (double)(r - start));
      if (!(mean > 0.0) || (flat && lane == count - 1)) mean = 0.0;
      out.gain[lane] = __double2float_rn(mean);
      out.start[lane] = (unsigned short)start;
    }
  }
};

// P <= 32 NT: every point in a register, all slopes of a step at once, no branches: 300 to 1000 clocks a step, growing with
// NT.  A curve of many vertices takes that many steps, while passes over its points in shared memory drop few of them and
// end early (one pass if it is concave, some 8 if it is noisy; a step costs as much as two to ten vectors of a pass).  So
// the first kHullWalk vertices are walked to, which is all there are on most rough curves (6 of 257 points on the
// benchmark's), and what is left goes to hull_rest.  us, is: P - kHullWalk entries of the warp's shared memory, may be
// out.gain + kHullWalk and out.start + kHullWalk.  Whole allocation of 8 concave curves of 513 points: 263 us as a walk
// alone, 29 us now (rough ones 23); 256 of 513 points 386 and 73 us, 256 of 257 points 105 and 61 us.
template <int NT>
__device__ __forceinline__ int hull_walk_regs(const float* __restrict__ U, int P, int lane, HullOut out, float* us,
                                              unsigned short* is) {
  float u[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) u[t] = lane + 32 * t < P ? __ldg(U + lane + 32 * t) : -INFINITY;
  float ui = __shfl_sync(0xffffffffu, u[0], 0);
  int i = 0;
  HullBlocks blocks;
#pragma unroll 1
  while (i < P - 1 && blocks.count < kHullWalk) {
    float sl[NT], best = -INFINITY;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int dist = lane + 32 * t - i;
      sl[t] = dist > 0 ? __fdividef(u[t] - ui, (float)dist) : -INFINITY;
      best = fmaxf(best, sl[t]);
    }
    best = warp_max(best);
    const float near = best * 0.999998f;  // infinite rises tie; if no slope is positive, nothing below matters
    int mine = -1, found = 0;
    float u_mine = 0.f;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      if (sl[t] >= near) {
        mine = lane + 32 * t;
        u_mine = u[t];
        ++found;
      }
    int next = __reduce_max_sync(0xffffffffu, mine);
    if (next < 0) next = P - 1;  // not a number: the rest is one block
    if (__reduce_add_sync(0xffffffffu, found) > 1) {
      // a lane with several candidates offers them one by one
      int win = -1;
      float u_win = 0.f;
#pragma unroll 1
      for (int t = 0; t < NT; ++t) {
        float ut = u[0], st = sl[0];
#pragma unroll
        for (int x = 1; x < NT; ++x)
          if (x == t) ut = u[x], st = sl[x];
        const int at = hull_resolve(ut, st >= near ? lane + 32 * t : -1, ui, i);
        if (at < 0) continue;
        const float u_at = __shfl_sync(0xffffffffu, ut, at & 31);
        // the winner of this turn against the winner so far
        const int a2 = hull_resolve(lane == 0 ? u_at : u_win, lane == 0 ? at : lane == 1 ? win : -1, ui, i);
        if (a2 == at) win = at, u_win = u_at;
      }
      next = win;
      mine = win;
      u_mine = u_win;
    }
    const bool flat = !(best > 0.f);
    if (flat) next = P - 1;
    const float u_next = __shfl_sync(0xffffffffu, u_mine, next & 31);
    blocks.add(i, ui, next, u_next, flat, next == P - 1, lane, out);
    ui = u_next;
    i = next;
  }
  if (i == P - 1) return blocks.count;
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (lane + 32 * t >= i && lane + 32 * t < P) {
      us[lane + 32 * t - i] = u[t];
      is[lane + 32 * t - i] = (unsigned short)(lane + 32 * t);
    }
  return kHullWalk + hull_rest(us, is, P - i, out.gain + kHullWalk, out.start + kHullWalk, lane);
}

// ---- long curves: drop the points that lie on or below the chord of their neighbours, until none does ----------------

// Survivors of the first pass that the shared memory of a curve holds; a fifth of the points of a noisy curve survive.
inline int hull_prune_cap(int P) { return (P * 3 / 10 + 63) & ~63; }
constexpr int kHullPasses = 48;

// The survivors of points base .. base + count - 1 behind the cnt (at most cap) there are, when they are too many to be added
// as they are: passes over what is there make room.  Returns how many there are then, or cap + 1 if a pass does not make enough.
__device__ __noinline__ int hull_squeeze(const float* __restrict__ U, int P, int base, int count, float* us, unsigned short* is,
                                         int cnt, int cap, int lane) {
#pragma unroll 1
  for (int v = 0; v < count; v += 32) {
    const int j = base + v + lane, jj = min(j, P - 1);
    const float u = __ldg(U + jj), lim = fmaf(5e-7f, fabsf(u), 2.f * u);
    bool below = false;  // clearly below a chord, as in the first pass
#pragma unroll
    for (int k = 4; k <= 16; k <<= 1)
      if (j >= k && j + k < P) below |= __ldg(U + j - k) + __ldg(U + j + k) > lim;
    const uint32_t kept = __ballot_sync(0xffffffffu, j < P && !below);
    if (cnt + __popc(kept) > cap) cnt = hull_pass(us, is, cnt, lane);
    if (cnt + __popc(kept) > cap) return cap + 1;
    if ((kept >> lane) & 1) {
      const int at = cnt + __popc(kept & ((1u << lane) - 1u));
      us[at] = u;
      is[at] = (unsigned short)j;
    }
    cnt += __popc(kept);
  }
  __syncwarp();
  return cnt;
}

// One warp per curve.  A point on or below the chord of two other points is no vertex of the majorant, whichever points
// they are, so a pass may test all points against their current neighbours at once; a polygon without such a point is the
// majorant.  The first pass reads the curve once and drops what lies clearly below the chord of the points
// 1, 2, 4, 8 or 32 places to either side (4001 points: about 700 stay); the survivors (value and index) are compacted in
// shared memory and tested against their neighbours, exactly, until none is dropped (9 passes over 1900 points in all, 53
// stay).  Where there is no room for 128 points' survivors, those before them go through a pass of their own (hull_squeeze); a
// curve for which that is not enough, or that needs more than kHullPasses, is left to hull_dense_kernel (count -1).  Blocks
// beyond the last positive slope are one block of gain 0.
// Bound by the latency of a warp's own instructions at 27 warps per SM (7300 bytes of shared memory each; the 52 curves of an SM
// are two rounds).  7680 curves of 4001 points: 3.07 ms as one serial stack walk per curve, 0.31 ms as a walk from
// vertex to vertex over chunk maxima, 0.22 ms with neighbours alone in the first pass, 0.157 ms with room
// for two fifths of the points (21 warps per SM, three rounds), 0.140 ms with a point a lane and five exchanges of 32 (chords of 16
// places instead of 32), 0.119 ms now; the profile build 223 and 196 us.  Smooth curves with 2 % noise in the increments (0.29 of
// the points survive) 485 and 475 us a build; without noise (0.65 survive, hull_dense_kernel takes them) 1880 and 1505.
__global__ void __launch_bounds__(32, 27) hull_prune_kernel(const float* __restrict__ curves, HullLists lists, int P, int cap) {
  extern __shared__ float hull_smem[];
  const int hid = blockIdx.x, lane = threadIdx.x;
  const float* U = curves + (size_t)hid * P;
  float* us = hull_smem;                                                    // [cap]
  unsigned short* is = reinterpret_cast<unsigned short*>(hull_smem + cap);  // [cap]
  const uint32_t lt_mask = (1u << lane) - 1u;
  pdl_launch_dependents();
  // Four consecutive points a lane, in aligned 16-byte units (the curve starts `phase` floats into the first one): the points 4, 8
  // and 32 places to either side are whole lanes away, those 1 and 2 places away mostly in the lane itself.  (Loading them instead
  // of exchanging them: 167 us, the shared memory leaves L1 too little room; tests of the ends in every turn: 181, all of them ALU
  // instructions.)
  const int phase = (int)(reinterpret_cast<uintptr_t>(U) >> 2 & 3), last = (P + phase - 1) >> 2;
  const float4* units = reinterpret_cast<const float4*>(U - phase);
  auto load = [&](int q, float (&x)[4]) {
    if (q > 0 && q < last) {
      const float4 v = __ldg(units + q);
      x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
    } else {  // the ends, which may lie inside a unit
#pragma unroll
      for (int c = 0; c < 4; ++c) x[c] = __ldg(U + min(max(4 * q - phase + c, 0), P - 1));
    }
  };
  int cnt = 0;
  float prev[4] = {}, u[4], nxt[4], ahead[4];
  load(lane, u), load(lane + 32, nxt);
#pragma unroll 1
  for (int base = 0; base <= last; base += 32) {  // 32 units
    const int before = cnt, q = base + lane, j0 = 4 * q - phase;
    load(q + 64, ahead);
    float l1[4], r1[4], l2[4], r2[4], l8[4], r8[4];
    auto exchange = [&](int lanes, float (&l)[4], float (&r)[4]) {  // lanes whose value wraps around stand for the units before, or behind
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        l[c] = __shfl_sync(0xffffffffu, lane >= 32 - lanes ? prev[c] : u[c], (lane + 32 - lanes) & 31);
        r[c] = __shfl_sync(0xffffffffu, lane < lanes ? nxt[c] : u[c], (lane + lanes) & 31);
      }
    };
    exchange(1, l1, r1), exchange(2, l2, r2), exchange(8, l8, r8);
    const float x[8] = {l1[2], l1[3], u[0], u[1], u[2], u[3], r1[0], r1[1]};
    // rises of at most a quarter of u are exact in fp32 (late on a curve they are a few units in the last place); the other chords
    // must pass by more than the roundings of the two sides (2.4e-7 |u| where they are close)
    bool keep[4];
    float d1[5], d2[6];
#pragma unroll
    for (int c = 0; c < 5; ++c) d1[c] = x[c + 2] - x[c + 1];
#pragma unroll
    for (int c = 0; c < 6; ++c) d2[c] = x[c + 2] - x[c];
    if (base > 0 && base + 40 < last) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float lim = fmaf(5e-7f, fabsf(u[c]), 2.f * u[c]), small = 0.25f * fabsf(u[c]);
        const float far = fmaxf(fmaxf(l1[c] + r1[c], l2[c] + r2[c]), l8[c] + r8[c]);
        bool below = far > lim;
        if (d1[c] <= d1[c + 1] && fmaxf(fabsf(d1[c]), fabsf(d1[c + 1])) <= small) below = true;
        if (d2[c] <= d2[c + 2] && fmaxf(fabsf(d2[c]), fabsf(d2[c + 2])) <= small) below = true;
        keep[c] = !below;
      }
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float lim = fmaf(5e-7f, fabsf(u[c]), 2.f * u[c]), small = 0.25f * fabsf(u[c]);
        const int j = j0 + c, room = min(j, P - 1 - j);  // points to the nearer end
        bool below = room >= 4 && l1[c] + r1[c] > lim;
        below = below || (room >= 8 && l2[c] + r2[c] > lim) || (room >= 32 && l8[c] + r8[c] > lim);
        below = below || (room >= 1 && d1[c] <= d1[c + 1] && fmaxf(fabsf(d1[c]), fabsf(d1[c + 1])) <= small);
        below = below || (room >= 2 && d2[c] <= d2[c + 2] && fmaxf(fabsf(d2[c]), fabsf(d2[c + 2])) <= small);
        keep[c] = room >= 0 && !below;
      }
    }
    int at = cnt;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint32_t kept = __ballot_sync(0xffffffffu, keep[c]);
      at += __popc(kept & lt_mask);
      cnt += __popc(kept);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (keep[c] && at < cap) {
        us[at] = u[c];
        is[at] = (unsigned short)(j0 + c);
      }
      at += keep[c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) prev[c] = u[c], u[c] = nxt[c], nxt[c] = ahead[c];
    // (not in the first turn: there is room for all of its points)
    if (cnt > cap && before <= cap) cnt = hull_squeeze(U, P, 4 * base - phase, 128, us, is, before, cap, lane);
  }
  int total = -1;
  if (cnt <= cap && (cnt = hull_passes(us, is, cnt, kHullPasses, lane)) > 0)
    total = hull_emit(us, is, cnt, lists.gain + (size_t)hid * (P - 1), lists.start + (size_t)hid * (P - 1), lane);
  if (lane == 0) lists.count[hid] = total;
}

// ---- long curves with many vertices: pool adjacent violators on 32 runs, then join --------------------------------

// Increments per lane: an odd count, so that the lanes' runs start in different banks.
__host__ __device__ inline int hull_run(int P) { return ((P - 1 + 31) / 32) | 1; }
inline size_t hull_dense_smem_bytes(int P) { return (size_t)P * 4 + (size_t)hull_run(P) * 64 + 128; }

// One warp per curve.  Every lane runs the pool-adjacent-violators stack over its run of the curve (a merge or a push per
// turn, so that the lanes stay together), which leaves the hull of the run as a list of block starts.  Then neighbouring
// hulls are joined pairwise, five times: the block across the joint absorbs blocks from the left while their mean does
// not exceed its own and from the right while its own does not exceed theirs, which is where the serial algorithm ends
// up as well (the projection is unique).
__device__ __forceinline__ void hull_dense_curve(const float* __restrict__ curves, const HullLists& lists, int P, int hid,
                                              float* hull_smem, int lane) {
  const float* U = curves + (size_t)hid * P;
  const int run = hull_run(P);
  float* Us = hull_smem;
  unsigned short* Ls = reinterpret_cast<unsigned short*>(Us + P);  // [32][run]
  volatile unsigned short* first = Ls + 32 * run;                  // [32] first entry of the lane's list
  volatile unsigned short* end = first + 32;                       // [32] one past its last entry
#pragma unroll 16
  for (int i = lane; i < P; i += 32) Us[i] = __ldg(U + i);
  __syncwarp();

  // the lane's own run: increments k0 .. k1-1
  const int k0 = min(lane * run, P - 1), k1 = min(k0 + run, P - 1);
  unsigned short* own = Ls + lane * run;
  int sp = 0;
  if (k0 < k1) {
    int k = k0, cur_l = k0, top_l = k0;
    float u_cur = Us[k0], u_next = Us[k0 + 1], u_top = u_cur;
    // the current block is [cur_l, k+1); below it on the stack lies [top_l, cur_l)
    while (k < k1) {
      if (sp > 0 && mean_le(u_top, u_cur, cur_l - top_l, u_cur, u_next, k + 1 - cur_l)) {
        cur_l = top_l;
        u_cur = u_top;
        --sp;
        if (sp > 0) {
          top_l = own[sp - 1];
          u_top = Us[top_l];
        }
      } else {
        own[sp++] = (unsigned short)cur_l;
        top_l = cur_l;
        u_top = u_cur;
        ++k;
        cur_l = k;
        u_cur = u_next;
        if (k < k1) u_next = Us[k + 1];
      }
    }
  }
  first[lane] = 0;
  end[lane] = (unsigned short)sp;

  // join hulls of `width` runs pairwise; the leader of a pair walks
#pragma unroll 1
  for (int width = 1; width < 32; width <<= 1) {
    __syncwarp();
    if ((lane & (2 * width - 1)) == 0) {
      const int last = lane + 2 * width - 1, stop = min((last + 1) * run, P - 1);  // the right hull ends at point `stop`
      int la = lane + width - 1, lb = lane + width;
      while (la > lane && first[la] == end[la]) --la;
      while (lb <= last && first[lb] == end[lb]) ++lb;
      if (lb <= last) {
        // start of the block behind entry `at` of list `list`, or the end of the right hull
        auto next_right = [&](int& list, int& at) {
          ++at;
          while (list <= last && at == end[list]) {
            ++list;
            if (list <= last) at = first[list];
          }
          return list <= last ? (int)Ls[list * run + at] : stop;
        };
        int ea = end[la];                                  // the left hull's last block is entry ea - 1 of list la
        int l = Ls[la * run + ea - 1], m = Ls[lb * run + first[lb]];
        int rl = lb, ra = first[lb];                       // where the right hull goes on
        int r = next_right(rl, ra);
        float ul = Us[l], um = Us[m], ur = Us[r];
        if (mean_le(ul, um, m - l, um, ur, r - m)) {
          bool more = true;
          while (more) {  // the joint block is [l, r)
            more = false;
            int pl = la, pe = ea - 1;                      // the block before it
            while (pl > lane && pe == first[pl]) {
              --pl;
              pe = end[pl];
            }
            if (pe > first[pl]) {
              const int p = Ls[pl * run + pe - 1];
              const float up = Us[p];
              if (mean_le(up, ul, l - p, ul, ur, r - l)) {
                end[la] = (unsigned short)(ea - 1);        // l is no block start any more
                la = pl;                                   // the lists in between are empty
                ea = pe;
                l = p;
                ul = up;
                more = true;
              }
            }
            if (r < stop) {
              int nl = rl, na = ra;
              const int r2 = next_right(nl, na);
              const float u2 = Us[r2];
              if (mean_le(ul, ur, r - l, ur, u2, r2 - r)) {
                r = r2;
                ur = u2;
                rl = nl;
                ra = na;
                more = true;
              }
            }
          }
          // the right hull keeps its blocks from entry ra of list rl on
          for (int i = lb; i < rl && i <= last; ++i) first[i] = end[i];
          if (rl <= last) first[rl] = (unsigned short)ra;
        }
      }
    }
  }
  __syncwarp();

  // the lists one behind the other: block starts and gains
  const int f0 = first[lane], cnt = end[lane] - f0;
  int incl = cnt;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  // end of this lane's last block: the first block start of the next non-empty list
  const uint32_t filled = __ballot_sync(0xffffffffu, cnt > 0);
  const uint32_t above = lane < 31 ? filled & ~((2u << lane) - 1u) : 0u;
  const int my_first = cnt > 0 ? (int)own[f0] : 0;
  const int next_first = __shfl_sync(0xffffffffu, my_first, above ? __ffs(above) - 1 : 0);
  const int tail = above ? next_first : P - 1;
  float* g_out = lists.gain + (size_t)hid * (P - 1) + (incl - cnt);
  unsigned short* s_out = lists.start + (size_t)hid * (P - 1) + (incl - cnt);
  for (int i = 0; i < cnt; ++i) {
    const int l = own[f0 + i], r = i + 1 < cnt ? (int)own[f0 + i + 1] : tail;
    const double mean = __ddiv_rn(__dsub_rn((double)Us[r], (double)Us[l]), (double)(r - l));
    g_out[i] = __double2float_rn(mean > 0.0 ? mean : 0.0);
    s_out[i] = (unsigned short)l;
  }
  if (lane == 0) lists.count[hid] = total;
}
// One warp looks at up to 32 curves at a time, `gridDim` apart, for those that the kernel before left.
__global__ void __launch_bounds__(32) hull_dense_kernel(const float* __restrict__ curves, HullLists lists, int P, int n_curves) {
  extern __shared__ float hull_smem[];
  const int lane = threadIdx.x, step = gridDim.x;
  // (the next launch comes when this one ends: the greedy kernel's CTAs would wait in the shared memory that the CTAs here need)
  pdl_wait();
  for (long long base = blockIdx.x; base < n_curves; base += 32LL * step) {
    const long long mine = base + (long long)lane * step;
    uint32_t todo = __ballot_sync(0xffffffffu, mine < n_curves && lists.count[mine] < 0);
    for (; todo; todo &= todo - 1) {
      __syncwarp();
      hull_dense_curve(curves, lists, P, (int)(base + (long long)(__ffs(todo) - 1) * step), hull_smem, lane);
    }
  }
}

constexpr int kHullRegsMaxP = 32 * 17;

__device__ __forceinline__ int hull_walk_short(const float* U, int P, int lane, HullOut out, float* us, unsigned short* is) {
  if (P <= 96) return hull_walk_regs<3>(U, P, lane, out, us, is);
  if (P <= 160) return hull_walk_regs<5>(U, P, lane, out, us, is);
  if (P <= 288) return hull_walk_regs<9>(U, P, lane, out, us, is);
  return hull_walk_regs<17>(U, P, lane, out, us, is);
}

// One warp (a block of its own) per curve of up to kHullRegsMaxP points.
// Bound by the latency of a step; a curve has few vertices (6 of 257 points on the benchmark's curves).  256 curves of 257
// points: 59 us beside the scorer as one serial stack walk per curve, 6 us now (curves of six vertices).
__global__ void hull_kernel(const float* __restrict__ curves, HullLists lists, int P) {
  __shared__ float us[kHullRegsMaxP];
  __shared__ unsigned short is[kHullRegsMaxP];
  const int hid = blockIdx.x, lane = threadIdx.x;
  const HullOut out = {lists.gain + (size_t)hid * (P - 1), lists.start + (size_t)hid * (P - 1)};
  pdl_launch_dependents();
  const int count = hull_walk_short(curves + (size_t)hid * P, P, lane, out, us, is);
  if (lane == 0) lists.count[hid] = count;
}

// ---- greedy --------------------------------------------------------------------------

constexpr int kGreedyMaxThreads = 1024;
constexpr int kGreedyMaxGroups = 8;
constexpr int kSeqPerLaunch = 128;

struct GreedyArgs {
  long long budget[kSeqPerLaunch];    // B_q
  long long row_base[kSeqPerLaunch];  // packed rows before sequence q
  int T[kSeqPerLaunch];               // context length of sequence q (the curve grid is T/(P-1) tokens per segment)
  int floor_tok[kSeqPerLaunch];       // tokens every head of sequence q keeps at least
  int seq0, count;                    // sequences seq0 .. seq0 + count - 1
  int uniform;                        // all of one length
};

struct SetStride {
  size_t budgets, offsets;  // elements between consecutive curve sets
};

// Tokens for sale in segments [0,c) of a head whose first `floor_tok` tokens were handed to it up
// front (the minimum retention of App. E; 0 = none).
__device__ __forceinline__ int capsum(int c, int seg, int n, int floor_tok) {
  return max(min(c * seg, n) - floor_tok, 0);  // c * seg <= T
}

// Threads that solve one problem together: whole warps, with a barrier of their own.
struct Group {
  int tid, nthr, bar;
  __device__ __forceinline__ void sync() const {
    if (nthr == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nthr) : "memory");
  }
};

// Sums of two values over the group; every thread gets them.  `buf` holds one pair per warp.  One barrier per
// call is enough only if consecutive calls use different buffers: the caller alternates between two.
__device__ __forceinline__ uint2 group_sum2(unsigned a, unsigned b, uint2* buf, const Group& g) {
  a = __reduce_add_sync(0xffffffffu, a);
  b = __reduce_add_sync(0xffffffffu, b);
  const int warps = g.nthr >> 5, lane = g.tid & 31;
  if (warps == 1) return make_uint2(a, b);
  if (lane == 0) buf[g.tid >> 5] = make_uint2(a, b);
  g.sync();
  const uint2 v = lane < warps ? buf[lane] : make_uint2(0u, 0u);
  return make_uint2(__reduce_add_sync(0xffffffffu, v.x), __reduce_add_sync(0xffffffffu, v.y));
}

// Exclusive scan over the group in thread order.  `sums` holds one value per warp; barriers inside.
__device__ __forceinline__ int group_scan(int v, int* sums, const Group& g) {
  const int lane = g.tid & 31, wv = g.tid >> 5;
  int incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  g.sync();  // the previous scan's sums are read
  if (lane == 31) sums[wv] = incl;
  g.sync();
  const int before = __reduce_add_sync(0xffffffffu, lane < wv ? sums[lane] : 0);
  return before + incl - v;
}

// The lists of a curve set as a CTA reads them: staged in shared memory (one behind the other, head h from at[h] on, each
// with one more entry that holds the end of the curve) or in place.
template <bool STAGED>
struct ListView {
  const float* gain_;
  const unsigned short* start_;
  const int* at_;     // staged: [N + 1] where a head's list starts
  const int* count_;  // in place
  int G1;
  __device__ int blocks(int h) const { return STAGED ? at_[h + 1] - at_[h] - 1 : count_[h]; }
  __device__ float gain(int h, int i) const { return STAGED ? gain_[at_[h] + i] : gain_[(size_t)h * G1 + i]; }
  __device__ int start(int h, int i) const {  // first segment of block i; the end of the curve behind the last block
    if (STAGED) return (int)start_[at_[h] + i];
    return i < count_[h] ? (int)start_[(size_t)h * G1 + i] : G1;
  }
};

struct GreedyShared {
  uint2 sum[2][32];
  int scan[32];
  unsigned cut[2];    // gain at which the budget runs out, tokens left for it
  unsigned range[2];  // smallest and largest gain
  unsigned sel[2];    // bin, tokens above it
  unsigned listed;
};
constexpr int kGreedyBins = 512;
constexpr int kGreedyList = kGreedyBins / 2;  // blocks that are ranked directly
constexpr int kGreedyWords = kGreedyBins + 2; // scratch of a group: bins, or a list of pairs

// body(gain bits, tokens) for the staged blocks with from <= gain <= to; the ends of the curves count as blocks without
// capacity.
template <typename Body>
__device__ __forceinline__ void each_block(const ListView<true>& lists, int N, int seg, int n, int floor_tok, unsigned from,
                                           unsigned to, const Group& grp, Body&& body) {
  const int entries = lists.at_[N] - 1;
#pragma unroll 4
  for (int e = grp.tid; e < entries; e += grp.nthr) {
    const unsigned g = __float_as_uint(lists.gain_[e]);
    if (g - from <= to - from)
      body(g, (unsigned)max(0, capsum(lists.start_[e + 1], seg, n, floor_tok) - capsum(lists.start_[e], seg, n, floor_tok)));
  }
}
// Smallest and largest positive gain of the staged lists (bit patterns; from > to: none).
__device__ __forceinline__ void gain_range(const ListView<true>& lists, int N, const Group& grp, GreedyShared& sh,
                                           unsigned& from, unsigned& to) {
  if (grp.tid == 0) {
    sh.range[0] = 0xFFFFFFFFu;
    sh.range[1] = 0u;
  }
  grp.sync();
  from = 0xFFFFFFFFu;
  to = 0u;
  for (int h = grp.tid; h < N; h += grp.nthr) {
    int x = lists.blocks(h) - 1;
    while (x > 0 && lists.gain(h, x) == 0.f) --x;
    const unsigned g = __float_as_uint(lists.gain(h, x));
    if (g != 0u) from = min(from, g);
    to = max(to, __float_as_uint(lists.gain(h, 0)));
  }
  from = __reduce_min_sync(0xffffffffu, from);
  to = __reduce_max_sync(0xffffffffu, to);
  if ((grp.tid & 31) == 0) {
    atomicMin(&sh.range[0], from);
    atomicMax(&sh.range[1], to);
  }
  grp.sync();
  from = sh.range[0];
  to = sh.range[1];
}
__device__ __forceinline__ int bin_bits(unsigned from, unsigned to) { return max(0, 23 - __clz(to - from)); }
// Tokens in the bins at or above each of the kGreedyBins bins (entry kGreedyBins: 0) over the range [from, to].
__device__ __forceinline__ void bins_at_least(const ListView<true>& lists, int N, int seg, int n, int floor_tok, unsigned from,
                                              unsigned to, const Group& grp, GreedyShared& sh, unsigned* bins) {
  for (int x = grp.tid; x <= kGreedyBins; x += grp.nthr) bins[x] = 0u;
  grp.sync();
  const int bits = bin_bits(from, to);
  each_block(lists, N, seg, n, floor_tok, from, to, grp,
             [&](unsigned g, unsigned tokens) { atomicAdd(&bins[(g - from) >> bits], tokens); });
  grp.sync();
  // a thread owns consecutive bins from the top
  const int own = (kGreedyBins + grp.nthr - 1) / grp.nthr, top = kGreedyBins - 1 - grp.tid * own;
  unsigned mine = 0;
  for (int x = top; x > top - own && x >= 0; --x) mine += bins[x];
  unsigned run = (unsigned)group_scan((int)mine, sh.scan, grp);
  for (int x = top; x > top - own && x >= 0; --x) {
    run += bins[x];
    bins[x] = run;
  }
  grp.sync();
}

// The first split of the gains, shared by the problems of a CTA where all have the same grid; bins null: none.
struct FirstSplit {
  const unsigned* bins;
  unsigned from, to;
};

// One problem: sequence i of `args` on the lists of one curve set, by the threads of a group; thread t owns the heads
// [t*per, (t+1)*per) (ONE: the head t).  The greedy buys segments in the order (gain desc, k asc, hid asc) until the
// budget is spent.
//   gain  Staged lists: the capacities of all blocks go into bins along the range of the gains (their bit patterns: a
//         logarithmic scale); the bin in which the budget runs out is split again until it holds at most kGreedyList blocks,
//         of which every thread adds up those that are steeper than its own.  Lists in place: bisection over the bits of the
//         gain; they are sorted by falling gain, so the blocks of a head whose gain agrees with the bits fixed so far form
//         a range [lo,hi); inside it the next bit is 1 up to some index and 0 from there on: one binary search per head
//         and bit (none when the range's ends agree), and the capacities of the 1s, summed over the heads, and the budget
//         decide which half holds the cut.
//   k     Of the segments with exactly that gain (a range [a,e) per head) those with the smaller index are bought
//         first: the index K at which the budget runs out, by bisection; not needed when one head has such segments.
//   hid   Segment K of the heads that have it, in head order, each whole while the budget lasts.
// lo, hi, mid: [N] words per head (unused when ONE).  bins: kGreedyWords words when STAGED.
template <bool STAGED, bool ONE>
__device__ __forceinline__ void greedy_problem(const ListView<STAGED> lists, const GreedyArgs& args, int i, int N, int w,
                                               int* lo, int* hi, int* mid, unsigned* bins, GreedyShared& sh,
                                               const FirstSplit first, const Group grp, int32_t* __restrict__ budgets, int32_t* __restrict__ offsets) {
  const int tid = grp.tid, nthr = grp.nthr, G1 = lists.G1;
  const int per = ONE ? 1 : (N + nthr - 1) / nthr;
  const int h_begin = min(N, tid * per), h_end = min(N, h_begin + per);
  int lo1 = 0, hi1 = 0, mid1 = 0;
  auto LO = [&](int h) -> int& { return ONE ? lo1 : lo[h]; };
  auto HI = [&](int h) -> int& { return ONE ? hi1 : hi[h]; };
  auto MID = [&](int h) -> int& { return ONE ? mid1 : mid[h]; };
  // the sequence's own grid: n rankable positions, seg tokens per curve segment, nseg segments with capacity
  const int n = args.T[i] - w, seg = args.T[i] / G1, nseg = (n + seg - 1) / seg;
  const int floor_tok = args.floor_tok[i], q = args.seq0 + i;
  const long long left = args.budget[i] - (long long)N * floor_tok;  // the floor is spent before the greedy
  const bool all_taken = (long long)N * (n - floor_tok) <= left;
  unsigned R = (unsigned)left;  // budgets are below 2^31
  unsigned round = 0;
  if (!all_taken) {
    if constexpr (STAGED) {
      unsigned from = first.from, to = first.to, gain = 0u;
      if (!first.bins) gain_range(lists, N, grp, sh, from, to);
      const unsigned* at_least = first.bins;                     // of the present range, if known
      bool rank = !at_least && lists.at_[N] - N <= kGreedyList;  // few blocks: no bins
#pragma unroll 1
      while (from <= to) {
        if (rank) {
          if (tid == 0) {
            sh.listed = 0u;
            sh.cut[0] = 0u;
          }
          grp.sync();
          uint2* list = reinterpret_cast<uint2*>(bins);
          auto add = [&](unsigned g, unsigned tokens) {
            const unsigned x = atomicAdd(&sh.listed, 1u);
            if (x < kGreedyList) list[x] = make_uint2(g, tokens);
          };
          if (lists.at_[N] > 8 * nthr) {
            // many blocks: a search in every head's list, which is sorted, instead of a look at all of them (256 heads of 53
            // blocks, 256 threads: 7500 clocks and 900)
            for (int h = h_begin; h < h_end; ++h) {
              const int c = lists.blocks(h);
              int x = 0, r = c;  // first block that is not steeper than the range
              while (x < r) {
                const int m = (x + r) >> 1;
                if (__float_as_uint(lists.gain(h, m)) > to) x = m + 1; else r = m;
              }
              for (; x < c; ++x) {
                const unsigned g = __float_as_uint(lists.gain(h, x));
                if (g < from) break;
                add(g, (unsigned)max(0, capsum(lists.start(h, x + 1), seg, n, floor_tok) - capsum(lists.start(h, x), seg, n, floor_tok)));
              }
            }
          } else {
            each_block(lists, N, seg, n, floor_tok, from, to, grp, add);
          }
          grp.sync();
          const int m = (int)sh.listed;
          if (m <= kGreedyList) {
            unsigned all = 0;
            for (int e0 = 0; e0 < m; e0 += nthr >> 2) {  // four lanes a block
              const int e = e0 + (tid >> 2);
              const uint2 own = e < m ? list[e] : make_uint2(0u, 0u);
              unsigned steeper = 0, same = 0;
#pragma unroll 4
              for (int x = tid & 3; x < m; x += 4) {
                const uint2 o = list[x];
                steeper += o.x > own.x ? o.y : 0u;
                same += o.x == own.x ? o.y : 0u;
              }
#pragma unroll
              for (int off = 1; off < 4; off <<= 1) {
                steeper += __shfl_xor_sync(0xffffffffu, steeper, off);
                same += __shfl_xor_sync(0xffffffffu, same, off);
              }
              if (e < m && steeper <= R && R < steeper + same) {  // one gain; every thread that holds it writes the same
                sh.cut[0] = own.x;
                sh.cut[1] = R - steeper;
              }
              if ((tid & 3) == 0) all += own.y;
            }
            all = group_sum2(all, 0u, sh.sum[round++ & 1], grp).x;
            grp.sync();
            gain = sh.cut[0];
            R = gain != 0u ? sh.cut[1] : R - all;  // else the budget reaches the segments without gain
            break;
          }
          grp.sync();
        }
        if (!at_least) {
          bins_at_least(lists, N, seg, n, floor_tok, from, to, grp, sh, bins);
          at_least = bins;
        }
        if (R >= at_least[0]) {  // the budget reaches the segments without gain
          R -= at_least[0];
          break;
        }
        for (int x = tid; x < kGreedyBins; x += nthr)
          if (at_least[x + 1] <= R && R < at_least[x]) {
            sh.sel[0] = (unsigned)x;
            sh.sel[1] = at_least[x + 1];
          }
        grp.sync();
        const int bits = bin_bits(from, to);
        R -= sh.sel[1];
        from += sh.sel[0] << bits;
        to = min(to, from + ((1u << bits) - 1u));
        if (bits == 0) {
          gain = from;
          break;
        }
        rank = true;
        at_least = nullptr;
        grp.sync();
      }
      const float g = __uint_as_float(gain);
      for (int h = h_begin; h < h_end; ++h) {
        const int c = lists.blocks(h);
        int l = 0, r = c;  // first block that is not steeper than g
        while (l < r) {
          const int m = (l + r) >> 1;
          if (lists.gain(h, m) > g) l = m + 1; else r = m;
        }
        r = l;
        while (r < c && lists.gain(h, r) == g) ++r;
        LO(h) = l;
        HI(h) = r;
      }
    } else {
      for (int h = h_begin; h < h_end; ++h) {
        LO(h) = 0;
        HI(h) = lists.blocks(h);
      }
#pragma unroll 1
      for (int bit = 30; bit >= 0; --bit) {  // gains are not negative
        unsigned local = 0, alive = 0;
        for (int h = h_begin; h < h_end; ++h) {
          const int l = LO(h), r = HI(h);
          int m = l;
          if (l < r) {
            alive += r - l;
            auto bit_at = [&](int k) { return (__float_as_uint(lists.gain(h, k)) >> bit) & 1u; };
            const unsigned bl = bit_at(l), br = bit_at(r - 1);
            if (bl) {
              m = r;
              if (!br) {
                int x = l, y = r - 1;  // bit(x) == 1, bit(y) == 0
#pragma unroll 1
                while (y - x > 1) {
                  const int c = (x + y) >> 1;
                  if (bit_at(c)) x = c; else y = c;
                }
                m = y;
              }
              local += capsum(lists.start(h, m), seg, n, floor_tok) - capsum(lists.start(h, l), seg, n, floor_tok);
            }
          }
          MID(h) = m;
        }
        const uint2 sum = group_sum2(local, alive, sh.sum[round++ & 1], grp);
        if (sum.y <= 1) break;  // the gain of the one block left
        if (sum.x > R) {
          for (int h = h_begin; h < h_end; ++h) HI(h) = MID(h);
        } else {
          R -= sum.x;
          for (int h = h_begin; h < h_end; ++h) LO(h) = MID(h);
        }
      }
    }
  }
  // segments [a,e) of every head have the gain at which the budget runs out, those before a are bought
  unsigned with = 0;
  for (int h = h_begin; h < h_end; ++h) {
    int a = nseg, e = nseg;
    if (!all_taken) {
      a = min(lists.start(h, LO(h)), nseg);
      e = HI(h) > LO(h) ? min(lists.start(h, HI(h)), nseg) : a;
    }
    LO(h) = a;
    HI(h) = e;
    with += e > a;
  }
  const bool tie = group_sum2(with, 0u, sh.sum[round++ & 1], grp).x > 1;
  int K = 0, rank = 0;
  unsigned cap_K = 0;
  if (tie) {
    // largest K with (tokens of the segments below K in the ranges) <= R
    auto below = [&](int k) {
      unsigned local = 0;
      for (int h = h_begin; h < h_end; ++h) {
        const int a = LO(h), e = HI(h);
        local += capsum(min(max(k, a), e), seg, n, floor_tok) - capsum(a, seg, n, floor_tok);
      }
      return group_sum2(local, 0u, sh.sum[round++ & 1], grp).x;
    };
    int top = 1;
    while (top <= nseg) top <<= 1;
    unsigned spent = 0;
#pragma unroll 1
    for (int b = top >> 1; b > 0; b >>= 1) {
      if (K + b > nseg) continue;
      const unsigned s = below(K + b);
      if (s <= R) {
        K += b;
        spent = s;
      }
    }
    R -= spent;
    cap_K = (unsigned)(capsum(K + 1, seg, n, floor_tok) - capsum(K, seg, n, floor_tok));
    int mine = 0;
    for (int h = h_begin; h < h_end; ++h) mine += LO(h) <= K && K < HI(h);
    rank = group_scan(mine, sh.scan, grp);
  }
  // budgets, then offsets = row_base + exclusive scan of (budget + w)
  int rows = 0;
  for (int h = h_begin; h < h_end; ++h) {
    const int a = LO(h), e = HI(h);
    int b = floor_tok + capsum(a, seg, n, floor_tok);
    if (tie) {
      b = floor_tok + capsum(min(max(K, a), e), seg, n, floor_tok);
      if (a <= K && K < e) {
        const unsigned before = (unsigned)rank++ * cap_K;
        b += before < R ? (int)min(cap_K, R - before) : 0;
      }
    } else if (e > a) {
      b += (int)R;
    }
    MID(h) = b;
    rows += b + w;
  }
  long long run = args.row_base[i] + group_scan(rows, sh.scan, grp);
  if (q == 0 && tid == 0) offsets[0] = 0;
  for (int h = h_begin; h < h_end; ++h) {
    budgets[(size_t)q * N + h] = MID(h);
    run += MID(h) + w;
    offsets[(size_t)q * N + h + 1] = (int32_t)run;
  }
  grp.sync();  // the shared words start over
}

// Shared memory of the greedy kernel: at [N+1], the groups' bins, gain and start [cap + N] when lists are staged;
// lo, hi, mid [N] when a thread owns several heads.
// The largest head count must leave room for the static arrays of the form with several heads per thread.
static_assert(sizeof(GreedyShared) + (kGreedyBins + 1) * 4 + 64 + kGreedyMaxHeads * 12 + 4 <= 227 * 1024, "kGreedyMaxHeads");
inline size_t greedy_smem_bytes(int N, int cap, int groups, bool one) {
  const size_t e = (size_t)cap + N, bins = (size_t)groups * kGreedyWords;
  return (cap > 0 ? ((size_t)N + 1) * 4 + e * 4 + ((e * 2 + 3) & ~(size_t)3) + bins * 4 + 4 : 0) +
         (one ? 0 : (size_t)N * 12 + 4);
}

// One CTA per (share of the sequences, curve set), of one or more groups of `group` threads, each with a sequence of its
// own at a time.  The lists of a set are short (6 blocks a head on the benchmark's curves, 53 of 4000 on the calibration
// curves) and are staged in shared memory once for all sequences of the CTA when they fit, else read through L1.
// Bound by latency (a pass over the blocks, a scan, a ranking), hence several groups per CTA where there are that many
// problems.  65536 segments in 256 heads: 91 us beside the scorer with a search per head for each of the 64 bits of (gain,
// k, hid) over expanded segments, 34 us with the bits of the gain over block lists, 16 us now; 2970 problems of
// 256 x 4000 segments 0.6 ms, 0.12 ms, 0.07 ms with the first split shared, 0.056 ms with the cut's blocks searched for and ranked by
// four lanes each.
// blockIdx.y selects one of several independent curve sets (the calibration queries of the offline profile, which
// share the budgets): set i reads the lists of curves i*N .., writes budgets + i*set.budgets and offsets +
// i*set.offsets.  The hot path launches one set.
template <bool ONE>
__global__ void __launch_bounds__(kGreedyMaxThreads) greedy_kernel(HullLists lists, const __grid_constant__ GreedyArgs args,
                                                                   int32_t* __restrict__ budgets,
                                                                   int32_t* __restrict__ offsets, SetStride set,
                                                                   int N, int P, int w, int cap, int group) {
  extern __shared__ __align__(16) unsigned char greedy_smem[];
  pdl_launch_dependents();
  pdl_wait();  // the lists come from the launch before
  __shared__ GreedyShared shared[ONE ? kGreedyMaxGroups : 1];  // several heads per thread: one group (launch_greedy)
  const int groups = blockDim.x / group;
  const int mine = threadIdx.x / group;
  const Group grp = {(int)threadIdx.x - mine * group, group, mine + 1}, all = {(int)threadIdx.x, (int)blockDim.x, 0};
  GreedyShared& sh = shared[mine];
  int* lo = reinterpret_cast<int*>(greedy_smem);     // [N] each, unless ONE
  int* hi = lo + (ONE ? 0 : N);
  int* mid = hi + (ONE ? 0 : N);
  int* at = lo + (ONE ? 0 : (3 * N + 1) & ~1);       // [N + 1]
  unsigned* bins = reinterpret_cast<unsigned*>(at + ((N + 2) & ~1));  // [groups][kGreedyWords], 8-byte aligned
  float* s_gain = reinterpret_cast<float*>(bins + groups * kGreedyWords);
  unsigned short* s_start = reinterpret_cast<unsigned short*>(s_gain + cap + N);

  const int tid = threadIdx.x, nthr = blockDim.x, G1 = P - 1;
  const size_t curve0 = (size_t)blockIdx.y * N;
  budgets += (size_t)blockIdx.y * set.budgets;
  offsets += (size_t)blockIdx.y * set.offsets;
  const int* count = lists.count + curve0;

  bool staged = false;
  if (cap > 0) {
    const int per = (N + nthr - 1) / nthr;
    const int h_begin = min(N, tid * per), h_end = min(N, h_begin + per);
    int local = 0;
    for (int h = h_begin; h < h_end; ++h) local += count[h] + 1;
    int run = group_scan(local, shared[0].scan, all);
    for (int h = h_begin; h < h_end; ++h) {
      at[h] = run;
      run += count[h] + 1;
      if (h == N - 1) at[N] = run;
    }
    __syncthreads();
    staged = at[N] - N <= cap;
    if (staged) {
      // eight lanes per list: four lists of a warp in flight at a time
      const int sub = tid & 7;
#pragma unroll 2
      for (int h = tid >> 3; h < N; h += nthr >> 3) {
        const int a0 = at[h], c = at[h + 1] - a0 - 1;
        const float* g = lists.gain + (curve0 + h) * G1;
        const unsigned short* s = lists.start + (curve0 + h) * G1;
#pragma unroll 4
        for (int x = sub; x <= c; x += 8) {
          s_gain[a0 + x] = x < c ? g[x] : 0.f;
          s_start[a0 + x] = x < c ? s[x] : (unsigned short)G1;
        }
      }
    }
    __syncthreads();
  }
  const ListView<true> in_smem = {s_gain, s_start, at, nullptr, G1};
  const ListView<false> in_place = {lists.gain + curve0 * G1, lists.start + curve0 * G1, nullptr, count, G1};
  unsigned* my_bins = bins + mine * kGreedyWords;
  FirstSplit first = {nullptr, 0u, 0u};
  if (staged && args.uniform && args.count > (int)(gridDim.x * groups)) {  // a group takes several problems of one grid
    __shared__ unsigned first_bins[kGreedyBins + 1];
    gain_range(in_smem, N, all, shared[0], first.from, first.to);
    const int T = args.T[0], n = T - w;
    if (first.from <= first.to)
      bins_at_least(in_smem, N, T / G1, n, args.floor_tok[0], first.from, first.to, all, shared[0], first_bins);
    first.bins = first_bins;
    __syncthreads();  // the groups go their own ways
  }
  for (int i = blockIdx.x * groups + mine; i < args.count; i += gridDim.x * groups) {
    if (staged) greedy_problem<true, ONE>(in_smem, args, i, N, w, lo, hi, mid, my_bins, sh, first, grp, budgets, offsets);
    else greedy_problem<false, ONE>(in_place, args, i, N, w, lo, hi, mid, my_bins, sh, first, grp, budgets, offsets);
  }
}

// Hull and greedy of up to 32 heads in one launch: one CTA per sequence, a warp per head walks the head's curve into
// shared memory (the curves are shared by the sequences; a walk costs less than handing lists over between launches).
// For calls of one or a few layers, where allocation is on the critical path: 8 heads x 129 points 29 + 34 us as two
// kernels before, 7 us now.
constexpr int kSmallMaxHeads = 32;

inline size_t alloc_small_smem_bytes(int N, int P) {
  return (size_t)N * P * 4 + (((size_t)N * P * 2 + 3) & ~(size_t)3);
}

__global__ void __launch_bounds__(32 * kSmallMaxHeads) alloc_small_kernel(const float* __restrict__ curves,
                                                                          const __grid_constant__ GreedyArgs args,
                                                                          int32_t* __restrict__ budgets,
                                                                          int32_t* __restrict__ offsets, int N, int P,
                                                                          int w) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  __shared__ GreedyShared sh;
  __shared__ int at[kSmallMaxHeads + 1];
  __shared__ __align__(8) unsigned bins[kGreedyWords];
  float* gain = reinterpret_cast<float*>(small_smem);                              // [N][P], then packed
  unsigned short* start = reinterpret_cast<unsigned short*>(gain + (size_t)N * P);
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int count = 0;
  if (warp < N) {
    const HullOut out = {gain + (size_t)warp * P, start + (size_t)warp * P};
    count = hull_walk_short(curves + (size_t)warp * P, P, lane, out, out.gain + kHullWalk, out.start + kHullWalk);
    if (lane == 0) {  // the end of the curve
      gain[(size_t)warp * P + count] = 0.f;
      start[(size_t)warp * P + count] = (unsigned short)(P - 1);
      at[warp + 1] = count + 1;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int v = lane < N ? at[lane + 1] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, v, off);
      if (lane >= off) v += o;
    }
    if (lane < N) at[lane + 1] = v;
    if (lane == 0) at[0] = 0;
  }
  __syncthreads();
  // pack the lists, head by head (a list only moves towards the front)
  for (int h = 1; h < N; ++h) {
    const int to = at[h], len = at[h + 1] - to;
    for (int x0 = 0; x0 < len; x0 += blockDim.x) {
      const int x = x0 + threadIdx.x;
      const float g = x < len ? gain[(size_t)h * P + x] : 0.f;
      const unsigned short s = x < len ? start[(size_t)h * P + x] : (unsigned short)0;
      __syncthreads();
      if (x < len) {
        gain[to + x] = g;
        start[to + x] = s;
      }
    }
  }
  __syncthreads();
  const ListView<true> lists = {gain, start, at, nullptr, P - 1};
  const Group grp = {(int)threadIdx.x, (int)blockDim.x, 0};
  greedy_problem<true, true>(lists, args, blockIdx.x, N, w, nullptr, nullptr, nullptr, bins, sh, FirstSplit{nullptr, 0u, 0u}, grp, budgets, offsets);
  pdl_wait();
}

GreedyArgs greedy_args(const Dims& dm, const int64_t* budgets_host, int q0, int cnt, long long* row_base) {
  GreedyArgs args = {};
  for (int i = 0; i < cnt; ++i) {
    args.budget[i] = budgets_host[q0 + i];
    args.row_base[i] = *row_base;
    args.T[i] = dm.seq_T ? dm.seq_T[q0 + i] : dm.T;
    args.floor_tok[i] = dm.seq_T ? seq_floor_tokens(dm, q0 + i) : dm.floor_tok;
    *row_base += budgets_host[q0 + i] + (long long)dm.N * dm.w;
  }
  args.seq0 = q0;
  args.count = cnt;
  args.uniform = dm.seq_T == nullptr;
  return args;
}

}  // namespace

HullLists hull_lists(void* base, int64_t n_curves, int P) {
  HullLists h;
  char* p = static_cast<char*>(base);
  const size_t cells = (size_t)n_curves * (P - 1);
  h.gain = reinterpret_cast<float*>(p);
  h.start = reinterpret_cast<unsigned short*>(p + cells * 4);
  h.count = reinterpret_cast<int*>(p + ((cells * 6 + 3) & ~(size_t)3));
  return h;
}
size_t hull_lists_bytes(int64_t n_curves, int P) {
  return (((size_t)n_curves * (P - 1) * 6 + 3) & ~(size_t)3) + (size_t)n_curves * 4;
}

cudaError_t launch_hull(const float* curves, const HullLists& out, int64_t n_curves, int P, LaunchCtx& lc) {
  const unsigned grid = (unsigned)n_curves;
  if (P <= kHullRegsMaxP) {
    hull_kernel<<<grid, 32, 0, lc.st>>>(curves, out, P);
    lc.mark("hull");
    return cudaGetLastError();
  }
  const int cap = hull_prune_cap(P);
  hull_prune_kernel<<<grid, 32, (size_t)cap * 6, lc.st>>>(curves, out, P, cap);
  lc.mark("hull_prune");
  // as many warps as the chip holds at 25 KB each: all curves may be left to it, most often none is.  (7680 smooth curves: 2180 us a
  // profile build with nine to an SM, which do not fit, and the next launch beside them, 1960 with eight, 1505 with eight alone.)
  const unsigned dense = std::min(grid, 8u * 148u);
  const cudaError_t e = launch_pdl(hull_dense_kernel, dim3(dense), dim3(32), hull_dense_smem_bytes(P), lc.st, true, curves,
                                   out, P, (int)n_curves);
  if (e != cudaSuccess) return e;
  lc.mark("hull_dense");
  return cudaGetLastError();
}

cudaError_t launch_greedy(const Dims& dm, const HullLists& lists, const int64_t* budgets_host, int32_t* budgets,
                          int32_t* offsets, int n_sets, bool one_cta, LaunchCtx& lc) {
  cudaError_t e;
  // lists of up to 16384 blocks in all are staged (two CTAs per SM then); with many heads the per-head words take the room
  const long long cells = (long long)dm.N * (dm.P - 1);
  const int cap = dm.N > 2048 ? 0 : (int)std::min(cells, 16384LL);
  const bool one = dm.N <= kGreedyMaxThreads;
  int group = (dm.N + 31) & ~31;  // one thread per head, whole warps
  if (group > kGreedyMaxThreads) group = kGreedyMaxThreads;
  // several problems per CTA where many sets share the budgets, or where one CTA takes all (never when a thread owns several
  // heads)
  const bool pack = (n_sets > 1 || one_cta) && one;
  const int groups = pack ? std::min(kGreedyMaxGroups, std::max(1, std::min(dm.S, kGreedyMaxThreads / group))) : 1;
  const size_t smem = greedy_smem_bytes(dm.N, cap, groups, one);
  auto kern = one ? greedy_kernel<true> : greedy_kernel<false>;
  if ((e = allow_smem((const void*)kern, smem)) != cudaSuccess) return e;
  SetStride set;
  set.budgets = (size_t)dm.S * dm.N;
  set.offsets = (size_t)dm.S * dm.N + 1;
  long long base = 0;
  for (int q0 = 0; q0 < dm.S; q0 += kSeqPerLaunch) {
    const int cnt = dm.S - q0 < kSeqPerLaunch ? dm.S - q0 : kSeqPerLaunch;
    const GreedyArgs args = greedy_args(dm, budgets_host, q0, cnt, &base);
    // one CTA per sequence; where many sets share the budgets, a set's staged lists serve several of them; beside a
    // persistent scorer a single CTA, which fits the SM that the scorer leaves free
    int ctas = one_cta ? 1 : (cnt + groups - 1) / groups;
    if (n_sets > 1) ctas = std::max(1, std::min(ctas, 2 * 148 / n_sets));
    e = launch_pdl(kern, dim3(ctas, n_sets), dim3(group * groups), smem, lc.st, true, lists, args, budgets, offsets, set,
                   dm.N, dm.P, dm.w, cap, group);
    if (e != cudaSuccess) return e;
    lc.mark("greedy");
  }
  return cudaGetLastError();
}

bool allocate_small(const Dims& dm) { return dm.N <= kSmallMaxHeads && dm.P <= kHullRegsMaxP && dm.S <= kSeqPerLaunch; }

cudaError_t launch_allocate_small(const Dims& dm, const float* curves, const int64_t* budgets_host, int32_t* budgets,
                                  int32_t* offsets, bool beside, LaunchCtx& lc) {
  long long base = 0;
  const GreedyArgs args = greedy_args(dm, budgets_host, 0, dm.S, &base);
  const size_t smem = alloc_small_smem_bytes(dm.N, dm.P);
  cudaError_t e;
  if ((e = allow_smem((const void*)alloc_small_kernel, smem)) != cudaSuccess) return e;
  e = launch_pdl(alloc_small_kernel, dim3(dm.S), dim3(32 * dm.N), smem, lc.st, beside, curves, args, budgets, offsets, dm.N,
                 dm.P, dm.w);
  if (e != cudaSuccess) return e;
  lc.mark("allocate");
  return cudaGetLastError();
}

cudaError_t launch_allocate(const Dims& dm, const float* curves, const int64_t* budgets_host, const HullLists& lists,
                            int32_t* budgets, int32_t* offsets, LaunchCtx& lc) {
  if (allocate_small(dm)) return launch_allocate_small(dm, curves, budgets_host, budgets, offsets, false, lc);
  cudaError_t e = launch_hull(curves, lists, dm.N, dm.P, lc);
  if (e != cudaSuccess) return e;
  return launch_greedy(dm, lists, budgets_host, budgets, offsets, 1, false, lc);
}

}  // namespace lukv
