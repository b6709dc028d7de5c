// Exact solution of the allocation problem on the curves as given (paper Sec. 4.2, Eq.
// "combinatorial_optimization"; the paper names the exact solver as the point of comparison for its
// relaxation): the multiple-choice-knapsack recursion over the heads,
//     f_h(x) = max over b in [0, min(x, n)] of  f_{h-1}(x - b) + U_h(b),      f_{-1}(0) = 0,
// at token resolution (curve point b = utility of keeping b tokens).  Every row f_h is kept, and the walk back from x = B
// looks the choices up again: the smallest b with f_{h-1}(x - b) + U_h(b) == f_h(x), which is the smallest b that attains the
// maximum.
//
// 2.2e11 pairs (x, b) for 256 heads x 3968 tokens at B = 0.3 N n if every one is evaluated.  What is done instead:
//   - tokens that no optimal solution can contain, and budgets on which none can pass, are left out before (see "which tokens
//     can matter" below): 1 % of the budgets and 8 % of the tokens are left there;
//   - of those, a warp owns 64 budgets; where many blocks of 64 values of b are left it skips every one that an upper bound
//     rules out: for any slope s a pair (y, b) can only matter if (f(y) - s y) + (U(b) - s b) reaches the smallest
//     f_h(x) - s x found so far, and maxima of f and U over runs of 16 bound the left side; half a block at a time is then
//     bounded by its own values.  Where a CTA has few blocks all are evaluated, by many warps: the bounds would take longer;
//   - in a block, a pair of additions is one packed instruction and two comparisons are one three-input maximum, on a
//     register tile of 8 budgets x 8 pairs of b per lane; the argmax is not carried along;
//   - all rows in one launch: a CTA keeps its part of the row before and the curve in shared memory and polls the values that
//     others compute themselves, so that a row costs one trip through L2; two narrow rows share one.
// The values are those of the full recursion wherever its solutions pass, bit for bit.
// What bounds it now: the latency of a row's straight-line code (1.8 us: poll, staging, a barrier, an evaluation spread over 18
// warps and its maxima) and of the walk back (0.5 us a head).  256 heads x 3968 tokens, B = 304742: 57.2 ms with every pair
// evaluated one by one and the argmax kept; 3.95 ms with bounds and a launch per row; 2.7 + 0.4 ms in one launch over all
// budgets; 0.99 ms over the tokens that can matter and all budgets that they add up to (rows 0.72, walk 0.20, greedy solution 0.09);
// 0.73 ms with the budgets' bands (335 -> 55 tiles a row: rows 0.69 -> 0.57), steps of narrow rows (0.47) and a walk by one warp
// (0.13).  Three rows a step 745 us, two where a CTA has up to 64, 100 or 160 blocks 733, 748, 753; two tiles to a CTA 776.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace lukv {
namespace {

constexpr int kDpWarps = 20;
constexpr int kDpThreads = 32 * kDpWarps;
constexpr int kDpX = 64;                      // budgets per tile (one warp); values of b per block
constexpr int kDpMaxBlocks = 64;              // n <= 4095: the curve grid has at most 4097 points
constexpr int kDpRun = 16;                    // entries per stored maximum
constexpr int kDpURuns = kDpMaxBlocks * kDpX / kDpRun;  // run maxima per curve
constexpr int kDpSub = 96;                    // most tiles whose part of the previous row is staged together
constexpr int kDpGroup = 80;                  // bytes of 8 packed pairs of f, padded: eight lanes at this stride hit all banks
constexpr int kDpWindow = 112;                // packed pairs of f that a warp makes of 128 values
constexpr int kDpUBlock = 2 * 128;            // bytes of a block's 32 packed pairs of U
constexpr int kDpWindowsPer = ((kDpMaxBlocks + kDpSub) * kDpX / kDpWindow + kDpWarps) / kDpWarps;  // per warp
constexpr int kDpMinTiles = 1;                // least tiles of a CTA in a row
constexpr int kDpWords = 2;                   // status, heads that have their tokens
constexpr int kDpTable = 1024;                // rows whose parts are worked out ahead
constexpr int kDpFewWork = 40;                // blocks of b times tiles that a CTA evaluates without bounds
constexpr int kDpJoin = 2;                    // rows that are made together where they are narrow
constexpr int kDpJoinTiles = 32;              // most tiles of the row before that a narrow step stages
constexpr int kDpStepWarps = kDpWarps - 2;    // warps that evaluate tiles in a narrow step; the others fetch the next curves
constexpr int kDpStepBytes = (kDpJoinTiles * kDpX + kDpWindow) / 8 * kDpGroup;  // one of a narrow step's two buffers of f
constexpr uint32_t kDpUnset = 0xFFFFFFFFu;    // a value that is still to come (a NaN that no addition or maximum makes)
constexpr int kDpBackThreads = 384;

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Maxima of every curve over runs of 16 values of b; -inf beyond n.  One CTA per head; the first also clears the words of
// the next kernel.
__global__ void __launch_bounds__(kDpURuns) dp_runs_kernel(const float* __restrict__ curves, float* __restrict__ runs,
                                                           int* __restrict__ words, int n_words, int n, int P) {
  const float* U = curves + (size_t)blockIdx.x * P;
  const int b0 = threadIdx.x * kDpRun;
  float m = -INFINITY;
  for (int b = b0; b < b0 + kDpRun && b <= n; ++b) m = fmaxf(m, __ldg(U + b));
  runs[(size_t)blockIdx.x * kDpURuns + threadIdx.x] = m;
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < n_words; i += kDpURuns) words[i] = 0;
}

struct DpArgs {
  const float* curves;  // [N][P]
  const float* u_runs;  // [N][kDpURuns]
  float* f;             // [N][stride]
  const int4* rows;     // [N] lowest and highest budget of the row, fewest and most tokens of the head
  int* words;           // [0] the status word
  long long stride;
  int P, N, n;
  uint32_t spin_limit;
  int drop;             // test hook: this CTA stores nothing (-1: none)
};
// Shared memory: the staged part of the previous row as packed pairs and its run maxima; the curve of this head and the
// next one as packed pairs and their run maxima; the rows' parts.
struct DpPlan {
  int blocks, entries, runs_off, u_off, u_blocks, u_bytes, u_runs_off, table_off, total;
};
__host__ __device__ inline DpPlan dp_plan(int n, int N) {
  DpPlan p;
  p.blocks = n / kDpX + 1;
  p.entries = ((p.blocks + kDpSub) * kDpX + kDpWindow - 1) / kDpWindow * kDpWindow;
  p.runs_off = p.entries / 8 * kDpGroup;
  p.u_off = p.runs_off + (p.entries + 32) / kDpRun * 4;
  p.u_off = (p.u_off + 15) & ~15;
  p.u_blocks = p.blocks > kDpJoinTiles ? p.blocks : kDpJoinTiles;
  p.u_bytes = p.u_blocks * kDpUBlock;
  p.u_runs_off = p.u_off + 2 * p.u_bytes;
  p.table_off = p.u_runs_off + 2 * p.blocks * 16;
  p.total = p.table_off + (N < kDpTable ? N : kDpTable) * (32 + 16);
  return p;
}

__device__ __forceinline__ void cp_async4(void* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// 32 values of b for the warp's 64 budgets.  Lane (xg, bg) takes budgets 8 xg .. 8 xg + 7 and, in the two halves of a packed
// pair, b = 4 bg + t and 4 bg + 16 + t, t < 4.  fw: the pairs of f from y = x0 + 8 xg - 4 bg - 20 on (from b = 0), of which
// the first four may be the second half of a padded group (odd); ub: the lane's four pairs of U.
__device__ __forceinline__ void dp_block(const unsigned char* fw, bool odd, const unsigned char* ub, float (&blo)[8],
                                         float (&bhi)[8]) {
  const unsigned char* fm = fw + (odd ? 48 : 32);
  // w[i]: pairs 2 i, 2 i + 1; pair 4 + r - t goes with budget r and value t of b
  const ulonglong2 w[6] = {*reinterpret_cast<const ulonglong2*>(fw),      *reinterpret_cast<const ulonglong2*>(fw + 16),
                           *reinterpret_cast<const ulonglong2*>(fm),      *reinterpret_cast<const ulonglong2*>(fm + 16),
                           *reinterpret_cast<const ulonglong2*>(fw + 80), *reinterpret_cast<const ulonglong2*>(fw + 96)};
#pragma unroll
  for (int t = 0; t < 4; t += 2) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(ub + 8 * t);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int e0 = 4 + r - t, e1 = e0 - 1;
      float a0, a1, b0, b1;
      unpack2(fadd2((e0 & 1) ? w[e0 >> 1].y : w[e0 >> 1].x, u.x), a0, a1);
      unpack2(fadd2((e1 & 1) ? w[e1 >> 1].y : w[e1 >> 1].x, u.y), b0, b1);
      blo[r] = max3(blo[r], a0, b0);
      bhi[r] = max3(bhi[r], a1, b1);
    }
  }
}

// Row h: the budgets [lo, hi], as tiles of 64 (from the tile of lo on, `per` to a CTA), and the blocks of b that it needs,
// of whose halves of 32 only those from byte 0 of `halves` to byte 1 (not included) hold tokens that are left; bit 17: all blocks
// are evaluated, without bounds.
struct __align__(16) DpRow {
  __device__ int half0() const { return halves & 255; }
  __device__ int half1() const { return halves >> 8 & 255; }
  __device__ bool few() const { return halves >> 17 & 1; }
  int lo, hi, tile0, tiles, per, blk0, blocks, halves;
};

// A tile's maxima out of the lanes' parts: a lane gets budgets dp_budget(lane) and the one behind it.
__device__ __forceinline__ int dp_budget(int lane) { return 8 * (lane & 7) + (lane & 16 ? 4 : 0) + (lane & 8 ? 2 : 0); }
__device__ __forceinline__ void dp_merge(const float (&blo)[8], const float (&bhi)[8], int lane, float (&best)[2]) {
  const bool hi16 = lane & 16, hi8 = lane & 8;
  float q[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float a = fmaxf(blo[r], bhi[r]), b = fmaxf(blo[r + 4], bhi[r + 4]);
    q[r] = fmaxf(hi16 ? b : a, __shfl_xor_sync(0xffffffffu, hi16 ? a : b, 16));
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) best[r] = fmaxf(hi8 ? q[r + 2] : q[r], __shfl_xor_sync(0xffffffffu, hi8 ? q[r] : q[r + 2], 8));
}
// Stores those of budgets x, x + 1 that the row has.
__device__ __forceinline__ void dp_store(float* next, int x, int lo, int hi, const float (&best)[2]) {
  if (x >= lo && x + 1 <= hi)
    asm volatile("st.relaxed.gpu.global.v2.f32 [%0], {%1, %2};" ::"l"(next + x), "f"(best[0]), "f"(best[1]) : "memory");
  else if (x >= lo && x <= hi)
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(next + x), "f"(best[0]) : "memory");
  else if (x + 1 >= lo && x + 1 <= hi)
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(next + x + 1), "f"(best[1]) : "memory");
}

// Row h at the 64 budgets from x0 on (those in [lo, hi]) over `blocks` blocks of b.  Blocks and tokens count from the first
// staged block; the staged values start 64 `blocks` budgets below what tile 0 reaches with the first token.  Of a row of few
// blocks, `parts` warps can share a tile (part_s: room for 64 values each).
__device__ __forceinline__ void dp_tile(const unsigned char* F2, const float* f_runs, const unsigned char* U2,
                                        const float4* u_runs, const DpRow& row, int tile, int x0, float* next, int lane,
                                        int part, int parts, float* part_s) {
  const int xg = lane & 7, bg = lane >> 3, blocks = row.blocks, lo = row.lo, hi = row.hi;
  // a sum of two bounds, plus what the rounding of their terms can take away (a few roundings of 2^-24 each)
  auto sum_up = [](float f, float u) { return f + u > -INFINITY ? f + u + 4e-7f * (fabsf(f) + fabsf(u)) : -INFINITY; };
  // Upper bound of (f(y) - s (y - x0)) + (U(b) - s b) over the pairs of block `blk` from the run maxima of its 64 values of
  // b and of its 128 values of y.
  const float4* runs0 = reinterpret_cast<const float4*>(f_runs) + blocks + tile;  // the runs of the tile's own budgets
  auto bound = [&](int blk, float s) {
    if (blk >= blocks) return -INFINITY;
    const float4 um = u_runs[blk];
    const float at = s * (float)(kDpX * blk), s16 = s * (float)kDpRun;
    float f = -INFINITY;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 v = runs0[i - blk - 1];  // four runs from y = x0 - 64 (blk + 1 - i) on
      const float o = (float)(4 * i - 4);
      f = max3(f, max3(v.x - s16 * o, v.y - s16 * (o + 1.f), v.z - s16 * (o + 2.f)), v.w - s16 * (o + 3.f));
    }
    f += at;
    const float u = fmaxf(max3(um.x, um.y - s16, um.z - 2.f * s16), um.w - 3.f * s16) - at;
    return sum_up(f, u);
  };
  auto blocks_where = [&](bool p0, bool p1) {
    const uint32_t m0 = __ballot_sync(0xffffffffu, p0), m1 = __ballot_sync(0xffffffffu, p1);
    return (uint64_t)m0 | ((uint64_t)m1 << 32);
  };
  // packed pairs from y = x0 - 64 (blk + 1) on; a block's packed pairs of U
  auto f_of = [&](int blk) { return F2 + (blocks + tile - blk - 1) * (kDpX / 8) * kDpGroup; };
  // The same bound from the block's own values instead of the run maxima, for its two halves of 32 values of b.
  auto halves = [&](int blk, float s, float& h0, float& h1) {
    const unsigned char* fe = f_of(blk) + (lane >> 3) * kDpGroup + (lane & 7) * 8 + 4;
    const unsigned char* ue = U2 + blk * kDpUBlock + (lane & 15) * 8 + (lane >> 4) * 4;
    const float y = (float)(lane - kDpX * (blk + 1)), b = (float)(kDpX * blk + lane);
    float g[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) g[k] = *reinterpret_cast<const float*>(fe + 4 * k * kDpGroup) - s * (y + 32.f * k);
    const float u0 = warp_max(*reinterpret_cast<const float*>(ue) - s * b);
    const float u1 = warp_max(*reinterpret_cast<const float*>(ue + 128) - s * (b + 32.f));
    const float f0 = warp_max(max3(g[1], g[2], g[3])), f1 = warp_max(max3(g[0], g[1], g[2]));
    h0 = sum_up(f0, u0);
    h1 = sum_up(f1, u1);
  };
  float blo[8], bhi[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) blo[r] = bhi[r] = -INFINITY;
  const int e_lane = 8 * xg - 4 * bg + 12;  // pairs of the lane, from y = x0 - 32 on for half 0
  const bool odd = (bg & 1) == 0;
  const unsigned char* f_lane = F2 + (e_lane >> 3) * kDpGroup + (e_lane & 7) * 8;
  auto evaluate = [&](int blk, int half) {
    dp_block(f_lane + ((blocks + tile - blk) * 8 - 4 - 4 * half) * kDpGroup, odd, U2 + blk * kDpUBlock + half * 128 + bg * 32,
             blo, bhi);
  };
  const int xl = dp_budget(lane);
  float best[2];
  auto merge = [&]() { dp_merge(blo, bhi, lane, best); };
  // smallest f_h(x) - s (x - x0) among the budgets that count, less the rounding of the terms in s
  auto lowest = [&](float s) {
    float neg = -INFINITY;
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (x0 + xl + r >= lo && x0 + xl + r <= hi) neg = fmaxf(neg, s * (float)(xl + r) - best[r]);
    const float low = -warp_max(neg);
    return low - 4e-7f * (s * 8192.f + fabsf(low));
  };
  auto slope = [&](float last, float first) {
    const float s = (last - first) * (1.f / 63.f);
    return s > 0.f && s < 1e30f ? s : 0.f;  // s times a distance of up to 8192 stays a number
  };

  if (row.few()) {
    // few tokens: all of them (bounds would take longer)
#pragma unroll 1
    for (int i = row.half0() + part; i < row.half1(); i += parts) evaluate(i >> 1, i & 1);
    merge();
    if (parts > 1) {
      float2* mine = reinterpret_cast<float2*>(part_s + part * kDpX + xl);
      *mine = make_float2(best[0], best[1]);
      bar_sync(1 + tile, 32 * parts);
      if (part > 0) return;
#pragma unroll 1
      for (int i = 1; i < parts; ++i) {
        const float2 o = mine[i * (kDpX / 2)];
        best[0] = fmaxf(best[0], o.x);
        best[1] = fmaxf(best[1], o.y);
      }
    }
  } else {
    // Any slope gives true bounds; that of the previous row at the same budgets gives close ones.
    const unsigned char* own = F2 + (blocks + tile) * (kDpX / 8) * kDpGroup;
    float s = slope(*reinterpret_cast<const float*>(own + 7 * kDpGroup + 7 * 8 + 4), *reinterpret_cast<const float*>(own + 4));
    float t0 = bound(lane, s), t1 = bound(lane + 32, s);
    const float top = warp_max(fmaxf(t0, t1));
    // the better half of the block with the largest bound first
    const int first = __ffsll((long long)blocks_where(t0 == top, t1 == top)) - 1;
    float h0, h1;
    halves(first, s, h0, h1);
    const int half = h1 > h0;
    evaluate(first, half);
    merge();
    float low = lowest(s);
    bool raised = !(fminf(h0, h1) < low);
    if (raised) evaluate(first, half ^ 1);
    uint64_t todo = blocks_where(t0 > -INFINITY && !(t0 < low), t1 > -INFINITY && !(t1 < low)) & ~(1ull << first);
    if (__popcll(todo) > 4) {  // along the slope of this row the bounds may be closer
      s = slope(__shfl_sync(0xffffffffu, best[1], 31), __shfl_sync(0xffffffffu, best[0], 0));
      t0 = bound(lane, s), t1 = bound(lane + 32, s);
      low = lowest(s);
      todo &= blocks_where(!(t0 < low), !(t1 < low));
    }
    // a block that is not left can raise no budget's value above what it has; the others are looked at once
#pragma unroll 1
    while (todo) {
      const int blk = __ffsll((long long)todo) - 1;
      todo &= todo - 1;
      halves(blk, s, h0, h1);
      if (!(h0 < low)) raised = true, evaluate(blk, 0);
      if (!(h1 < low)) raised = true, evaluate(blk, 1);
    }
    if (raised) merge();
  }
  if (next) dp_store(next, x0 + xl, lo, hi, best);
}

// One row of a narrow step: `count` tiles from tile t0 on, their halves of blocks shared out over kDpStepWarps warps.  The values go to
// `next` (global memory; the tiles from `own` on) and, as staged values of the row behind it, to `onward` (shared memory), where given.
__device__ __forceinline__ void dp_narrow(const unsigned char* F2, const unsigned char* U2, const DpRow& row, int t0, int count,
                                          int own, float* next, unsigned char* onward, const unsigned short* parts_of, int warp,
                                          int lane, float* part_s) {
  const int xg = lane & 7, bg = lane >> 3, e_lane = 8 * xg - 4 * bg + 12, xl = dp_budget(lane);
  const bool odd = (bg & 1) == 0;
  const unsigned char* f_lane = F2 + (e_lane >> 3) * kDpGroup + (e_lane & 7) * 8;
  const int half0 = row.half0(), half1 = row.half1();
  const int parts = min((int)parts_of[min(count, kDpStepWarps)], half1 - half0);
  const int per = parts_of[32 + parts];  // 1024 / parts, rounded up: the quotients below are exact
#pragma unroll 1
  for (int v = warp; v < count * parts; v += kDpStepWarps) {
    const int tile = v * per >> 10, part = v - tile * parts;
    float blo[8], bhi[8], best[2];
#pragma unroll
    for (int r = 0; r < 8; ++r) blo[r] = bhi[r] = -INFINITY;
    const unsigned char* f = f_lane + ((row.blocks + tile) * 8 - 4) * kDpGroup;
#pragma unroll 1
    for (int i = half0 + part; i < half1; i += parts) dp_block(f - 4 * kDpGroup * i, odd, U2 + 128 * i + bg * 32, blo, bhi);
    dp_merge(blo, bhi, lane, best);
    if (parts > 1) {
      float2* mine = reinterpret_cast<float2*>(part_s + v * kDpX + xl);
      *mine = make_float2(best[0], best[1]);
      bar_sync(1 + tile, 32 * parts);
      if (part > 0) break;
#pragma unroll 4
      for (int i = 1; i < parts; ++i) {
        const float2 o = mine[i * (kDpX / 2)];
        best[0] = fmaxf(best[0], o.x);
        best[1] = fmaxf(best[1], o.y);
      }
    }
    const int x = (t0 + tile) * kDpX + xl;
    if (onward) {
      const int e = kDpX * tile + xl;
      const float g0 = x >= row.lo && x <= row.hi ? best[0] : -INFINITY, g1 = x + 1 >= row.lo && x + 1 <= row.hi ? best[1] : -INFINITY;
      float* second = reinterpret_cast<float*>(onward + (e >> 3) * kDpGroup + (e & 7) * 8 + 4);
      second[0] = g0, second[2] = g1;
      if (e >= 16) {  // (the last 16 pairs of a row are never read)
        float* first = reinterpret_cast<float*>(onward + ((e >> 3) - 2) * kDpGroup + (e & 7) * 8);
        first[0] = g0, first[2] = g1;
      }
    }
    if (next && tile >= own) dp_store(next, x, row.lo, row.hi, best);
  }
}

// ---- which tokens can matter -------------------------------------------------------------------------------------
//
// For any slope l, a choice b of head j falls short of c_j = max over b of (U_j(b) - l b) by d_j(b) >= 0, and a solution of
// sum B has the value l B + sum c_j - sum d_j(b_j).  With the value LB of some solution, the choices of an optimal one have
// d_j(b_j) <= l B + sum c_j - LB each.  The recursion adds in fp32: every row's addition errs by at most 2^-24 of the sum, so
// whatever path attains the recursion's result (and with it every place where the walk back finds its target) has a true
// value of at least LB less twice the sum of those errors.  With that allowance the tokens [b0, b1] of a head that are
// left, and the budgets that such tokens add up to, hold every path that the full recursion could return, and the rows
// restricted to them have the full recursion's values on those paths.  l and LB come from the greedy solution of the
// relaxed problem, which is close: 325 of 3968 tokens a head are left on utility curves of 256 heads, and 7 % of the budgets, of
// which the bands (dp_band) leave a sixth.

constexpr int kDpCoreThreads = 256;
__device__ __forceinline__ double dp_warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}
// Sum over the CTA in a fixed order, for all threads.
__device__ __forceinline__ double dp_cta_sum(double v, double* part) {
  v = dp_warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int i = 0; i < kDpCoreThreads / 32; ++i) t += part[i];
  return t;
}

struct DpCore {
  const float* curves;      // [N][P]
  HullLists lists;          // of the curves
  const int32_t* budgets;   // [N] the greedy solution
  double* slope;            // [1]
  double* c;                // [N] c_j
  double* u;                // [N] U_j at the greedy solution
  double* size;             // [N] max |U_j|
  float* f;                 // [N][stride]: before the rows are made, kDpSlopes doubles at the start of each hold the bounds' sums
  long long stride;
  int4* rows;               // [N]
  int* done;                // [1] heads that have their tokens, zero before
  int P, N, n, B;
};
// Slopes whose bounds are used: l and l (1 +- 2^-i), i = 1 .. 7 (15 is l again).  Steps by two lose at most 6 % of a quadratic's
// width; i up to 15 leaves as many budgets.
constexpr int kDpSlopes = 16;
__device__ __forceinline__ double dp_slope(double l, int k) {
  const int i = (k + 1) >> 1;
  return k == 0 || k == kDpSlopes - 1 ? l : l + ((k & 1) ? l : -l) * __longlong_as_double((long long)(1023 - i) << 52);
}
// The slope, every head's c_j, and c_j for the slopes next to it.  One CTA per head.
__global__ void __launch_bounds__(kDpCoreThreads) dp_reduced_kernel(const DpCore a) {
  __shared__ double part[kDpCoreThreads / 32], part_size[kDpCoreThreads / 32];
  __shared__ float gain_s[kDpCoreThreads / 32];
  const int j = blockIdx.x, tid = threadIdx.x;
  // the smallest gain among the blocks that the solution takes from; the largest of all if it takes nothing
  float least = INFINITY, most = 0.f;
  for (int i = tid; i < a.N; i += kDpCoreThreads) {
    const size_t row = (size_t)i * (a.P - 1);
    const int count = a.lists.count[i], b = a.budgets[i];
    if (count < 1) continue;
    most = fmaxf(most, a.lists.gain[row]);
    if (b < 1) continue;
    int lo = 0, hi = count - 1;  // the last block that starts before token b
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((int)a.lists.start[row + mid] < b) lo = mid;
      else hi = mid - 1;
    }
    least = fminf(least, a.lists.gain[row + lo]);
  }
  least = -warp_max(-least);
  if ((tid & 31) == 0) gain_s[tid >> 5] = least;
  __syncthreads();
  for (int i = 0; i < kDpCoreThreads / 32; ++i) least = fminf(least, gain_s[i]);
  if (!(least < INFINITY)) {
    __syncthreads();
    most = warp_max(most);
    if ((tid & 31) == 0) gain_s[tid >> 5] = most;
    __syncthreads();
    for (int i = 0; i < kDpCoreThreads / 32; ++i) most = fmaxf(most, gain_s[i]);
    least = most;
  }
  const double slope = (double)least;
  const float* U = a.curves + (size_t)j * a.P;
  double c = -INFINITY, size = 0.0;
  for (int b = tid; b <= a.n; b += kDpCoreThreads) {
    const double x = (double)__ldg(U + b);
    c = fmax(c, x - slope * b);
    size = fmax(size, fabs(x) < INFINITY ? fabs(x) : INFINITY);  // no number: the greedy solution may be none
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    c = fmax(c, __shfl_xor_sync(0xffffffffu, c, off));
    size = fmax(size, __shfl_xor_sync(0xffffffffu, size, off));
  }
  if ((tid & 31) == 0) {
    part[tid >> 5] = c;
    part_size[tid >> 5] = size;
  }
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < kDpCoreThreads / 32; ++i) {
      c = fmax(c, part[i]);
      size = fmax(size, part_size[i]);
    }
    a.c[j] = c;
    a.size[j] = size;
    a.u[j] = (double)__ldg(U + min(max(a.budgets[j], 0), a.n));
    if (j == 0) *a.slope = slope;
  }
  constexpr int kPer = kDpSlopes / (kDpCoreThreads / 32);  // slopes a warp
  const int lane = tid & 31, k0 = kPer * (tid >> 5);
  double s[kPer], most_at[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) s[k] = -dp_slope(slope, k0 + k), most_at[k] = -INFINITY;
  double at = (double)lane;
  for (int b = lane; b <= a.n; b += 32, at += 32.0) {
    const double x = (double)__ldg(U + b);
#pragma unroll
    for (int k = 0; k < kPer; ++k) most_at[k] = fmax(most_at[k], fma(s[k], at, x));
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) most_at[k] = fmax(most_at[k], __shfl_xor_sync(0xffffffffu, most_at[k], off));
    if (lane == k) reinterpret_cast<double*>(a.f + (size_t)j * a.stride)[k0 + k] = most_at[k];
  }
}

// Every head's tokens; the last CTA to finish makes the rows' budgets of them.
__global__ void __launch_bounds__(kDpCoreThreads) dp_ranges_kernel(const DpCore a) {
  __shared__ double part[kDpCoreThreads / 32];
  __shared__ int range_s[2], last_s;
  const int j = blockIdx.x, tid = threadIdx.x;
  int b0 = a.n, b1 = 0;
  double c = 0.0, u = 0.0, size = 0.0, sizes = 0.0;
  for (int i = tid; i < a.N; i += kDpCoreThreads) {
    c += a.c[i];
    u += a.u[i];
    size += a.size[i];
    sizes += a.size[i] * (double)(a.N - i);  // a head's size is part of its own row's sum and of all later ones
  }
  c = dp_cta_sum(c, part), u = dp_cta_sum(u, part), size = dp_cta_sum(size, part), sizes = dp_cta_sum(sizes, part);
  const double slope = *a.slope;
  double slack = slope * (double)a.B + c - u + 2.0 * (1.001 * sizes * 0x1p-24 + a.N * 0x1p-125);
  slack += 1e-12 * (size + slope * (double)a.n * a.N);  // of the sums here
  if (!(size < 1e37)) slack = INFINITY;               // sums might leave fp32
  const double bar = a.c[j] - slack;
  const float* U = a.curves + (size_t)j * a.P;
  for (int b = tid; b <= a.n; b += kDpCoreThreads)
    if (!((double)__ldg(U + b) - slope * b < bar)) {
      b0 = min(b0, b);
      b1 = max(b1, b);
    }
  if (tid == 0) range_s[0] = a.n, range_s[1] = 0;
  __syncthreads();
  b0 = __reduce_min_sync(0xffffffffu, b0);
  b1 = __reduce_max_sync(0xffffffffu, b1);
  if ((tid & 31) == 0) {
    atomicMin(&range_s[0], b0);
    atomicMax(&range_s[1], b1);
  }
  __syncthreads();
  if (tid == 0) {
    // (no token is left where a curve holds something that is no number: then all are)
    a.rows[j] = range_s[0] <= range_s[1] ? make_int4(0, 0, range_s[0], range_s[1]) : make_int4(0, 0, 0, a.n);
    __threadfence();
    last_s = atomicAdd(a.done, 1) == a.N - 1;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  // sums of the fewest and of the most tokens up to every head, 256 heads at a time
  __shared__ long long sum0_s[kDpCoreThreads / 32], sum1_s[kDpCoreThreads / 32];
  long long carry0 = 0, carry1 = 0, total0 = 0, total1 = 0;
  bool sound = true;
  for (int pass = 0; pass < 2; ++pass) {
    for (int i0 = 0; i0 < a.N; i0 += kDpCoreThreads) {
      const int i = i0 + tid;
      int4 r = make_int4(0, 0, 0, 0);
      if (i < a.N) r = __ldcg(a.rows + i);
      if (pass == 1 && !sound && i < a.N) r.z = 0, r.w = a.n;
      long long s0 = r.z, s1 = r.w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const long long o0 = __shfl_up_sync(0xffffffffu, s0, off), o1 = __shfl_up_sync(0xffffffffu, s1, off);
        if ((tid & 31) >= off) s0 += o0, s1 += o1;
      }
      if ((tid & 31) == 31) sum0_s[tid >> 5] = s0, sum1_s[tid >> 5] = s1;
      __syncthreads();
      long long all0 = carry0, all1 = carry1;
      for (int k = 0; k < kDpCoreThreads / 32; ++k) {
        if (k < (tid >> 5)) s0 += sum0_s[k], s1 += sum1_s[k];
        all0 += sum0_s[k], all1 += sum1_s[k];
      }
      s0 += carry0, s1 += carry1;
      if (pass == 1 && i < a.N) {
        // what the heads behind take at the least and at the most bounds the budget from the other side
        r.x = (int)max(s0, (long long)a.B - (total1 - s1));
        r.y = (int)min(s1, (long long)a.B - (total0 - s0));
        a.rows[i] = r;
      }
      carry0 = all0, carry1 = all1;
      __syncthreads();
    }
    if (pass == 0) {
      total0 = carry0, total1 = carry1, carry0 = carry1 = 0;
      sound = total0 <= a.B && a.B <= total1;  // always, for curves of numbers
      if (!sound) total0 = 0, total1 = (long long)a.N * a.n;
    }
  }
  // running sums over the heads of every slope's c_j, in place; all heads' sums take the place of `size`, and the least value that
  // a solution must have that of `u` (both have been read)
  __shared__ double seg_s[kDpCoreThreads / 32][32];
  const int lane = tid & 31, warp = tid >> 5, per = (a.N + kDpCoreThreads / 32 - 1) / (kDpCoreThreads / 32);
  const int first = warp * per, end = min(a.N, first + per);
  auto sum_at = [&](int i) { return reinterpret_cast<double*>(a.f + (size_t)i * a.stride) + lane; };
  double run = 0.0;
  auto over_heads = [&](bool store) {
    for (int i = first; i < end; i += 8) {
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = i + k < end && lane < kDpSlopes ? __ldcg(sum_at(i + k)) : 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        run += v[k];
        if (store && i + k < end && lane < kDpSlopes) *sum_at(i + k) = run;
      }
    }
  };
  over_heads(false);
  seg_s[warp][lane] = run;
  __syncthreads();
  run = 0.0;
  double all = 0.0;
  for (int i = 0; i < kDpCoreThreads / 32; ++i) {
    if (i < warp) run += seg_s[i][lane];
    all += seg_s[i][lane];
  }
  over_heads(true);
  if (warp == 0 && lane < kDpSlopes) a.size[lane] = all;
  if (tid == 0) a.u[0] = sound ? slope * (double)a.B + c - slack : -INFINITY;
}

// The budgets of row h on which a solution can pass.  With C(l) the sum of c_j(l) over the heads up to h and S(l) that over the
// others, a solution that has x tokens up to h is worth at most C(l) + l x + S(l') + l' (B - x) for any two slopes; where that is
// below the least value that it must have, x does not count.  The heads share the slack here, instead of each having all of it:
// 55 tiles of budgets a row are left on average instead of 333 (256 heads x 3968 tokens).  Lane k takes slope k against all others.
__device__ __forceinline__ int4 dp_band(const DpCore& a, int h, int4 r) {
  const int lane = threadIdx.x & (kDpSlopes - 1);
  const double l = dp_slope(*a.slope, lane), up_to = reinterpret_cast<const double*>(a.f + (size_t)h * a.stride)[lane];
  const double others = a.size[lane] - up_to + l * (double)a.B, need = a.u[0] - up_to;
  int lo = r.x, hi = r.y;
  for (int k = 0; k < kDpSlopes - 1; ++k) {
    const double lk = __shfl_sync(0xffffffffu, l, k), sk = __shfl_sync(0xffffffffu, others, k);
    const double x = (need - sk) / (l - lk);
    if (x > -1e9 && x < 1e9) {  // (a number; not for equal slopes)
      if (l > lk) lo = max(lo, (int)floor(x));
      if (l < lk) hi = min(hi, (int)ceil(x));
    }
  }
  lo = __reduce_max_sync(0xffffffffu, lo);
  hi = __reduce_min_sync(0xffffffffu, hi);
  if (lo <= hi) r.x = lo, r.y = hi;
  return r;
}

__device__ __forceinline__ DpRow dp_row(const DpArgs& a, int h) {
  const int4 v = __ldg(a.rows + h);
  DpRow r;
  r.lo = v.x, r.hi = v.y;
  r.tile0 = r.lo / kDpX;
  r.tiles = r.hi / kDpX - r.tile0 + 1;
  r.per = max(kDpMinTiles, (r.tiles + (int)gridDim.x - 1) / (int)gridDim.x);
  r.blk0 = v.z / kDpX;
  r.blocks = v.w / kDpX - r.blk0 + 1;
  const int skip = v.z / 32 - 2 * r.blk0;
  r.halves = skip | (v.w / 32 - 2 * r.blk0 + 1) << 8 | (r.blocks * min(r.per, r.tiles) <= kDpFewWork) << 17;
  return r;
}

// Marks the values of the rows that are to come, and their vectors' other elements as -inf.  One CTA per row.  `B` (or
// -1: the rows are known, but for the bands): rows of all tokens are made first, those budgets that can still reach B.
__global__ void __launch_bounds__(256) dp_clear_kernel(const DpArgs a, const DpCore core, int4* rows, int B) {
  const int h = blockIdx.x;
  int4 r;
  if (B >= 0) {
    r = make_int4((int)max(0LL, B - (long long)(a.N - 1 - h) * a.n), (int)min((long long)B, (long long)(h + 1) * a.n), 0, a.n);
    if (threadIdx.x == 0) rows[h] = r;
  } else {
    __shared__ int4 row_s;
    if (threadIdx.x < 32) {
      r = dp_band(core, h, rows[h]);
      __syncwarp();
      if (threadIdx.x == 0) row_s = rows[h] = r;
    }
    __syncthreads();  // (the sums at the start of the row are read)
    r = row_s;
  }
  float* f = a.f + (size_t)h * a.stride;
  const float unset = __uint_as_float(kDpUnset);
  for (int y = (r.x & ~3) + 4 * threadIdx.x; y <= r.y; y += 4 * 256)
    *reinterpret_cast<float4*>(f + y) =
        make_float4(y >= r.x ? unset : -INFINITY, y + 1 >= r.x && y + 1 <= r.y ? unset : -INFINITY,
                    y + 2 >= r.x && y + 2 <= r.y ? unset : -INFINITY, y + 3 <= r.y ? unset : -INFINITY);
}

// All rows in one launch.  The tiles of every row are dealt to the CTAs in stretches.  A tile of row h needs f_{h-1} at its
// own budgets and at what the head's tokens take off them: a CTA polls those values themselves, which the CTAs that had them
// store as they get them (every row is kept, so nobody waits to overwrite, and there is no other signal).
__global__ void __launch_bounds__(kDpThreads, 1) dp_rows_kernel(const DpArgs a) {
  extern __shared__ __align__(16) unsigned char dp_smem[];
  __shared__ int next_tile;
  __shared__ volatile int stop_s[2];  // a wait of a narrow step ran out (steps take them in turn)
  __shared__ unsigned short parts_of[64];
  __shared__ __align__(16) float part_s[kDpWarps * kDpX];
  const DpPlan plan = dp_plan(a.n, a.N);
  unsigned char* F2 = dp_smem;                                       // packed pairs (f(y + 16), f(y))
  float* f_runs = reinterpret_cast<float*>(dp_smem + plan.runs_off);
  DpRow* table = reinterpret_cast<DpRow*>(dp_smem + plan.table_off);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = blockIdx.x;
  for (int i = threadIdx.x; i < min(a.N, kDpTable); i += kDpThreads) table[i] = dp_row(a, i);
  __syncthreads();
  // Narrow steps: kDpJoin rows of few blocks (those whose numbers follow a multiple of it), or one.  A CTA makes the values that it
  // needs of all but the last row itself, from the row before all of them, so that one trip through L2 serves all of a step.
  // steps[h]: first tile and number of tiles to be staged, tiles of this CTA in the last row, rows (0: not a narrow step).
  const int listed = min(a.N, kDpTable);
  int4* steps = reinterpret_cast<int4*>(table + listed);
  for (int h = threadIdx.x; h < listed; h += kDpThreads) {
    int4 st = make_int4(0, 0, 0, 0);
    for (int rows = kDpJoin; rows > 0 && st.w == 0; rows = rows > 1 ? 1 : 0) {
      if (h + rows > listed || (rows > 1 && h % rows != 0)) continue;
      const DpRow last = table[h + rows - 1];
      const int mine = min(last.per, last.tiles - cta * last.per);
      int t = last.tile0 + cta * last.per, tiles = min(last.per, last.tiles);  // (the same answer in all CTAs)
      bool narrow = true;
      for (int i = rows - 1; i >= 0; --i) {
        const DpRow r = table[h + i];
        narrow = narrow && tiles * r.blocks <= kDpFewWork;
        tiles += r.blocks;
        t -= r.blk0 + r.blocks;
      }
      if (narrow && tiles <= kDpJoinTiles) st = make_int4(t, tiles - min(last.per, last.tiles) + mine, mine, rows);
    }
    steps[h] = st;
  }
  if (threadIdx.x < 64) {
    const int i = threadIdx.x & 31;
    parts_of[threadIdx.x] = i == 0 ? 1 : threadIdx.x < 32 ? max(1, kDpStepWarps / i) : (1024 + i - 1) / i;
  }
  if (threadIdx.x < 2) stop_s[threadIdx.x] = 0;
  __syncthreads();
  auto row_of = [&](int h) { return h < kDpTable ? table[h] : dp_row(a, h); };
  auto step_of = [&](int h) { return h < listed ? steps[h] : make_int4(0, 0, 0, 0); };
  auto fetch_curve = [&](int h, const DpRow& r, int buf, int at, int warp0) {  // the blocks that the row needs, by warps from warp0 on
    const int tid0 = threadIdx.x - 32 * warp0, threads = kDpThreads - 32 * warp0;
    unsigned char* U2 = dp_smem + plan.u_off + buf * plan.u_bytes + at * kDpUBlock;
    const float* U = a.curves + (size_t)h * a.P + r.blk0 * kDpX;
    const int last = a.n - r.blk0 * kDpX;
    for (int b = tid0; b < r.blocks * kDpX; b += threads) {
      unsigned char* to = U2 + (b >> 5) * 128 + (b & 15) * 8 + ((b >> 4) & 1) * 4;  // pairs (U(b), U(b + 16))
      if (b <= last) cp_async4(to, U + b);
      else *reinterpret_cast<float*>(to) = -INFINITY;
    }
    if (r.few()) return;
    float* ur = reinterpret_cast<float*>(dp_smem + plan.u_runs_off) + buf * plan.blocks * 4;
    for (int i = tid0; i < r.blocks * 4; i += threads)
      cp_async4(ur + i, a.u_runs + (size_t)h * kDpURuns + r.blk0 * 4 + i);
  };
  auto next_row = [&](int h) {  // the next step from row h on in which this CTA has a part
    while (h < a.N) {
      const int4 st = step_of(h);
      if (st.w > 0) {
        if (st.z > 0) break;
        h += st.w;
      } else {
        const DpRow r = row_of(h);
        if (cta * r.per < r.tiles) break;
        ++h;
      }
    }
    return h;
  };
  auto fetch_curves = [&](int h, int buf, int warp0) {
    if (h >= a.N) return;
    const int rows = max(1, step_of(h).w);
    for (int i = 0, at = 0; i < rows; ++i) {
      const DpRow r = row_of(h + i);
      fetch_curve(h + i, r, buf, at, warp0);
      at += r.blocks;
    }
  };
  int h = next_row(0), buf = 0;
  fetch_curves(h, 0, 0);

  // Stages f_{h-1} from budget ybase on (at least 64 `tiles` values); false if a wait ran out.
  auto stage = [&](int h, int ybase, int tiles) -> bool {
    const int old_lo = h > 0 ? row_of(h - 1).lo : 0, old_hi = h > 0 ? row_of(h - 1).hi : 0;
    const float* prev = a.f + (size_t)(h > 0 ? h - 1 : 0) * a.stride;
    const int windows = (tiles * kDpX + kDpWindow - 1) / kDpWindow;
    // f_{h-1} at ybase + 112 i + 4 lane .. + 3 for this warp's windows i
    float4 v[kDpWindowsPer];
    uint32_t left = 0;
#pragma unroll
    for (int k = 0; k < kDpWindowsPer; ++k) {
      const int y = ybase + kDpWindow * (warp + k * kDpWarps) + 4 * lane;
      v[k] = make_float4(h == 0 && y == 0 ? 0.f : -INFINITY, -INFINITY, -INFINITY, -INFINITY);
      if (h > 0 && warp + k * kDpWarps < windows && y + 3 >= old_lo && y <= old_hi) left |= 1u << k;
    }
    bool ok = true;
    for (uint32_t spins = 0; left;) {
#pragma unroll
      for (int k = 0; k < kDpWindowsPer; ++k)
        if (left >> k & 1)
          asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(v[k].x), "=f"(v[k].y), "=f"(v[k].z), "=f"(v[k].w)
                       : "l"(prev + ybase + kDpWindow * (warp + k * kDpWarps) + 4 * lane)
                       : "memory");
#pragma unroll
      for (int k = 0; k < kDpWindowsPer; ++k)
        if (__float_as_uint(v[k].x) != kDpUnset && __float_as_uint(v[k].y) != kDpUnset &&
            __float_as_uint(v[k].z) != kDpUnset && __float_as_uint(v[k].w) != kDpUnset)
          left &= ~(1u << k);
      if (left && (++spins >= a.spin_limit || ((spins & 255) == 0 && *reinterpret_cast<volatile int*>(a.words) != 0))) {
        atomicExch(a.words, (int)LUKV_ERR_TIMEOUT);
        ok = false;
        break;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!__syncthreads_and(ok)) return false;  // (and the tiles before have been read)
    if (threadIdx.x == 0) next_tile = kDpWarps;
#pragma unroll
    for (int k = 0; k < kDpWindowsPer; ++k) {
      const int i = warp + k * kDpWarps;
      if (i < windows) {
        // lane l >= 4 holds the first parts of pairs 4 l - 16 .. + 3, lane l - 4 their second parts
        const float g0 = __shfl_up_sync(0xffffffffu, v[k].x, 4), g1 = __shfl_up_sync(0xffffffffu, v[k].y, 4);
        const float g2 = __shfl_up_sync(0xffffffffu, v[k].z, 4), g3 = __shfl_up_sync(0xffffffffu, v[k].w, 4);
        if (lane >= 4) {
          float4* to_s = reinterpret_cast<float4*>(F2 + (kDpWindow / 8 * i + ((lane - 4) >> 1)) * kDpGroup + (lane & 1) * 32);
          to_s[0] = make_float4(v[k].x, g0, v[k].y, g1);
          to_s[1] = make_float4(v[k].z, g2, v[k].w, g3);
        }
        float m = fmaxf(max3(v[k].x, v[k].y, v[k].z), v[k].w);
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        if ((lane & 3) == 0 && (lane < 28 || i == windows - 1)) f_runs[kDpWindow / kDpRun * i + (lane >> 2)] = m;
      }
    }
    __syncthreads();
    return true;
  };

  bool settled = true;  // no warp may still read staged values of a step that is not narrow
  int turn = 0;
  int side = 0;         // buffer that the next narrow step is staged in: none of its warps may still read from it
  for (int h_next = a.N; h < a.N; h = h_next, buf ^= 1) {
    const int4 st = step_of(h);
    if (st.w > 0) {
      // f_{h-1} from the first tile on, a window of 112 values a warp; no barrier ahead of the stores: the step before ended in
      // the other buffer
      if (!settled) __syncthreads();
      settled = true;
      unsigned char* F = F2 + side * kDpStepBytes;
      if (warp * kDpWindow < st.y * kDpX) {
        const int y = st.x * kDpX + kDpWindow * warp + 4 * lane;
        float4 v = make_float4(h == 0 && y == 0 ? 0.f : -INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (h > 0) {
          const DpRow* before = table + h - 1;
          if (y + 3 >= before->lo && y <= before->hi) {
            const float* from = a.f + (size_t)(h - 1) * a.stride + y;
            for (uint32_t spins = 0;;) {
              asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                           : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(from) : "memory");
              if (__float_as_uint(v.x) != kDpUnset && __float_as_uint(v.y) != kDpUnset && __float_as_uint(v.z) != kDpUnset &&
                  __float_as_uint(v.w) != kDpUnset)
                break;
              if (++spins >= a.spin_limit || ((spins & 255) == 0 && *reinterpret_cast<volatile int*>(a.words) != 0)) {
                atomicExch(a.words, (int)LUKV_ERR_TIMEOUT);
                stop_s[turn] = 1;
                break;
              }
            }
          }
        }
        __syncwarp();
        const float g0 = __shfl_up_sync(0xffffffffu, v.x, 4), g1 = __shfl_up_sync(0xffffffffu, v.y, 4);
        const float g2 = __shfl_up_sync(0xffffffffu, v.z, 4), g3 = __shfl_up_sync(0xffffffffu, v.w, 4);
        if (lane >= 4) {
          float4* to_s = reinterpret_cast<float4*>(F + (kDpWindow / 8 * warp + ((lane - 4) >> 1)) * kDpGroup + (lane & 1) * 32);
          to_s[0] = make_float4(v.x, g0, v.y, g1);
          to_s[1] = make_float4(v.z, g2, v.w, g3);
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      if (stop_s[turn]) return;
      turn ^= 1;
      h_next = next_row(h + st.w);
      const bool next_narrow = step_of(h_next).w > 0;
      if (warp >= kDpStepWarps && next_narrow) fetch_curves(h_next, buf ^ 1, kDpStepWarps);
      const unsigned char* U2 = dp_smem + plan.u_off + buf * plan.u_bytes;
      int t0 = st.x, count = st.y;
#pragma unroll 1
      for (int i = 0; i < st.w; ++i) {
        const DpRow row = table[h + i];
        t0 += row.blk0 + row.blocks;
        count -= row.blocks;
        if (i > 0) __syncthreads();
        // The row's top st.z tiles are this CTA's to store (the walk back reads every row), and all of them the first one's.
        if (warp < kDpStepWarps)
          dp_narrow(F2 + (side ^ (i & 1)) * kDpStepBytes, U2, row, t0, count, cta == 0 ? 0 : count - st.z,
                    cta != a.drop ? a.f + (size_t)(h + i) * a.stride : nullptr,
                    i + 1 < st.w ? F2 + (side ^ (~i & 1)) * kDpStepBytes : nullptr, parts_of, warp, lane, part_s);
        U2 += row.blocks * kDpUBlock;
      }
      side = (side + st.w) & 1;
      if (!next_narrow) fetch_curves(h_next, buf ^ 1, 0);
      continue;
    }
    settled = false;
    const DpRow row = row_of(h);
    const int tile0 = row.tile0 + cta * row.per, tiles = min(row.per, row.tiles - cta * row.per);
    float* next = a.f + (size_t)h * a.stride;
    const unsigned char* U2 = dp_smem + plan.u_off + buf * plan.u_bytes;
    const float4* u_runs = reinterpret_cast<const float4*>(dp_smem + plan.u_runs_off) + buf * plan.blocks;
    for (int t_sub = 0; t_sub < tiles; t_sub += kDpSub) {
      const int n_sub = min(kDpSub, tiles - t_sub), xs = (tile0 + t_sub) * kDpX;
      const int ybase = xs - (row.blk0 + row.blocks) * kDpX;
      if (!stage(h, ybase, row.blocks + n_sub)) return;

      // several warps to a tile where there are few, one warp to several tiles (as they come: they differ in what there is to
      // look at) where there are many; warps without one fetch the next curve at once
      const int halves = row.half1() - row.half0();
      const int parts = row.few() ? max(1, min(kDpWarps / n_sub, halves)) : 1, busy = n_sub * parts;
      if (busy <= kDpWarps) {
        const bool last = t_sub + n_sub == tiles;
        if (warp < busy) {
          const int tile = warp / parts;
          dp_tile(F2, f_runs, U2, u_runs, row, tile, xs + tile * kDpX, cta != a.drop ? next : nullptr, lane,
                  warp - tile * parts, parts, part_s + tile * parts * kDpX);
        }
        if (last) {
          h_next = next_row(h + 1);
          const int from = busy < kDpWarps ? busy : 0;
          if (warp >= from) fetch_curves(h_next, buf ^ 1, from);
        }
      } else {
        for (int tile = warp; tile < n_sub;) {
          dp_tile(F2, f_runs, U2, u_runs, row, tile, xs + tile * kDpX, cta != a.drop ? next : nullptr, lane, 0, 1, part_s);
          if (lane == 0) tile = atomicAdd(&next_tile, 1);
          tile = __shfl_sync(0xffffffffu, tile, 0);
        }
        if (t_sub + n_sub == tiles) {
          h_next = next_row(h + 1);
          fetch_curves(h_next, buf ^ 1, 0);
        }
      }
    }
  }
}

// Walks back from x = B; also writes the optimum and the packed-row offsets of this sequence, and clears the word
// of the next sequence's heads.  One CTA; the chain over the heads is serial.  A step compares the head's tokens (one load of
// f_{h-1} and one of U each, one barrier); what a step kWalkAhead heads on can read is touched meanwhile, so that it is in
// L1 by then: the budget falls by what the tokens allow.  The value at the budget that a step arrives at comes with the match.
constexpr int kWalkAhead = 4;
__global__ void __launch_bounds__(kDpBackThreads) dp_backtrack_kernel(const DpArgs a, int B, int w, long long row_base, int q,
                                                                      int32_t* __restrict__ budgets,
                                                                      int32_t* __restrict__ offsets,
                                                                      double* __restrict__ values) {
  constexpr int kWarps = kDpBackThreads / 32;
  __shared__ int match_b[2][kWarps];
  __shared__ float match_f[2][kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, N = a.N;
  const bool failed = a.words[0] != 0;
  __syncthreads();
  if (tid == 0) a.words[1] = 0;
  if (tid == 0 && q == 0) offsets[0] = 0;
  if (failed) {  // a wait of the rows' kernel ran out: no solution
    if (tid == 0) values[q] = __longlong_as_double(0x7FF8000000000000LL);
    for (int h = tid; h < N; h += kDpBackThreads) {
      budgets[(size_t)q * N + h] = 0;
      offsets[(size_t)q * N + h + 1] = (int32_t)(row_base + (long long)(h + 1) * w);
    }
    return;
  }
  int x = B;
  float target = __ldg(a.f + (size_t)(N - 1) * a.stride + B);
  if (tid == 0) values[q] = (double)target;
  auto touch = [](const float* p) { asm volatile("{\n\t.reg .f32 t;\n\tld.global.nc.f32 t, [%0];\n\t}" ::"l"(p)); };
  int4 row = __ldg(a.rows + N - 1);
  for (int h = N - 1; h >= 0; --h) {
    const int4 old = h > 0 ? __ldg(a.rows + h - 1) : make_int4(0, 0, 0, 0);
    const float* prev = a.f + (size_t)max(h - 1, 0) * a.stride;
    const float* U = a.curves + (size_t)h * a.P;
    int mine = 1 << 30;
    float mine_f = 0.f;
#pragma unroll 4
    for (int b = row.z + tid; b <= row.w; b += kDpBackThreads) {
      const int y = x - b;
      if (y >= old.x && y <= old.y) {
        const float e = h > 0 ? __ldg(prev + y) : 0.f;
        if (mine == 1 << 30 && e + __ldg(U + b) == target) {
          mine = b;
          mine_f = e;
        }
      }
    }
    const int least = __reduce_min_sync(0xffffffffu, mine);
    if (mine == least && (mine < (1 << 30) || lane == 0)) {  // one lane: every b is one thread's
      match_b[h & 1][warp] = least;
      match_f[h & 1][warp] = mine_f;
    }
    const int ahead = h - kWalkAhead;
    if (ahead > 0) {
      long long down0 = 0, down1 = 0;  // fewest and most tokens until then
#pragma unroll
      for (int i = 0; i < kWalkAhead; ++i) {
        const int4 r = __ldg(a.rows + h - i);
        down0 += r.z, down1 += r.w;
      }
      const int4 r = __ldg(a.rows + ahead);
      const long long y0 = max((long long)__ldg(a.rows + ahead - 1).x, x - down1 - r.w) & ~31LL, y1 = x - down0 - r.z;
      if (y0 + 32LL * tid <= y1) touch(a.f + (size_t)(ahead - 1) * a.stride + y0 + 32 * tid);
      if (r.z + 32 * tid <= r.w + 31) touch(a.curves + (size_t)ahead * a.P + min(r.z + 32 * tid, r.w));
    }
    __syncthreads();
    const int theirs = lane < kWarps ? match_b[h & 1][lane] : 1 << 30;
    const float theirs_f = lane < kWarps ? match_f[h & 1][lane] : 0.f;
    const int found = __reduce_min_sync(0xffffffffu, theirs);
    // a match exists for finite curves; without one, as many tokens as there are
    const int b = found < (1 << 30) ? found : min(x, a.n);
    if (tid == 0) {
      budgets[(size_t)q * N + h] = b;
      // the rows up to and with head h: x tokens and the windows
      offsets[(size_t)q * N + h + 1] = (int32_t)(row_base + x + (long long)(h + 1) * w);
    }
    x -= b;
    target = __shfl_sync(0xffffffffu, theirs_f, __ffs(__ballot_sync(0xffffffffu, theirs == found)) - 1);
    if (found == 1 << 30 && h > 0) target = __ldg(prev + x);
    row = old;
  }
}

// The same where few tokens of a head are left: one warp walks, its step a load out of L1 (a lane has eight values of b), a comparison
// and a reduction, no barrier; the curve's values and the next rows' ranges are asked for a step ahead.  The other warps bring
// what the steps up to kWalkReach heads on can read into L1, following the walk through shared memory.
constexpr int kWalkWarps = 8, kWalkReach = 8, kWalkPer = 8;
__global__ void __launch_bounds__(32 * kWalkWarps) dp_walk_kernel(const DpArgs a, int B, int w, long long row_base, int q,
                                                                  int32_t* __restrict__ budgets, int32_t* __restrict__ offsets,
                                                                  double* __restrict__ values) {
  __shared__ volatile unsigned long long at_s;  // the step the walk is at: head << 32 | budget
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = a.N;
  const bool failed = a.words[0] != 0;
  if (threadIdx.x == 0) at_s = (unsigned long long)(N - 1) << 32 | (uint32_t)B;
  __syncthreads();
  if (threadIdx.x == 0) {
    a.words[1] = 0;
    if (q == 0) offsets[0] = 0;
  }
  if (failed) {  // a wait of the rows' kernel ran out: no solution
    if (threadIdx.x == 0) values[q] = __longlong_as_double(0x7FF8000000000000LL);
    for (int h = threadIdx.x; h < N; h += 32 * kWalkWarps) {
      budgets[(size_t)q * N + h] = 0;
      offsets[(size_t)q * N + h + 1] = (int32_t)(row_base + (long long)(h + 1) * w);
    }
    return;
  }
  if (warp > 0) {
    auto touch = [](const float* p) { asm volatile("{\n\t.reg .f32 t;\n\tld.global.nc.f32 t, [%0];\n\t}" ::"l"(p)); };
    for (int t = N - warp; t > 0; t -= kWalkWarps - 1) {
      int h = 0, x = 0;
      for (int spin = 0; spin < 1 << 20; ++spin) {
        const unsigned long long at = at_s;
        h = (int)(at >> 32), x = (int)(uint32_t)at;
        if (h - t <= kWalkReach) break;
      }
      if (h < t) continue;
      // what the heads from t + 1 to h take at the least and at the most, then this one's tokens
      int4 r = make_int4(0, 0, 0, 0);
      if (lane <= h - t && lane <= kWalkReach) r = __ldg(a.rows + t + lane);
      const long long y1 = x - (long long)__reduce_add_sync(0xffffffffu, r.z);
      const long long y0 = max((long long)__ldg(a.rows + t - 1).x, x - (long long)__reduce_add_sync(0xffffffffu, r.w)) & ~31LL;
      for (long long y = y0 + 32 * lane; y <= y1; y += 32 * 32) touch(a.f + (size_t)(t - 1) * a.stride + y);
      const int z = __shfl_sync(0xffffffffu, r.z, 0), most = __shfl_sync(0xffffffffu, r.w, 0);
      for (int b = z + 32 * lane; b <= most + 31; b += 32 * 32) touch(a.curves + (size_t)t * a.P + min(b, most));
    }
    return;
  }
  int x = B;
  float target = __ldg(a.f + (size_t)(N - 1) * a.stride + B);
  if (lane == 0) values[q] = (double)target;
  const int4 nothing = make_int4(0, 0, 0, 0);
  int4 row = __ldg(a.rows + N - 1), old = N > 1 ? __ldg(a.rows + N - 2) : nothing;
  const float* prev = a.f + (size_t)max(N - 2, 0) * a.stride;
  const float* U = a.curves + (size_t)(N - 1) * a.P;
  int32_t* out_b = budgets + (size_t)q * N + N - 1;
  int32_t* out_o = offsets + (size_t)q * N + N;
  int rows = (int)(row_base + (long long)N * w);  // the windows' rows up to and with head h
  const float none = __uint_as_float(kDpUnset);   // equals nothing
  for (int h = N - 1; h > 0; --h) {
    const int4 older = __ldg(a.rows + max(h - 2, 0));
    // the tokens of the head with which the row before has a value
    const int b0 = max(row.z, x - old.y), last = min(row.w, x - old.x);
    int found = 1 << 30;
    for (int b1 = b0 + lane; b1 - lane <= last; b1 += 32 * kWalkPer) {
      const float* ep = prev + (x - b1);
      const float* up = U + b1;
      float e[kWalkPer], u[kWalkPer];
#pragma unroll
      for (int k = 0; k < kWalkPer; ++k) {
        const bool in = b1 + 32 * k <= last;
        e[k] = in ? __ldg(ep - 32 * k) : none;
        u[k] = in ? __ldg(up + 32 * k) : 0.f;
      }
      int mine = 1 << 30;
#pragma unroll
      for (int k = kWalkPer - 1; k >= 0; --k)
        if (e[k] + u[k] == target) mine = b1 + 32 * k;
      found = __reduce_min_sync(0xffffffffu, mine);
      if (found < 1 << 30) break;
    }
    // a match exists for finite curves; without one, as many tokens as there are
    const int b = found < (1 << 30) ? found : min(x, a.n);
    if (lane == 0) {
      *out_b = b;
      *out_o = rows + x;  // the rows up to and with head h: x tokens and the windows
      at_s = (unsigned long long)(h - 1) << 32 | (uint32_t)(x - b);
    }
    x -= b;
    target = __ldg(prev + x);
    --out_b, --out_o, rows -= w;
    prev -= h > 1 ? a.stride : 0, U -= a.P;
    row = old, old = older;
  }
  // the first head: what is left
  if (lane == 0) {
    const float u = row.z <= x && x <= row.w ? __ldg(U + x) : none;
    *out_b = u == target ? x : min(x, a.n);
    *out_o = rows + x;
  }
}

size_t align256x(size_t x) { return (x + 255) & ~(size_t)255; }
// floats of one row f_h: rows start on 256-byte boundaries
size_t dp_stride(int64_t budget) { return align256x(((size_t)budget + 1) * sizeof(float)) / sizeof(float); }
}  // namespace

// the rows' values; the curves' run maxima; the words; the heads' c, u, size and the slope; the rows; the hull lists
struct DpSpace {
  size_t f, u_runs, words, core, rows, hull, total;
};
static DpSpace dp_space(const Dims& dm, int64_t max_budget) {
  DpSpace s;
  s.f = 0;
  s.u_runs = (size_t)dm.N * dp_stride(max_budget) * sizeof(float);
  s.words = s.u_runs + align256x((size_t)dm.N * kDpURuns * sizeof(float));
  s.core = s.words + align256x(kDpWords * sizeof(int));
  s.rows = s.core + align256x((3 * (size_t)dm.N + 1) * sizeof(double));
  s.hull = s.rows + align256x((size_t)dm.N * sizeof(int4));
  s.total = s.hull + hull_lists_bytes(dm.N, dm.P);
  return s;
}
size_t exact_workspace_bytes(const Dims& dm, int64_t max_budget) { return dp_space(dm, max_budget).total; }

cudaError_t launch_exact_allocate(const Dims& dm, const float* curves, const int64_t* budgets_host, int32_t* budgets,
                                  int32_t* offsets, double* values, void* ws, LaunchCtx& lc) {
  if (dm.n / kDpX + 1 > kDpMaxBlocks) return cudaErrorInvalidValue;
  cudaError_t e;
  int sms = 0;
  if ((e = device_sms(&sms)) != cudaSuccess) return e;
  const size_t smem = dp_plan(dm.n, dm.N).total;
  if ((e = allow_smem((const void*)dp_rows_kernel, smem)) != cudaSuccess) return e;
  int64_t most = 0;
  for (int q = 0; q < dm.S; ++q) most = std::max(most, budgets_host[q]);
  const DpSpace at = dp_space(dm, most);
  char* base = static_cast<char*>(ws);
  float* u_runs = reinterpret_cast<float*>(base + at.u_runs);
  DpArgs a;
  a.curves = curves;
  a.u_runs = u_runs;
  a.rows = reinterpret_cast<int4*>(base + at.rows);
  a.words = reinterpret_cast<int*>(base + at.words);
  a.f = reinterpret_cast<float*>(base + at.f);
  a.P = dm.P, a.N = dm.N, a.n = dm.n;
  score_test_hooks(&a.spin_limit, &a.drop);
  DpCore c;
  c.curves = curves;
  c.lists = hull_lists(base + at.hull, dm.N, dm.P);
  c.slope = reinterpret_cast<double*>(base + at.core);
  c.c = c.slope + 1, c.u = c.c + dm.N, c.size = c.u + dm.N;
  c.rows = reinterpret_cast<int4*>(base + at.rows);
  c.done = a.words + 1;
  c.P = dm.P, c.N = dm.N, c.n = dm.n;
  dp_runs_kernel<<<(unsigned)dm.N, kDpURuns, 0, lc.st>>>(curves, u_runs, a.words, kDpWords, dm.n, dm.P);
  lc.mark("dp_runs");
  // the greedy solutions of all sequences; each is read before the walk overwrites it.  They and what is made of them cost 30 to
  // 90 us and shorten a row by up to 5 us: 16 heads x 968 tokens 92 us with them and 67 without, x 1968 100 and 90, x 3968 121
  // and 170; 32 x 568 117 and 110, x 968 127 both, x 3968 166 and 295; 48 x 268 133 and 130, x 468 137 and 155; 128 x 68 237 and
  // 247.  (From 16 heads on also because kDpSlopes sums find room in what N heads have.)
  const bool greedy = dm.N >= kDpSlopes && (int64_t)dm.N * dm.N * dm.n >= 600000 && dm.N <= kGreedyMaxHeads;
  if (greedy) {
    if ((e = launch_hull(curves, c.lists, dm.N, dm.P, lc)) != cudaSuccess) return e;
    if ((e = launch_greedy(dm, c.lists, budgets_host, budgets, offsets, 1, false, lc)) != cudaSuccess) return e;
  }
  long long row_base = 0;
  for (int q = 0; q < dm.S; ++q) {
    c.B = (int)budgets_host[q];  // below 2^31, as the packed rows
    c.budgets = budgets + (size_t)q * dm.N;
    a.stride = (long long)dp_stride(c.B);
    c.f = a.f, c.stride = a.stride;
    if (greedy) {
      dp_reduced_kernel<<<(unsigned)dm.N, kDpCoreThreads, 0, lc.st>>>(c);
      lc.mark("dp_reduced");
      dp_ranges_kernel<<<(unsigned)dm.N, kDpCoreThreads, 0, lc.st>>>(c);
      lc.mark("dp_ranges");
    }
    dp_clear_kernel<<<(unsigned)dm.N, 256, 0, lc.st>>>(a, c, c.rows, greedy ? -1 : c.B);
    lc.mark("dp_clear");
    void* params[] = {(void*)&a};
    // cooperative launch: CTAs wait for one another, so all must be resident
    const int ctas = std::min(sms, c.B / kDpX / kDpMinTiles + 1);
    e = cudaLaunchCooperativeKernel((const void*)dp_rows_kernel, dim3((unsigned)ctas), dim3(kDpThreads), params, smem, lc.st);
    if (e != cudaSuccess) return e;
    lc.mark("dp_rows");
    // (tokens left out: mostly a few hundred a head are left)
    if (greedy) dp_walk_kernel<<<1, 32 * kWalkWarps, 0, lc.st>>>(a, c.B, dm.w, row_base, q, budgets, offsets, values);
    else dp_backtrack_kernel<<<1, kDpBackThreads, 0, lc.st>>>(a, c.B, dm.w, row_base, q, budgets, offsets, values);
    lc.mark("dp_backtrack");
    row_base += c.B + (long long)dm.N * dm.w;
  }
  return cudaGetLastError();
}

}  // namespace lukv
