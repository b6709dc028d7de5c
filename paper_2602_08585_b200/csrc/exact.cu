// Exact solution of the allocation problem on the curves as given (paper Sec. 4.2, Eq.
// "combinatorial_optimization"; the paper names the exact solver as the point of comparison for its
// relaxation): the multiple-choice-knapsack recursion over the heads,
//     f_h(x) = max over b in [0, min(x, n)] of  f_{h-1}(x - b) + U_h(b),      f_{-1}(0) = 0,
// at token resolution (curve point b = utility of keeping b tokens).  One launch per head.  Only the states
// that can still reach sum b = B are evaluated: after head h, x lies in [B - (N-1-h)*n, (h+1)*n].  Every row
// f_h is kept, and the walk back from x = B looks the choices up again: the smallest b with
// f_{h-1}(x - b) + U_h(b) == f_h(x), which is the smallest b that attains the maximum.
//
// What bounds it: additions and comparisons (2.2e11 pairs for 256 heads x 3968 tokens at B = 0.3 N n) if every pair is
// evaluated, then the latency of a step.  Three measures:
//   - a warp owns 64 budgets and skips every block of 64 values of b that an upper bound rules out: with s the slope of
//     f_h over its budgets, a pair (y, b) can only matter if (f(y) - s y) + (U(b) - s b) reaches the smallest
//     f_h(x) - s x found so far, and maxima of f and U over runs of 16 bound the left side (every step leaves the maxima
//     of its row for the next one).  On utility curves the blocks far from the optimum drop out (6 % are evaluated); on
//     curves where they do not, everything is evaluated.  The values are those of the full recursion, bit for bit: a
//     skipped block holds no pair that could raise a maximum;
//   - in a block, a pair of additions is one packed instruction and two comparisons are one three-input maximum, on a
//     register tile of 8 budgets x 8 pairs of b per lane; the argmax is not carried along;
//   - warps share nothing (a block's 128 values of f and 64 of U go through a warp's own shared memory), and a step
//     starts while the one before it drains.
// Measured (256 heads x 3968 tokens, B = 304742): 57.2 ms with every pair evaluated one by one and the argmax kept
// (220 us a head); 3.9 ms now, 13 us a head, of which a warp's 2 to 4 dependent reads of L2 are the larger part, and
// 0.47 ms for the walk back.  Tried: f and U staged once per CTA (5.4 ms: staging costs more than the few blocks that are
// left), 32 instead of 20 warps per SM at 64 registers (4.5 ms, spills), three blocks fetched ahead (4.1 ms).
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace lukv {
namespace {

constexpr int kDpWarps = 4;
constexpr int kDpThreads = 32 * kDpWarps;
constexpr int kDpX = 64;                      // budgets per warp; values of b per block
constexpr int kDpTile = kDpX * kDpWarps;      // budgets per CTA
constexpr int kDpMaxBlocks = 64;              // n <= 4095: the curve grid has at most 4097 points
constexpr int kDpRun = 16;                    // entries per stored maximum
constexpr int kDpURuns = kDpMaxBlocks * kDpX / kDpRun;  // run maxima per curve
constexpr int kDpGroup = 80;                  // bytes of 8 packed entries, padded: eight lanes at this stride hit all banks
constexpr int kDpBackThreads = 384;
constexpr int kDpFBytes = 12 * kDpGroup, kDpUBytes = 4 * kDpGroup;

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Maxima of every curve over runs of 16 values of b; -inf beyond n.  One CTA per head.
__global__ void __launch_bounds__(kDpURuns) dp_runs_kernel(const float* __restrict__ curves, float* __restrict__ runs, int n,
                                                           int P) {
  const float* U = curves + (size_t)blockIdx.x * P;
  const int b0 = threadIdx.x * kDpRun;
  float m = -INFINITY;
  for (int b = b0; b < b0 + kDpRun && b <= n; ++b) m = fmaxf(m, __ldg(U + b));
  runs[(size_t)blockIdx.x * kDpURuns + threadIdx.x] = m;
}

struct DpStep {
  const float* U;          // curve of this head
  const float* u_runs;     // its run maxima
  const float* prev;       // f_{h-1}, or null for the first head (f = 0 at y = 0)
  const float* prev_runs;  // maxima of f_{h-1} over runs of 16, for the runs of the tiles that hold [plo, phi]
  float* next;             // f_h
  float* next_runs;
  int lo, hi;              // budgets to evaluate
  int plo, phi;            // where prev is defined; anything outside counts as -inf
  int n;
};

// What a lane fetches of one block: f at y0 + 4 lane .. + 3, U at b0 + lane and b0 + 32 + lane.
struct DpFetch {
  float4 f;
  float u0, u1;
};
__device__ __forceinline__ DpFetch dp_fetch(const DpStep& a, int x0, int blk, int lane) {
  DpFetch r;
  r.f = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  const int y = x0 - kDpX * (blk + 1) + 4 * lane;  // a multiple of 4, as the rows' start
  if (y + 3 >= a.plo && y <= a.phi) {
    const float4 v = a.prev ? *reinterpret_cast<const float4*>(a.prev + y) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (y >= a.plo) r.f.x = v.x;  // y <= phi here
    if (y + 1 >= a.plo && y + 1 <= a.phi) r.f.y = v.y;
    if (y + 2 >= a.plo && y + 2 <= a.phi) r.f.z = v.z;
    if (y + 3 <= a.phi) r.f.w = v.w;
  }
  const int b = kDpX * blk + lane;
  r.u0 = b <= a.n ? __ldg(a.U + b) : -INFINITY;
  r.u1 = b + 32 <= a.n ? __ldg(a.U + b + 32) : -INFINITY;
  return r;
}

// Stores the fetched block packed for dp_block.  F2: entry j (0..95) = (f(yw + 32 + j), f(yw + j)), yw the first of the
// block's 128 values of y; U2: entry t (0..31) = (U(b0 + t), U(b0 + 32 + t)); groups of 8 entries at a padded stride.
__device__ __forceinline__ void dp_store(const DpFetch& r, unsigned char* F2, unsigned char* U2, int lane) {
  // lane l >= 8 holds the first parts of entries 4 l - 32 .. + 3, lane l - 8 their second parts
  const float g0 = __shfl_up_sync(0xffffffffu, r.f.x, 8), g1 = __shfl_up_sync(0xffffffffu, r.f.y, 8);
  const float g2 = __shfl_up_sync(0xffffffffu, r.f.z, 8), g3 = __shfl_up_sync(0xffffffffu, r.f.w, 8);
  float4* to = reinterpret_cast<float4*>(F2 + ((lane - 8) >> 1) * kDpGroup + (lane & 1) * 32);
  if (lane >= 8) {
    to[0] = make_float4(r.f.x, g0, r.f.y, g1);
    to[1] = make_float4(r.f.z, g2, r.f.w, g3);
  }
  *reinterpret_cast<float2*>(U2 + (lane >> 3) * kDpGroup + (lane & 7) * 8) = make_float2(r.u0, r.u1);
}

// One block of b for the warp's 64 budgets.  Lane (xg, bg) takes budgets 8 xg .. 8 xg + 7 and, in the two halves of a
// packed pair, b = 8 bg + t and 8 bg + 32 + t, t < 8: the 16 entries of F2 from group xg - bg + 3 on.
__device__ __forceinline__ void dp_block(const unsigned char* fw, const unsigned char* ub, float (&blo)[8], float (&bhi)[8]) {
  // entry 8 + r - t pairs budget r with value t of b; the window slides down as t grows
  ulonglong2 w[8];  // w[i]: entries 2 i, 2 i + 1
#pragma unroll
  for (int i = 3; i < 8; ++i)
    w[i] = *reinterpret_cast<const ulonglong2*>(fw + (i >> 2) * kDpGroup + (i & 3) * 16);
#pragma unroll
  for (int t = 0; t < 8; t += 2) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(ub + 8 * t);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int e0 = 8 + r - t, e1 = e0 - 1;
      float a0, a1, b0, b1;
      unpack2(fadd2((e0 & 1) ? w[e0 >> 1].y : w[e0 >> 1].x, u.x), a0, a1);
      unpack2(fadd2((e1 & 1) ? w[e1 >> 1].y : w[e1 >> 1].x, u.y), b0, b1);
      blo[r] = max3(blo[r], a0, b0);
      bhi[r] = max3(bhi[r], a1, b1);
    }
    if (t < 6) {
      const int i = 2 - t / 2;
      w[i] = *reinterpret_cast<const ulonglong2*>(fw + i * 16);
    }
  }
}

__global__ void __launch_bounds__(kDpThreads, 5) dp_step_kernel(const DpStep a) {
  __shared__ __align__(16) unsigned char dp_smem[kDpWarps][kDpFBytes + kDpUBytes];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int x0 = (a.lo & ~(kDpX - 1)) + (int)blockIdx.x * kDpTile + warp * kDpX;
  unsigned char* F2 = dp_smem[warp];
  unsigned char* U2 = F2 + kDpFBytes;
  const int xg = lane & 7, bg = lane >> 3;
  const unsigned char* fw = F2 + (xg - bg + 3) * kDpGroup;
  const unsigned char* ub = U2 + bg * kDpGroup;

  pdl_launch_dependents();
  pdl_wait();
  if (x0 > a.hi) return;  // whole warps; nothing below waits for another warp

  // Upper bound of (f(y) - s (y - x0)) + (U(b) - s b) over the pairs of block `blk` from the run maxima of its 64 values of
  // b and of its 128 values of y, and the size of its terms.  The maxima are read again for every check (L1 holds them):
  // registers decide how many tiles an SM has in flight.
  auto bound = [&](int blk, float s, float& size) {
    const float4 um = __ldg(reinterpret_cast<const float4*>(a.u_runs) + blk);
    const float at = s * (float)(kDpX * blk), s16 = s * (float)kDpRun;
    float f = -INFINITY;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      // four runs from y = x0 - 64 (blk + 1 - i) on; the tiles of the previous row start at multiples of 64
      const int y = x0 - kDpX * (blk + 1 - i);
      float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      if (y + kDpX - 1 >= a.plo && y <= a.phi) {
        if (a.prev) v = *reinterpret_cast<const float4*>(a.prev_runs + y / kDpRun);
        else v.x = 0.f;
      }
      const float o = (float)(4 * i - 4);
      f = max3(f, max3(v.x - s16 * o, v.y - s16 * (o + 1.f), v.z - s16 * (o + 2.f)), v.w - s16 * (o + 3.f));
    }
    f += at;
    const float u = fmaxf(max3(um.x, um.y - s16, um.z - 2.f * s16), um.w - 3.f * s16) - at;
    size = fabsf(f) + fabsf(u);
    return f + u;
  };
  auto blocks_where = [&](bool p0, bool p1) {
    const uint32_t m0 = __ballot_sync(0xffffffffu, p0), m1 = __ballot_sync(0xffffffffu, p1);
    return (uint64_t)m0 | ((uint64_t)m1 << 32);
  };

  float blo[8], bhi[8], best[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) blo[r] = bhi[r] = best[r] = -INFINITY;
  float s = 0.f, low = -INFINITY;
  uint64_t done = 0;
#pragma unroll 1
  for (;;) {
    // the blocks still to be evaluated: those whose bound comes within the rounding of these expressions (every
    // term carries a few roundings of 2^-24) of `low`; the one with the largest bound goes first
    float size0, size1;
    float t0 = bound(lane, s, size0), t1 = bound(lane + 32, s, size1);
    const float lin = s * 8192.f + fabsf(low);
    const bool any = !(low > -INFINITY);
    const uint64_t todo = blocks_where(t0 > -INFINITY && (any || t0 + 4e-7f * (size0 + lin) >= low),
                                       t1 > -INFINITY && (any || t1 + 4e-7f * (size1 + lin) >= low)) & ~done;
    if (!todo) break;
    if (!((todo >> lane) & 1)) t0 = -INFINITY;
    if (!((todo >> (lane + 32)) & 1)) t1 = -INFINITY;
    const float top = warp_max(fmaxf(t0, t1));
    const uint64_t first = blocks_where(t0 == top, t1 == top) & todo;
    // alone while `low` still rises a lot (the first time), then together with all others
    uint64_t batch = done ? todo : first & (~first + 1);
    done |= batch;
    DpFetch cur = dp_fetch(a, x0, __ffsll((long long)batch) - 1, lane);
#pragma unroll 1
    do {
      // the same bound once more, from the block's own values instead of the run maxima: what passed on the slack of the
      // runs alone (up to 16 tokens on either side) drops out before the 4096 pairs are formed
      const int blk = __ffsll((long long)batch) - 1;
      batch &= batch - 1;
      const float y4 = (float)(4 * lane - kDpX * (blk + 1)), b1 = (float)(kDpX * blk + lane);
      const float fmax = warp_max(fmaxf(max3(cur.f.x - s * y4, cur.f.y - s * (y4 + 1.f), cur.f.z - s * (y4 + 2.f)),
                                        cur.f.w - s * (y4 + 3.f)));
      const float umax = warp_max(fmaxf(cur.u0 - s * b1, cur.u1 - s * (b1 + 32.f)));
      const bool keep = any || fmax + umax + 4e-7f * (fabsf(fmax) + fabsf(umax) + lin) >= low;
      if (keep) {
        __syncwarp();
        dp_store(cur, F2, U2, lane);
        __syncwarp();
      }
      if (batch) cur = dp_fetch(a, x0, __ffsll((long long)batch) - 1, lane);
      if (keep) dp_block(fw, ub, blo, bhi);
    } while (batch);
    // f_h of the tile so far, its slope, and the smallest f_h(x) - s (x - x0) among the budgets that count
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float m = fmaxf(blo[r], bhi[r]);
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
      best[r] = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    }
    s = (__shfl_sync(0xffffffffu, best[7], 7) - __shfl_sync(0xffffffffu, best[0], 0)) * (1.f / 63.f);
    if (!(s > 0.f && s < 1e30f)) s = 0.f;  // s times a distance of up to 8192 stays a number
    float neg = -INFINITY;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int x = x0 + 8 * xg + r;
      if (x >= a.lo && x <= a.hi) neg = fmaxf(neg, s * (float)(8 * xg + r) - best[r]);
    }
    low = -warp_max(neg);
  }

  // the row, and its maxima over runs of 16 (budgets outside [lo, hi] count as -inf)
  const int x = x0 + 8 * xg;
  float run = -INFINITY;
#pragma unroll
  for (int r = 0; r < 8; ++r)
    if (x + r >= a.lo && x + r <= a.hi) run = fmaxf(run, best[r]);
  run = fmaxf(run, __shfl_xor_sync(0xffffffffu, run, 1));
  if (bg == 0) {
    if (!(xg & 1)) __stcg(a.next_runs + x / kDpRun, run);
    if (x >= a.lo && x + 7 <= a.hi) {  // rows start at multiples of 64 floats, x is a multiple of 8
      __stcg(reinterpret_cast<float4*>(a.next + x), make_float4(best[0], best[1], best[2], best[3]));
      __stcg(reinterpret_cast<float4*>(a.next + x + 4), make_float4(best[4], best[5], best[6], best[7]));
    } else {
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (x + r >= a.lo && x + r <= a.hi) __stcg(a.next + x + r, best[r]);
    }
  }
}

// Walks back from x = B; also writes the optimum and the packed-row offsets of this sequence.  One CTA; the chain over
// the heads is serial and a step reads f_{h-1} at up to n + 1 places (one L2 latency and one barrier), so the next row
// is asked for while a step runs, and the next head's curve is staged in shared memory.
__global__ void __launch_bounds__(kDpBackThreads) dp_backtrack_kernel(const float* __restrict__ curves, int P,
                                                                      const float* __restrict__ f, long long stride,
                                                                      long long B, int N, int n, int w,
                                                                      long long row_base, int q,
                                                                      int32_t* __restrict__ budgets,
                                                                      int32_t* __restrict__ offsets,
                                                                      double* __restrict__ values) {
  constexpr int kVecs = 3;  // 16-byte vectors of f per thread: 12 * 384 places cover n + 4
  constexpr int kUPer = (kDpMaxBlocks * kDpX + kDpBackThreads - 1) / kDpBackThreads;
  __shared__ float Us[2][kDpMaxBlocks * kDpX];
  __shared__ int first_b[3];
  const int tid = threadIdx.x;
  long long x = B;
  float target = f[(size_t)(N - 1) * stride + B];
  if (tid == 0) {
    values[q] = (double)target;
    first_b[0] = first_b[1] = first_b[2] = 1 << 30;
    if (q == 0) offsets[0] = 0;
  }
  for (int b = tid; b <= n; b += kDpBackThreads) Us[(N - 1) & 1][b] = __ldg(curves + (size_t)(N - 1) * P + b);
  __syncthreads();
  for (int h = N - 1; h >= 0; --h) {
    const float* prev = h > 0 ? f + (size_t)(h - 1) * stride : nullptr;
    const long long plo = h > 0 ? max(0LL, B - (long long)(N - h) * n) : 0;
    const long long phi = h > 0 ? min(B, (long long)h * n) : 0;
    // y = x - b for b = 0 .. n, as aligned vectors of four from the top down
    const int top = (int)(x & 3);
    float4 v[kVecs];
#pragma unroll
    for (int i = 0; i < kVecs; ++i) {
      const long long y = (x & ~3LL) - 4LL * (tid + i * kDpBackThreads);
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (prev && y + 3 >= max(plo, x - n) && y <= phi) v[i] = __ldcg(reinterpret_cast<const float4*>(prev + y));
    }
    float u_next[kUPer];
#pragma unroll
    for (int i = 0; i < kUPer; ++i) {
      const int b = tid + i * kDpBackThreads;
      u_next[i] = h > 0 && b <= n ? __ldg(curves + (size_t)(h - 1) * P + b) : 0.f;
    }
    if (h > 1) {  // x falls by at most n a head: what the next step reads lies within 2 n
      const long long y = x - 2LL * n + (long long)tid * 32;
      if (tid <= n / 16 + 1 && y >= 0 && y <= x)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(f + (size_t)(h - 2) * stride + y));
    }
    const float* U = Us[h & 1];
    int mine = 1 << 30;
#pragma unroll
    for (int i = kVecs - 1; i >= 0; --i) {
      const float e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int b = top - c + 4 * (tid + i * kDpBackThreads);
        const long long y = x - b;
        if (b >= 0 && b <= n && y >= plo && y <= phi && e[c] + U[b] == target) mine = min(mine, b);
      }
    }
#pragma unroll
    for (int i = 0; i < kUPer; ++i) {
      const int b = tid + i * kDpBackThreads;
      if (b <= n) Us[(h + 1) & 1][b] = u_next[i];
    }
    mine = __reduce_min_sync(0xffffffffu, mine);
    if ((tid & 31) == 0 && mine < (1 << 30)) atomicMin(&first_b[h % 3], mine);
    __syncthreads();
    const int b = (int)min((long long)first_b[h % 3], min(x, (long long)n));  // a match exists for finite curves
    if (tid == 0) {
      first_b[(h + 1) % 3] = 1 << 30;  // the slot of the step before, which every thread has read: for two steps on
      budgets[(size_t)q * N + h] = b;
      // the rows up to and with head h: x tokens and the windows
      offsets[(size_t)q * N + h + 1] = (int32_t)(row_base + x + (long long)(h + 1) * w);
    }
    x -= b;
    if (prev) target = __ldcg(prev + x);
  }
}

size_t align256x(size_t x) { return (x + 255) & ~(size_t)255; }
// floats of one row f_h: rows start on 256-byte boundaries
size_t dp_stride(int64_t budget) { return align256x(((size_t)budget + 1) * sizeof(float)) / sizeof(float); }

}  // namespace

size_t exact_workspace_bytes(const Dims& dm, int64_t max_budget) {
  const size_t stride = dp_stride(max_budget);
  // the rows, two sets of run maxima, the curves' run maxima
  return ((size_t)dm.N * stride + 2 * (stride / kDpRun + kDpX) + (size_t)dm.N * kDpURuns) * sizeof(float);
}

cudaError_t launch_exact_allocate(const Dims& dm, const float* curves, const int64_t* budgets_host, int32_t* budgets,
                                  int32_t* offsets, double* values, void* ws, LaunchCtx& lc) {
  if (dm.n / kDpX + 1 > kDpMaxBlocks) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kDpThreads);
  cfg.stream = lc.st;
  // a step may start while the one before it drains
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cudaError_t e;
  float* u_runs = static_cast<float*>(ws);
  dp_runs_kernel<<<(unsigned)dm.N, kDpURuns, 0, lc.st>>>(curves, u_runs, dm.n, dm.P);
  lc.mark("dp_runs");
  long long row_base = 0;
  for (int q = 0; q < dm.S; ++q) {
    const long long B = budgets_host[q];
    const size_t stride = dp_stride(B), runs = stride / kDpRun + kDpX;
    float* f_runs = u_runs + (size_t)dm.N * kDpURuns;
    float* f = f_runs + 2 * runs;
    DpStep st;
    st.plo = st.phi = 0;
    st.prev = st.prev_runs = nullptr;
    st.n = dm.n;
    for (int h = 0; h < dm.N; ++h) {
      st.U = curves + (size_t)h * dm.P;
      st.u_runs = u_runs + (size_t)h * kDpURuns;
      st.next = f + (size_t)h * stride;
      st.next_runs = f_runs + (size_t)(h & 1) * runs;
      st.lo = (int)std::max(0LL, B - (long long)(dm.N - 1 - h) * dm.n);  // B < 2^31, as the packed rows
      st.hi = (int)std::min(B, (long long)(h + 1) * dm.n);
      cfg.gridDim = dim3((unsigned)((st.hi - (st.lo & ~(kDpX - 1))) / kDpTile + 1));
      // the first step of a sequence waits for all before it: its rows overwrite what the last walk reads, and it
      // reads the curves' run maxima
      cfg.numAttrs = h > 0 ? 1 : 0;
      if ((e = cudaLaunchKernelEx(&cfg, dp_step_kernel, st)) != cudaSuccess) return e;
      lc.mark("dp_step");
      st.plo = st.lo;
      st.phi = st.hi;
      st.prev = st.next;
      st.prev_runs = st.next_runs;
    }
    dp_backtrack_kernel<<<1, kDpBackThreads, 0, lc.st>>>(curves, dm.P, f, (long long)stride, B, dm.N, dm.n, dm.w, row_base,
                                                         q, budgets, offsets, values);
    lc.mark("dp_backtrack");
    row_base += B + (long long)dm.N * dm.w;
  }
  return cudaGetLastError();
}

}  // namespace lukv
