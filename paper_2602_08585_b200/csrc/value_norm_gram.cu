// Value norms of the oracle importance (Sec. 4.1, Eq. "oracle_importance"; App. E) through the Gram matrix of the projection:
//   vnorm[u][g][j]^2 = || v_j W ||^2 = v_j (W W^T) v_j^T ,   W = W_O^(g) [d][D_model], bf16.
// The direct contraction (value_norm_tc.cu) costs d D_model multiplications per position; here they are 1.7 d^2, and d^2
// D_model once per projection slice.
//
// One persistent CTA per SM, one item = (projection slice, run of 128-position tiles of the sequences that use it):
//   warp 0      TMA producer of value tiles (128 positions x d channels)
//   warp 1      TMA producer of projection panels (d rows x 64 columns; the contraction runs along the rows as they are
//               stored, so nothing is transposed, and a panel is both operands of its MMA)
//   warp 2      MMA issuer of the tiles:  D[position][c] = sum over k of v[k] B[c][k], B = hi + mid + lo
//   warp 3      MMA issuer of the Gram matrix of the NEXT item
//   warps 4-11  epilogue in two quads: a position per thread, q = sum over c of D[c] v[c], norm = sqrt(q)
//   warps 12-19 Gram sums: every 64 (d = 64: 32) projection columns the accumulator is added to fp32 sums in registers; at
//               the end B
// Precision.  Products of bf16 are exact; the tensor core, whose sums err towards zero, adds four (two) instructions' worth
// before they continue in round-to-nearest fp32 registers.  The matrix enters the second contraction as three bf16 pieces
// (24 bits).  It is symmetric, so only blocks of 16 channels on and above the diagonal are multiplied, those above it doubled.
// Cancellation.  With y_b the projection of a position's first b blocks of 16 channels, q = |y_last|^2, and the terms D[c] v[c]
// of block b add up to |y_b|^2 - |y_b-1|^2.  q is taken where t, the sum of the blocks' sums without their signs, and s, the sum of
// G[c][c] v[c]^2, are both at most 1.5 q.  t >= 2 max |y_b|^2 - q, so that |y_b|^2 <= 1.25 q and no partial sum of D[c] is beyond
// 2.3 |w_c| sqrt(q).  With e a few 2^-24: an entry of G is wrong by e |w_c| |w_k|, which moves q by at most e d s, and by about e s
// as the errors have either sign; a step of D is wrong by e |w_c| sqrt(q), which moves q by at most e sqrt(d s q).  Other
// positions, and those whose squares leave fp32 or its normal range, are left to the direct kernel, a bit each.  Without the
// rule a projection with a common component in its rows, and values that cancel it, loses 1e-7 to 3e-5 of the norm, and
// t and s are 1.5 to 1100 q there (multiplied out: 0.5e-7 to 1.2e-7).
// Against 64 bits (normal values, projections of 520 to 4096 columns) the norms' error is 0.75e-7 to 0.87e-7 rms here and
// 1.15e-7 multiplied out (d = 64: 0.66e-7 to 0.73e-7 and 0.76e-7); with twice the columns between the fp32 additions it would
// be 1.28e-7.  Where rows share components, single rows are a hundred times the others or singular values fall as k^-1/4 to k^-2,
// what is taken is as good as multiplied out (0.75e-7 to 1.1e-7).  With a limit of 3 instead of 1.5 the first of these would lose
// half as much again.
// What bounds it: shared-memory bandwidth (an MMA reads both operands there: 24 steps per tile, 256 per projection slice)
// beside the 1.07 GB of projections at 256 heads x 4 query heads x 4096 columns.  There, with 3968 positions a head: 0.38 ms
// against 2.81 ms multiplied out, 0.37 without t and s, and 0.44 where rows differ in length (s added up for every
// position: 0.43 if it were so for all); 0.26 ms with one tile per slice, 0.28 ms with 512 columns.  A single epilogue quad
// 0.39 ms and blocks below the diagonal multiplied too 0.43 ms (both without t and s).
// Every wait is bounded; the waits are between the warps of one CTA only.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "tc_ptx.cuh"

namespace lukv {
namespace {

constexpr int kGmThreads = 640;
constexpr int kGmGramWarps = 8;
constexpr float kGmMost = 1.5f;  // most (sum of a position's terms without their signs) / q that is taken

template <int NH>  // halves of 64 channels: d = 64 NH
struct GmPlan {
  static constexpr int kD = 64 * NH;
  static constexpr int kVTile = NH * kHalfBytes;     // 128 positions
  static constexpr int kVStages = 3;
  static constexpr int kWStage = kD * 128;           // d rows x 64 columns
  static constexpr int kWStages = NH == 2 ? 3 : 10;
  static constexpr int kGBufs = 4 / NH;               // Gram accumulators of d columns
  static constexpr int kStepK = 2 * NH;              // MMAs of 16 columns between two additions to the fp32 sums
  // one piece: 64 channels x d columns of D, then (d = 128) the other 64 channels x columns 64-127, the only ones that
  // they reach
  static constexpr int kBHalf = kD * 128;
  static constexpr int kPiece = kBHalf + (NH - 1) * 64 * 128;
  static constexpr int kVOff = 3 * kPiece;
  static constexpr int kWOff = kVOff + kVStages * kVTile;
  // the MMA reads 128 rows from a panel of 64 (d = 64; rows beyond d make accumulator rows that nothing reads)
  static constexpr int kTotal = kWOff + kWStages * kWStage + (NH == 1 ? kWStage : 0) + 1024;
};
enum {
  kGmVFull = 0, kGmVEmpty = 3, kGmWFull = 6, kGmWEmpty = 16, kGmDFull = 26, kGmDEmpty = 28, kGmGFull = 30, kGmGEmpty = 34,
  kGmBFull = 38, kGmBEmpty = 42, kGmBars = 43
};

struct GmArgs {
  float* vnorm;          // [heads][G][n]
  uint32_t* left;        // [heads][G][tiles][4] a bit per position that is left to the direct kernel
  int S, LH, G, T, n, Dm;
  int tiles;             // 128-position tiles per head
  int per_item;          // tiles per item (of the S * tiles that a slice has)
  int items_per_slice;
  int items;
  uint32_t spin_limit;
  int drop_item;         // test hook: the value tiles of this item are never loaded (-1: none)
  int32_t* status;
};

template <int NH>
__global__ void __launch_bounds__(kGmThreads, 1)
    value_norm_gram_kernel(const __grid_constant__ CUtensorMap v_map, const __grid_constant__ CUtensorMap w_map,
                           const GmArgs a) {
  using P = GmPlan<NH>;
  static_assert(P::kTotal <= 232448 - 512, "exceeds the shared memory of one CTA");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* v_tiles = smem + P::kVOff;
  __shared__ __align__(8) uint64_t bars[kGmBars];
  __shared__ __align__(16) float diag_s[4][128];  // the diagonal of G, for the last items
  __shared__ float gmax_s[4][kGmGramWarps];       // its largest entry, per warp
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto bar = [&](int kind, int i) { return smem_u32(&bars[kind + i]); };
  auto wait = [&](uint32_t b, uint32_t parity) { return mbar_wait(b, parity, abort_flag, a.status, a.spin_limit); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < P::kVStages; ++i) {
      mbar_init(bar(kGmVFull, i), 1);
      mbar_init(bar(kGmVEmpty, i), 4);  // the epilogue has read the tile, which it does after the MMAs
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(kGmDFull, i), 1);
      mbar_init(bar(kGmDEmpty, i), 4);
    }
    for (int i = 0; i < P::kGBufs; ++i) {
      mbar_init(bar(kGmGFull, i), 1);
      mbar_init(bar(kGmGEmpty, i), kGmGramWarps);
    }
    for (int i = 0; i < P::kWStages; ++i) {
      mbar_init(bar(kGmWFull, i), 1);
      mbar_init(bar(kGmWEmpty, i), 1);
    }
    for (int i = 0; i < 4; ++i) mbar_init(bar(kGmBFull, i), kGmGramWarps);
    mbar_init(bar(kGmBEmpty, 0), 1);
    abort_s = 0;
    // the first kernel of the call clears the word; a wait runs out milliseconds after this, at the earliest
    if (blockIdx.x == 0) atomicExch(a.status, 0);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) tmem_alloc(smem_u32(&tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;           // columns 0-255: D, two buffers; 256-511: Gram accumulators
  const int panels = (a.Dm + 63) / 64;            // of 64 projection columns
  const int steps = panels * (4 / P::kStepK);
  const int all_tiles = a.S * a.tiles;

  if (warp == 0) {
    // ---------------- TMA producer: value tiles ----------------
    if (lane == 0) {
      uint32_t s = 0, ph = 1;
      bool ok = true;
      for (int idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x) {
        const int slice = idx / a.items_per_slice, t0 = (idx % a.items_per_slice) * a.per_item;
        const int t1 = min(t0 + a.per_item, all_tiles);
        if (idx == a.drop_item) break;
        for (int t = t0; t < t1; ++t) {
          if (!(ok = wait(bar(kGmVEmpty, s), ph))) break;
          mbar_expect_tx(bar(kGmVFull, s), P::kVTile);
          const int seq = t / a.tiles, row = (seq * a.LH + slice / a.G) * a.T + (t - seq * a.tiles) * 128;
          for (int h = 0; h < NH; ++h)  // rows past the head's positions are never written back
            tma_load_2d(smem_u32(v_tiles) + s * P::kVTile + h * kHalfBytes, &v_map, bar(kGmVFull, s), h * 64, row);
          if (++s == P::kVStages) s = 0, ph ^= 1;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- TMA producer: projection panels ----------------
    if (lane == 0) {
      const uint64_t once = l2_policy_evict_first();
      uint32_t s = 0, ph = 1;
      bool ok = true;
      for (int idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x) {
        const int row = idx / a.items_per_slice * P::kD;
        for (int p = 0; p < panels; ++p) {
          if (!(ok = wait(bar(kGmWEmpty, s), ph))) break;
          mbar_expect_tx(bar(kGmWFull, s), P::kWStage);
          tma_load_2d_hint(smem_u32(smem) + P::kWOff + s * P::kWStage, &w_map, bar(kGmWFull, s), p * 64, row, once);
          if (++s == P::kWStages) s = 0, ph ^= 1;
        }
      }
    }
  } else if (warp == 2) {
    // ---------------- MMA issuer: tiles ----------------
    if (lane == 0) {
      uint32_t tt = 0, it = 0, vs = 0, vph = 0;
      bool ok = true;
      for (int idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x, ++it) {
        const int t0 = (idx % a.items_per_slice) * a.per_item, t1 = min(t0 + a.per_item, all_tiles);
        if (!(ok = wait(bar(kGmBFull, it & 3), (it >> 2) & 1))) break;
        for (int t = t0; t < t1; ++t, ++tt) {
          const uint32_t s = tt & 1, ph = (tt >> 1) & 1;
          if (!(ok = wait(bar(kGmDEmpty, s), ph ^ 1))) break;
          if (!(ok = wait(bar(kGmVFull, vs), vph))) break;
          tc_fence_after();
          const uint32_t vt = smem_u32(v_tiles) + vs * P::kVTile;
          if (++vs == P::kVStages) vs = 0, vph ^= 1;
#pragma unroll
          for (int piece = 2; piece >= 0; --piece) {  // the smallest first
            const uint32_t bp = smem_u32(smem) + piece * P::kPiece;
#pragma unroll
            for (int ks = 0; ks < 4 * NH; ++ks) {
              // channels 16 ks .. + 15 into the columns from 16 ks on
              const uint64_t da = smem_desc_sw128(vt + (ks >> 2) * kHalfBytes) + (uint64_t)((ks & 3) * 2);
              const uint64_t db = smem_desc_sw128(bp + (ks >> 2) * P::kBHalf + (16 * ks - 64 * (ks >> 2)) * 128) + (uint64_t)((ks & 3) * 2);
              umma_bf16(tmem_base + s * 128 + 16 * ks, da, db, instr_desc_bf16(128, P::kD - 16 * ks), piece < 2 || ks > 0);
            }
          }
          umma_commit(bar(kGmDFull, s));
        }
        if (ok) umma_commit(bar(kGmBEmpty, 0));  // the pieces may be overwritten
      }
    }
  } else if (warp == 3) {
    // ---------------- MMA issuer: Gram matrices ----------------
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc_bf16(128, P::kD);
      uint32_t gc = 0, s = 0, ph = 0;
      bool ok = true;
      for (int idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x)
        for (int p = 0; p < panels && ok; ++p) {
          if (!(ok = wait(bar(kGmWFull, s), ph))) break;
          const uint32_t wt = smem_u32(smem) + P::kWOff + s * P::kWStage;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint32_t b = gc % P::kGBufs;
            if (ks % P::kStepK == 0) {
              if (!(ok = wait(bar(kGmGEmpty, b), ((gc / P::kGBufs) & 1) ^ 1))) break;
              tc_fence_after();
            }
            const uint64_t dw = smem_desc_sw128(wt) + (uint64_t)(ks * 2);
            umma_bf16(tmem_base + 256 + b * P::kD, dw, dw, idesc, ks % P::kStepK > 0);
            if (ks % P::kStepK == P::kStepK - 1) {
              umma_commit(bar(kGmGFull, b));
              ++gc;
            }
          }
          if (ok) umma_commit(bar(kGmWEmpty, s));
          if (++s == P::kWStages) s = 0, ph ^= 1;
        }
    }
  } else if (warp < 12) {
    // ---------------- epilogue: a position per thread ----------------
    // two quads of warps take alternate tiles: a quad alone is slower than the MMAs
    const int quad = warp & 3, parity = (warp - 4) >> 2, row = 32 * quad + lane;
    const uint32_t lane_addr = (uint32_t)(32 * quad) << 16;
    uint32_t tt = 0, it = 0, vs = 0, vph = 0, seen = ~0u;  // seen: the last item whose diagonal was waited for
    bool ok = true;
    for (int idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x, ++it) {
      const int slice = idx / a.items_per_slice, t0 = (idx % a.items_per_slice) * a.per_item;
      const int t1 = min(t0 + a.per_item, all_tiles);
      const int uh = slice / a.G, g = slice - uh * a.G;
      bool uneven = false;  // the projection's rows differ in length (as far as this warp has seen)
      for (int t = t0; t < t1; ++t, ++tt) {
        const uint32_t stage = vs, stage_ph = vph;
        if (++vs == P::kVStages) vs = 0, vph ^= 1;
        if ((int)(tt & 1) != parity) continue;
        const uint32_t s = tt & 1, ph = (tt >> 1) & 1;
        // The accumulator, and what ordinary loads below read beside it: the tile of values (by its copy) and the diagonal
        // (published by the Gram warps).  The MMAs waited for both, but their completion orders only the accumulator for
        // this thread.  None of the three barriers can be a phase ahead: this tile's buffers are still to be given back.
        if (!(ok = (seen == it || wait(bar(kGmBFull, it & 3), (it >> 2) & 1)) && wait(bar(kGmDFull, s), ph))) break;
        seen = it;
        tc_fence_after();
        // a slot is written again four items on, when this tile's buffer has long been given back
        float gmax = 0.f;
#pragma unroll
        for (int i = 0; i < kGmGramWarps; ++i) gmax = fmaxf(gmax, gmax_s[it & 3][i]);
        const unsigned char* vrow = v_tiles + stage * P::kVTile + row * 128;
        auto value8 = [&](int c8) {  // channels 8 c8 .. + 7
          return *reinterpret_cast<const uint4*>(vrow + (c8 >> 3) * kHalfBytes + (((c8 & 7) ^ (row & 7)) << 4));
        };
        auto pair_of = [](uint32_t w) { return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); };
        const float* diag = diag_s[it & 3];
        float q = 0.f, terms = 0.f;
        uint64_t vv2[2] = {0, 0}, own2[2] = {0, 0};
        float d[32];
        tmem_ld32(tmem_base + lane_addr + s * 128, d);
        ok = wait(bar(kGmVFull, stage), stage_ph);  // (behind the load: the test is a round trip to shared memory)
        if (!ok) {
          tmem_ld_wait(d);
          break;
        }
        auto add_up = [&](auto with_own) {
#pragma unroll
          for (int c0 = 0; c0 < 2 * NH; ++c0) {
            if (c0 > 0) tmem_ld32(tmem_base + lane_addr + s * 128 + 32 * c0, d);
            uint4 v[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = value8(4 * c0 + c);
            tmem_ld_wait(d);
#pragma unroll
            for (int b = 0; b < 2; ++b) {  // a block of 16 channels
              uint64_t sum = 0;
#pragma unroll
              for (int c = 2 * b; c < 2 * b + 2; ++c) {
                const uint32_t w4[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const uint64_t x = pair_of(w4[i]);
                  sum = ffma2(pack2(d[8 * c + 2 * i], d[8 * c + 2 * i + 1]), x, sum);
                  vv2[b] = ffma2(x, x, vv2[b]);
                  if constexpr (decltype(with_own)::value) {
                    const uint64_t g = *reinterpret_cast<const uint64_t*>(diag + 32 * c0 + 8 * c + 2 * i);
                    own2[b] = ffma2(fmul2(g, x), x, own2[b]);
                  }
                }
              }
              float even, odd;
              unpack2(sum, even, odd);
              q += even + odd, terms += fabsf(even + odd);
            }
          }
        };
        const bool with_own = uneven;
        if (with_own) add_up(std::true_type{});
        else add_up(std::false_type{});
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kGmDEmpty, s), 1);
        const float vv = sum4(vv2[0], vv2[1]), most = kGmMost * q;
        bool sound = terms <= most && q >= 1e-30f && q <= 1e37f && vv >= 1e-30f && vv <= 1e30f && q >= 1e-25f * vv;
        // rows of alike length: the longest bounds the sum of G[c][c] v[c]^2; else it is added up, from the next tile on above
        if (!with_own && __any_sync(0xffffffffu, sound && !(gmax * vv <= most))) {
          uneven = true;
#pragma unroll 2
          for (int c = 0; c < 8 * NH; ++c) {
            const uint4 v = value8(c);
            const ulonglong2 g0 = *reinterpret_cast<const ulonglong2*>(diag + 8 * c);
            const ulonglong2 g1 = *reinterpret_cast<const ulonglong2*>(diag + 8 * c + 4);
            const uint64_t x0 = pair_of(v.x), x1 = pair_of(v.y), x2 = pair_of(v.z), x3 = pair_of(v.w);
            own2[0] = ffma2(fmul2(g0.x, x0), x0, own2[0]);
            own2[1] = ffma2(fmul2(g0.y, x1), x1, own2[1]);
            own2[0] = ffma2(fmul2(g1.x, x2), x2, own2[0]);
            own2[1] = ffma2(fmul2(g1.y, x3), x3, own2[1]);
          }
          __syncwarp();
        }
        if (uneven) sound = sound && sum4(own2[0], own2[1]) <= most;
        // a value of zeros has the norm zero (if the projection holds numbers); squares below fp32's range look the same
        if (__any_sync(0xffffffffu, vv == 0.f)) {
          uint32_t any = 0;
#pragma unroll 2
          for (int c = 0; c < 8 * NH; ++c) {
            const uint4 v = value8(c);
            any |= v.x | v.y | v.z | v.w;
          }
          sound = sound || ((any & 0x7FFF7FFFu) == 0 && q == 0.f);
          __syncwarp();
        }
        if (lane == 0) mbar_arrive(bar(kGmVEmpty, stage), 1);
        const int seq = t / a.tiles, tile = t - seq * a.tiles, j = tile * 128 + row;
        const size_t ug = (size_t)(seq * a.LH + uh) * a.G + g;
        if (j < a.n) a.vnorm[ug * a.n + j] = sqrtf(q);
        const uint32_t left = __ballot_sync(0xffffffffu, j < a.n && !sound);
        if (lane == 0) a.left[(ug * a.tiles + tile) * 4 + quad] = left;
      }
    }
  } else {
    // ---------------- Gram sums and pieces ----------------
    const int quad = warp & 3, half = (warp - 12) >> 2;
    const int row = 32 * quad + lane;               // row of G = column of D
    constexpr int kCols = 32 * NH;                  // this warp's columns of G, from kCols * half on
    const uint32_t lane_addr = (uint32_t)(32 * quad) << 16;
    const bool live = 32 * quad < P::kD;
    uint32_t gc = 0, it = 0;
    bool ok = true;
    for (int idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x, ++it) {
      float acc[kCols];
#pragma unroll
      for (int i = 0; i < kCols; ++i) acc[i] = 0.f;
#pragma unroll 1
      for (int step = 0; step < steps; ++step, ++gc) {
        const uint32_t b = gc % P::kGBufs;
        if (!(ok = wait(bar(kGmGFull, b), (gc / P::kGBufs) & 1))) break;
        tc_fence_after();
        if (live) {
          constexpr int kLd = NH == 2 ? 16 : 32;    // columns a load: what the registers have room for
#pragma unroll
          for (int c = 0; c < kCols; c += kLd) {
            float d[kLd];
            const uint32_t at = tmem_base + lane_addr + 256 + b * P::kD + kCols * half + c;
            if constexpr (NH == 2) tmem_ld16(at, d);
            else tmem_ld32(at, d);
            tmem_ld_wait(d);
#pragma unroll
            for (int i = 0; i < kLd; ++i) acc[c + i] += d[i];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kGmGEmpty, b), 1);
      }
      if (!ok) break;
      float own = 0.f;  // G[row][row], where it is one of this thread's columns
      // the tiles of the item before have been multiplied
      if (!(ok = wait(bar(kGmBEmpty, 0), (it & 1) ^ 1))) break;
      if (live) {
#pragma unroll
        for (int c = 0; c < kCols / 8; ++c) {
          const int k0 = kCols * half + 8 * c;      // eight channels of the contraction
          const float f = (k0 >> 4) < (row >> 4) ? 2.f : 1.f;
          uint32_t w[3][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float x = acc[8 * c + 2 * i] * f, y = acc[8 * c + 2 * i + 1] * f;
            if (k0 + 2 * i == row) own = x;  // f is 1 there
            if (k0 + 2 * i + 1 == row) own = y;
#pragma unroll
            for (int piece = 0; piece < 3; ++piece) {
              const __nv_bfloat162 p = __floats2bfloat162_rn(x, y);
              w[piece][i] = *reinterpret_cast<const uint32_t*>(&p);
              x -= __low2float(p);
              y -= __high2float(p);
            }
          }
          if (half && row < 64 && NH == 2) continue;  // not reached
#pragma unroll
          for (int piece = 0; piece < 3; ++piece)
            *reinterpret_cast<uint4*>(smem + piece * P::kPiece + (k0 >> 6) * P::kBHalf + (row - 64 * (k0 >> 6)) * 128 +
                                      ((((k0 >> 3) & 7) ^ (row & 7)) << 4)) =
                make_uint4(w[piece][0], w[piece][1], w[piece][2], w[piece][3]);
        }
      }
      if (live && row / kCols == half) diag_s[it & 3][row] = own;
      own = warp_max(own);
      if (lane == 0) gmax_s[it & 3][warp - 12] = own;
      // the MMA reads shared memory through the asynchronous proxy: order these writes before it
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kGmBFull, it & 3), 1);
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// 2-D bf16 tensor [rows][cols] with boxes of 64 columns x d rows, 128-byte swizzle, zero fill.
bool make_panel_map(CUtensorMap* map, const void* base, uint64_t rows, int cols, int d) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)d};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int gm_tiles(const Dims& dm) { return (dm.n + 127) / 128; }

// Tiles per item and the time that the call would take, by this kernel and by the direct one.
struct GmChoice {
  int per_item;
  double gram_us, direct_us;
};
GmChoice gm_choose(const Dims& dm, int d_model, int sms) {
  const bool wide = dm.d == 128;
  // measured with every SM busy (48 query heads x 3 to 1024 x 31 tiles, 512 to 4096 columns), us: 64 projection columns into
  // the Gram matrix, a tile through it, a tile times 256 columns
  const double panel = wide ? 0.55 : 0.4, tile = wide ? 1.1 : 0.7, direct = wide ? 0.72 : 0.4;
  const long long slices = (long long)dm.N * dm.G, all = (long long)dm.S * gm_tiles(dm);
  const double gram = panel * ((d_model + 63) / 64);
  GmChoice best = {(int)all, 1e30, 0.0};
  for (int c = 1; c <= 16 && c <= all; ++c) {  // more items than that only repeat the Gram matrix
    const long long per = (all + c - 1) / c, rounds = (slices * ((all + per - 1) / per) + sms - 1) / sms;
    const double us = gram + (rounds - 1) * std::max(gram, per * tile) + per * tile;
    if (us < 0.99 * best.gram_us) best.gram_us = us, best.per_item = (int)per;
  }
  best.gram_us += 5.0;  // the direct kernel's look at the flags
  const long long items = dm.heads() * dm.G * ((dm.n + 4095) / 4096);  // of the direct kernel
  best.direct_us = direct * (double)((items + sms - 1) / sms) * std::min(32, gm_tiles(dm)) * ((d_model + 255) / 256);
  return best;
}
}  // namespace

bool value_norm_gram_pays(const Dims& dm, int d_model, const void* w_o) {
  if (!value_norm_tc_supported(dm) || (d_model & 7) || (reinterpret_cast<uintptr_t>(w_o) & 15)) return false;
  if ((int64_t)dm.N * dm.G * dm.d >= ((int64_t)1 << 31) || dm.heads() * dm.G * (int64_t)gm_tiles(dm) >= ((int64_t)1 << 31))
    return false;
  // the bits of the positions that are left lie where the importance will (groups beyond 32, or a few positions: no room)
  if ((int64_t)dm.G * gm_tiles(dm) * 16 > (int64_t)dm.n * 4) return false;
  int sms = 0;
  if (device_sms(&sms) != cudaSuccess) return false;
  // LUKV_VALUE_NORM=gram or direct: that form wherever the shape allows it (for A/B checks; read at every call)
  const char* form = getenv("LUKV_VALUE_NORM");
  if (form && (form[0] == 'g' || form[0] == 'd')) return form[0] == 'g';
  const GmChoice c = gm_choose(dm, d_model, sms);
  return c.gram_us < c.direct_us;
}

cudaError_t launch_value_norm_gram(const Dims& dm, int d_model, const void* v, const void* w_o, float* vnorm,
                                   uint32_t* left, int32_t* status, LaunchCtx& lc) {
  CUtensorMap vm, wm;
  if (!make_map(&vm, v, (uint64_t)dm.heads() * dm.T, dm.d) ||
      !make_panel_map(&wm, w_o, (uint64_t)dm.L * dm.H * dm.G * dm.d, d_model, dm.d))
    return cudaErrorNotSupported;
  GmArgs a;
  a.vnorm = vnorm;
  a.left = left;
  a.S = dm.S, a.LH = dm.N, a.G = dm.G, a.T = dm.T, a.n = dm.n, a.Dm = d_model;
  a.tiles = gm_tiles(dm);
  a.status = status;
  score_test_hooks(&a.spin_limit, &a.drop_item);
  int sms = 0;
  cudaError_t e;
  if ((e = device_sms(&sms)) != cudaSuccess) return e;
  const int slices = dm.N * dm.G, all = dm.S * a.tiles;
  a.per_item = gm_choose(dm, d_model, sms).per_item;
  a.items_per_slice = (all + a.per_item - 1) / a.per_item;
  a.items = slices * a.items_per_slice;
  auto kern = dm.d == 128 ? value_norm_gram_kernel<2> : value_norm_gram_kernel<1>;
  const int smem = dm.d == 128 ? GmPlan<2>::kTotal : GmPlan<1>::kTotal;
  if ((e = allow_smem((const void*)kern, smem)) != cudaSuccess) return e;
  kern<<<std::min(a.items, sms), kGmThreads, smem, lc.st>>>(vm, wm, a);  // one CTA per SM: each owns the SM's tensor memory
  lc.mark("value_norm_gram");
  return cudaGetLastError();
}

}  // namespace lukv
