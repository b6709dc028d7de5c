// Attention part of the oracle importance (Sec. 4.1, Eq. "oracle_importance") on the tensor cores, bf16 inputs:
//   lse[u][g][k]     row log-sum-exp of the query of head g, decode step k over the cached keys and, if decode keys are
//                    given, the keys of steps up to k
//   importance[u][j] max over k of  sum_g 2^(x_{g,k,j} - lse_{g,k}) * vnorm[u][g][j]
// The rows of a query tile are (step, query head) pairs, the head running fastest and padded to GP = 1, 2, 4 or 8 (the
// padding rows are zeros from the tensor map's bounds), so that the 128 rows of a tile are whole steps and the sum over
// the group and the maximum over the steps stay in the thread that owns a key.
//   imp_tc_kernel<LSE>  D[row][key]: a thread owns a query row, as in pass 1 of the tensor-core scorer
//   imp_tc_kernel       D[key][row] (operands swapped): a thread owns a key and runs over the rows
// Both are persistent with static items (equal shares of the key tiles for the second) and warp roles: warps 0-7 two epilogue quads that take alternate key tiles out of
// four accumulator buffers, warp 8 TMA producer, warp 9 tensor memory and MMA issue.  Every wait is bounded and between the
// warps of one CTA only; should one run out, here or in the value norms, what depends on it becomes NaN.
// Bound by the exp2 of the epilogue (2 x 2.6e8 for 256 heads x 256 rows x 4000 keys).  Measured there: 1.90 + 1.82 ms
// on the FP32 pipes, 0.106 + 0.112 ms here.
#define LUKV_POLY_SEL1(i) false  // every exp2 on the special-function unit: the values keep their precision
#include <algorithm>

#include "score_chunks.cuh"

namespace lukv {
namespace {

constexpr int kItEpiThreads = 256;
constexpr int kItThreads = kItEpiThreads + 64;

template <int NH, bool LSE>  // halves of 64 channels: d = 64 NH
struct ItPlan {
  static constexpr int kTile = NH * kHalfBytes;  // one tile of 128 rows
  static constexpr int kQPer = LSE ? 1 : 2;      // query tiles per item
  static constexpr int kQSlots = LSE ? 2 : 1;    // items whose query tiles are held
  static constexpr int kStages = 4;              // key tiles in flight
  static constexpr int kKOff = kQSlots * kQPer * kTile;
  static constexpr int kNlseOff = kKOff + kStages * kTile;     // [2][256] floats
  static constexpr int kMergeOff = kNlseOff + 2 * 256 * 4;       // [128] (reference, sum) of the second quad
  static constexpr int kTotal = kMergeOff + 128 * 8 + 1024;
};
enum { kItKFull = 0, kItKEmpty = 4, kItQFull = 8, kItQEmpty = 10, kItTFull = 12, kItTEmpty = 16, kItBars = 20 };

struct ItArgs {
  float* part;        // [heads][chunks][splits][128] log-sum-exp (exp2 domain) of a split's keys
  const float* vnorm; // [heads][G][n]
  float* importance;  // [heads][n]
  int T, n, G, Kmax, gp_log2;
  int chunks;         // query tiles per head
  int chunk0, nchunk; // imp: the query tiles of this launch (at most two)
  int accumulate;     // imp: the maximum goes on from what `importance` holds
  int splits, tiles_per_split, tiles_T, tiles_D;  // lse: tiles_D tiles of decode keys follow the cached ones
  int items;          // lse: items; imp: key tiles of all heads
  float scale_log2;
  uint32_t spin_limit;
  int drop_item;      // test hook: the query tiles of this item are never loaded (-1: none)
  int32_t* status;    // where a wait that ran out is reported
};

// Both kernels (LSE: the row log-sum-exps): one item is a head, its query tiles (one, or up to two) and a run of key tiles.
template <int NH, bool LSE, int GPL>  // GPL: log2 of GP (the form without LSE)
__global__ void __launch_bounds__(kItThreads, 1)
    imp_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                  const __grid_constant__ CUtensorMap kd_map, const ItArgs a) {
  using P = ItPlan<NH, LSE>;
  constexpr int kItStages = P::kStages;
  static_assert(P::kTotal <= 232448, "exceeds the shared memory of one CTA");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  float* nlse_s = reinterpret_cast<float*>(smem + P::kNlseOff);
  float2* merge_s = reinterpret_cast<float2*>(smem + P::kMergeOff);
  __shared__ __align__(8) uint64_t bars[kItBars];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto bar = [&](int kind, int i) { return smem_u32(&bars[kind + i]); };
  auto wait = [&](uint32_t b, uint32_t parity) { return mbar_wait(b, parity, abort_flag, a.status, a.spin_limit); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < kItStages; ++i) {
      mbar_init(bar(kItKFull, i), 1);
      mbar_init(bar(kItKEmpty, i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(kItQFull, i), 1);
      mbar_init(bar(kItQEmpty, i), 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(bar(kItTFull, i), 1);
      mbar_init(bar(kItTEmpty, i), 4);
    }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) tmem_alloc(smem_u32(&tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  // a wait of the kernels before, or of this one, ran out: their values are not to be used
  const bool spoiled = !LSE && *reinterpret_cast<volatile int32_t*>(a.status) != 0;

  // an item: head u, query tiles [c0, c0 + nq), key tiles [t0, t0 + nt)
  struct Item {
    int u, c0, nq, split, t0, nt;
  };
  // The items of this CTA in order: for the log-sum-exps every gridDim-th of all; for the importance its share of the key tiles of
  // all heads, cut where a head ends.  (Eight items per SM of a few tiles of one head each spent as long on the start of an item,
  // its row log-sum-exps and value norms, as on its tiles: 256 heads x 31 tiles x 2 query tiles 154 us, 112 so.)
  struct Walk {
    int idx, pos, end;
  };
  auto walk = [&]() {
    const long long all = a.items;
    return Walk{(int)blockIdx.x, (int)(all * blockIdx.x / gridDim.x), (int)(all * (blockIdx.x + 1) / gridDim.x)};
  };
  auto next = [&](Walk& w, Item& it) -> bool {
    if (LSE) {
      if (w.idx >= a.items) return false;
      it.split = w.idx % a.splits;
      const int uc = w.idx / a.splits;
      it.c0 = uc % a.chunks;
      it.u = uc / a.chunks;
      it.nq = 1;
      it.t0 = it.split * a.tiles_per_split;
      it.nt = max(0, min(a.tiles_per_split, a.tiles_T + a.tiles_D - it.t0));
    } else {
      if (w.pos >= w.end) return false;
      it.u = w.pos / a.tiles_T;
      it.split = 0;
      it.c0 = a.chunk0;
      it.nq = a.nchunk;
      it.t0 = w.pos - it.u * a.tiles_T;
      it.nt = min(a.tiles_T - it.t0, w.end - w.pos);
      w.pos += it.nt;
    }
    w.idx += gridDim.x;
    return true;
  };
  const int gp_log2 = LSE ? a.gp_log2 : GPL;
  const int steps_log2 = 7 - gp_log2;  // a query tile holds 128 / GP steps

  if (warp == 8) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      uint32_t tt = 0, jq = 0;
      bool ok = true;
      Walk w = walk();
      Item it;
      while (ok && next(w, it)) {
        const uint32_t slot = jq % P::kQSlots;
        // with one slot the query tiles follow the first key tiles, which need not wait for the item before to end
        const int q_after = P::kQSlots == 1 ? min(kItStages, it.nt) : 0;
        auto load_q = [&]() -> bool {
          if (!wait(bar(kItQEmpty, slot), ((jq / P::kQSlots) & 1) ^ 1)) return false;
          mbar_expect_tx(bar(kItQFull, slot), it.nq * P::kTile);
          for (int c = 0; c < it.nq && w.idx - (int)gridDim.x != a.drop_item; ++c)
            for (int h = 0; h < NH; ++h) {
              const uint32_t dst = smem_u32(smem) + (P::kQPer * slot + c) * P::kTile + h * kHalfBytes;
              asm volatile(
                  "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                  ::"r"(dst), "l"(&q_map), "r"(bar(kItQFull, slot)), "r"(h * 64), "r"(0), "r"((it.c0 + c) << steps_log2),
                  "r"(it.u)
                  : "memory");
            }
          ++jq;
          return true;
        };
        if (q_after == 0 && !(ok = load_q())) break;
        for (int t = 0; t < it.nt; ++t, ++tt) {
          const uint32_t s = tt % kItStages, ph = (tt / kItStages) & 1;
          if (!(ok = wait(bar(kItKEmpty, s), ph ^ 1))) break;
          mbar_expect_tx(bar(kItKFull, s), P::kTile);
          const uint32_t dst = smem_u32(smem) + P::kKOff + s * P::kTile;
          const int tile = it.t0 + t;
          for (int h = 0; h < NH; ++h) {  // rows past the head are masked or never stored
            if (!LSE || tile < a.tiles_T) tma_load_2d(dst + h * kHalfBytes, &k_map, bar(kItKFull, s), h * 64, it.u * a.T + tile * 128);
            else tma_load_2d(dst + h * kHalfBytes, &kd_map, bar(kItKFull, s), h * 64, it.u * a.Kmax + (tile - a.tiles_T) * 128);
          }
          if (t + 1 == q_after && !(ok = load_q())) break;
        }
      }
    }
  } else if (warp == 9) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc_bf16(128, 128);
      uint32_t tt = 0, jq = 0, used[2] = {0, 0};
      bool ok = true;
      Walk w = walk();
      Item it;
      for (; ok && next(w, it); ++jq) {
        const uint32_t slot = jq % P::kQSlots;
        if (!(ok = wait(bar(kItQFull, slot), (jq / P::kQSlots) & 1))) break;
        for (int t = 0; t < it.nt && ok; ++t, ++tt) {
          const uint32_t s = tt % kItStages, quad = tt & 1;
          if (!(ok = wait(bar(kItKFull, s), (tt / kItStages) & 1))) break;
          const uint32_t kt = smem_u32(smem) + P::kKOff + s * P::kTile;
          for (int c = 0; c < it.nq; ++c) {
            const uint32_t n_use = used[quad]++, buf = 2 * quad + (n_use & 1);  // a quad's buffers in turn
            if (!(ok = wait(bar(kItTEmpty, buf), ((n_use >> 1) & 1) ^ 1))) break;
            tc_fence_after();
            const uint32_t qd = smem_u32(smem) + (P::kQPer * slot + c) * P::kTile;
#pragma unroll
            for (int ks = 0; ks < 4 * NH; ++ks) {
              const uint64_t dq = smem_desc_sw128(qd + (ks >> 2) * kHalfBytes) + (uint64_t)((ks & 3) * 2);
              const uint64_t dk = smem_desc_sw128(kt + (ks >> 2) * kHalfBytes) + (uint64_t)((ks & 3) * 2);
              umma_bf16(tmem_base + buf * 128, LSE ? dq : dk, LSE ? dk : dq, idesc, ks > 0);
            }
            umma_commit(bar(kItTFull, buf));
          }
          if (ok) umma_commit(bar(kItKEmpty, s));
        }
        if (ok) umma_commit(bar(kItQEmpty, slot));
      }
    }
  } else {
    // ---------------- epilogue quads ----------------
    const int quad = warp >> 2, qtid = threadIdx.x & 127;
    const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
    uint32_t tt = 0, n_use = 0, jq = 0;
    bool ok = true;
    Walk w = walk();
    Item it;
    for (; next(w, it); ++jq) {
      if (LSE) {
        const int step = (it.c0 << steps_log2) + (qtid >> gp_log2);
        const bool row_ok = step < a.Kmax && (qtid & ((1 << gp_log2) - 1)) < a.G;
        const uint64_t sc2 = pack2(a.scale_log2, a.scale_log2);
        float m = -INFINITY, l = 0.f;
        for (int t = 0; t < it.nt; ++t, ++tt) {
          if ((int)(tt & 1) != quad) continue;
          const uint32_t buf = 2 * quad + (n_use & 1);
          ok = ok && wait(bar(kItTFull, buf), (n_use >> 1) & 1);
          ++n_use;
          if (!ok) continue;
          tc_fence_after();
          const int tile = it.t0 + t;
          const bool decode = tile >= a.tiles_T;
          const int j0 = (decode ? tile - a.tiles_T : tile) * 128;
          const int lim = !row_ok ? -1 : decode ? step : a.T - 1;  // last visible key
          const bool masked = decode || j0 + 128 > a.T;
          const uint32_t tcol = tmem_base + lane_addr + buf * 128;
          // a tile in one stretch where all its keys are visible, chunk by chunk where not, as in the scorer's pass 1
          float va[32], vb[32];
          bool redo = true;
          if (!masked) {
            uint64_t acc0 = 0ull, acc1 = 0ull;
            float pmax = -INFINITY;  // (no argument goes through the polynomial here)
            tmem_ld32(tcol, va);
            tmem_ld_wait(va);
            tmem_ld32(tcol + 32, vb);
            if (m == -INFINITY) m = p1_reference(va, a.scale_log2);
            const uint64_t nm2 = pack2(-m, -m);
            p1_terms(va, sc2, nm2, acc0, acc1, pmax);
            tmem_ld_wait(vb);
            tmem_ld32(tcol + 64, va);
            p1_terms(vb, sc2, nm2, acc0, acc1, pmax);
            tmem_ld_wait(va);
            tmem_ld32(tcol + 96, vb);
            p1_terms(va, sc2, nm2, acc0, acc1, pmax);
            tmem_ld_wait(vb);
            p1_terms(vb, sc2, nm2, acc0, acc1, pmax);
            const float cs = sum4(acc0, acc1);
            if (cs <= kP1Limit) {
              l += cs;
              redo = false;
            }
          }
          if (__any_sync(0xffffffffu, redo)) {
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              tmem_ld32(tcol + 32 * c, vb);
              tmem_ld_wait(vb);
              if (redo) p1_exact(vb, j0 + 32 * c, lim, a.scale_log2, m, l);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(kItTEmpty, buf), 1);
        }
        // the quads hold partials of the same rows over different tiles
        if (quad == 1) merge_s[qtid] = make_float2(m, l);
        bar_sync(1, kItEpiThreads);
        if (quad == 0) {
          const float2 o = merge_s[qtid];
          const float mn = fmaxf(m, o.x);
          float v = -INFINITY;
          if (row_ok && mn > -INFINITY) v = p1_log(mn, (l > 0.f ? l * ex2(m - mn) : 0.f) + (o.y > 0.f ? o.y * ex2(o.x - mn) : 0.f));
          a.part[(((size_t)it.u * a.chunks + it.c0) * a.splits + it.split) * 128 + qtid] = v;
        }
        bar_sync(1, kItEpiThreads);
      } else {
        // -lse of the item's rows; rows without a query get -inf and add nothing
        float* nlse = nlse_s + (jq & 1) * 256;
        {
          const int c = threadIdx.x >> 7;
          float v = -INFINITY;
          if (c < it.nq) {
            const float* p = a.part + ((size_t)it.u * a.chunks + it.c0 + c) * a.splits * 128 + qtid;
            float m = -INFINITY, l = 0.f;
            for (int s = 0; s < a.splits; ++s) m = fmaxf(m, __ldg(p + (size_t)s * 128));
            for (int s = 0; s < a.splits; ++s) l += ex2(__ldg(p + (size_t)s * 128) - m);
            const int step = ((it.c0 + c) << steps_log2) + (qtid >> gp_log2);
            if (step < a.Kmax && (qtid & ((1 << gp_log2) - 1)) < a.G) v = -(m + (a.splits > 1 ? log2f(l) : 0.f));
          }
          nlse[threadIdx.x] = v;
        }
        bar_sync(1, kItEpiThreads);
        const uint64_t sc2 = pack2(a.scale_log2, a.scale_log2);
        // value norms of this thread's key: those of the quad's next tile are on their way during a tile
        constexpr int GP = 1 << GPL;
        float vg[GP], vg_next[GP];
        auto fetch_norms = [&](int t) {
          const int j = (it.t0 + t) * 128 + qtid;
#pragma unroll
          for (int g = 0; g < GP; ++g)
            vg_next[g] = g < a.G && t < it.nt && j < a.n ? __ldg(a.vnorm + ((size_t)it.u * a.G + g) * a.n + j) : 0.f;
        };
        fetch_norms((int)(tt & 1) == quad ? 0 : 1);
        for (int t = 0; t < it.nt; ++t, ++tt) {
          if ((int)(tt & 1) != quad) continue;
          const int j = (it.t0 + t) * 128 + qtid;
#pragma unroll
          for (int g = 0; g < GP; ++g) vg[g] = vg_next[g];
          fetch_norms(t + 2);
          float best = a.accumulate && j < a.n ? a.importance[(size_t)it.u * a.n + j] : 0.f;  // importance is not negative
          for (int c = 0; c < it.nq; ++c) {
            const uint32_t buf = 2 * quad + (n_use & 1);
            ok = ok && wait(bar(kItTFull, buf), (n_use >> 1) & 1);
            ++n_use;
            if (!ok) continue;
            tc_fence_after();
            const uint32_t tcol = tmem_base + lane_addr + buf * 128;
            const float* nl = nlse + 128 * c;
            // 32 rows: whole steps
            auto rows = [&](const float (&v)[32], const float* nlc) {
              float e[32];
#pragma unroll
              for (int i = 0; i < 32; i += 4) {
                const ulonglong2 ls = *reinterpret_cast<const ulonglong2*>(nlc + i);
                unpack2(ex2_pair(ffma2(pack2(v[i], v[i + 1]), sc2, ls.x)), e[i], e[i + 1]);
                unpack2(ex2_pair(ffma2(pack2(v[i + 2], v[i + 3]), sc2, ls.y)), e[i + 2], e[i + 3]);
              }
#pragma unroll
              for (int i = 0; i < 32; i += 1 << GPL) {
                float s = e[i] * vg[0];
#pragma unroll
                for (int g = 1; g < 1 << GPL; ++g) s = fmaf(e[i + g], vg[g], s);
                best = fmaxf(best, s);
              }
            };
            float va[32], vb[32];
            tmem_ld32(tcol, va);
#pragma unroll 1  // (unrolled: spills, 119 against 112 us)
            for (int i = 0; i < 4; i += 2) {
              tmem_ld_wait(va);
              tmem_ld32(tcol + 32 * (i + 1), vb);
              rows(va, nl + 32 * i);
              tmem_ld_wait(vb);
              if (i + 2 < 4) tmem_ld32(tcol + 32 * (i + 2), va);
              rows(vb, nl + 32 * (i + 1));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kItTEmpty, buf), 1);
          }
          if (j < a.n) a.importance[(size_t)it.u * a.n + j] = ok && !spoiled ? best : __int_as_float(0x7FC00000);
        }
      }
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

int log2_ceil(int x) {
  int b = 0;
  while ((1 << b) < x) ++b;
  return b;
}
int imp_chunks(const Dims& dm, int k_max) {
  const int steps = 128 >> log2_ceil(dm.G);
  return (k_max + steps - 1) / steps;
}
// Splits of the keys in the log-sum-exp pass: enough items for the SMs, at least four key tiles each.
int imp_splits(const Dims& dm, int k_max) {
  const long long tiles = (dm.T + 127) / 128 + (k_max + 127) / 128;
  const long long items = dm.heads() * imp_chunks(dm, k_max);
  return (int)std::max(1LL, std::min((6 * 148 + items - 1) / items, tiles / 4));
}

// Query rows as [heads][steps][G][d] in the order the kernels want; boxes of 64 channels x GP heads x 128/GP steps.
bool make_query_map(CUtensorMap* map, const void* base, int d, int G, int k_max, uint64_t heads, int gp) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t row = (cuuint64_t)d * 2;
  const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)G, (cuuint64_t)k_max, heads};
  const cuuint64_t strides[3] = {row * k_max, row, row * k_max * G};
  const cuuint32_t box[4] = {64, (cuuint32_t)gp, (cuuint32_t)(128 / gp), 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int NH>
cudaError_t launch_importance_tc_t(const Dims& dm, int k_max, const void* q_dec, const void* k, const void* k_dec,
                                   const float* vnorm, float* part, float* importance, int32_t* status, LaunchCtx& lc) {
  const int gp_log2 = log2_ceil(dm.G), gp = 1 << gp_log2;
  CUtensorMap qm, km, kdm;
  if (!make_query_map(&qm, q_dec, dm.d, dm.G, k_max, (uint64_t)dm.heads(), gp) ||
      !make_map(&km, k, (uint64_t)dm.heads() * dm.T, dm.d) ||
      !make_map(&kdm, k_dec ? k_dec : k, (uint64_t)dm.heads() * (k_dec ? k_max : dm.T), dm.d))
    return cudaErrorNotSupported;
  ItArgs a = {};
  a.part = part;
  a.vnorm = vnorm;
  a.importance = importance;
  a.T = dm.T, a.n = dm.n, a.G = dm.G, a.Kmax = k_max, a.gp_log2 = gp_log2;
  a.chunks = imp_chunks(dm, k_max);
  a.splits = imp_splits(dm, k_max);
  a.scale_log2 = dm.scale_log2;
  a.status = status;
  score_test_hooks(&a.spin_limit, &a.drop_item);
  int sms = 0;
  cudaError_t e;
  if ((e = device_sms(&sms)) != cudaSuccess) return e;
  auto lse = imp_tc_kernel<NH, true, 0>;
  auto imp = gp_log2 == 0 ? imp_tc_kernel<NH, false, 0> : gp_log2 == 1 ? imp_tc_kernel<NH, false, 1>
             : gp_log2 == 2 ? imp_tc_kernel<NH, false, 2> : imp_tc_kernel<NH, false, 3>;
  constexpr int lse_smem = ItPlan<NH, true>::kTotal, imp_smem = ItPlan<NH, false>::kTotal;
  if ((e = allow_smem((const void*)lse, lse_smem)) != cudaSuccess) return e;
  if ((e = allow_smem((const void*)imp, imp_smem)) != cudaSuccess) return e;
  a.tiles_T = (dm.T + 127) / 128;
  a.tiles_D = k_dec ? (k_max + 127) / 128 : 0;
  a.tiles_per_split = (a.tiles_T + a.tiles_D + a.splits - 1) / a.splits;
  a.items = (int)dm.heads() * a.chunks * a.splits;
  lse<<<std::min(a.items, sms), kItThreads, lse_smem, lc.st>>>(qm, km, kdm, a);
  lc.mark("imp_lse_tc");
  a.tiles_T = (dm.n + 127) / 128;
  a.items = (int)dm.heads() * a.tiles_T;
  for (a.chunk0 = 0; a.chunk0 < a.chunks; a.chunk0 += 2) {
    a.nchunk = std::min(2, a.chunks - a.chunk0);
    a.accumulate = a.chunk0 > 0;
    imp<<<std::min(a.items, sms), kItThreads, imp_smem, lc.st>>>(qm, km, kdm, a);
    lc.mark("importance_tc");
  }
  return cudaGetLastError();
}

}  // namespace

bool importance_tc_supported(const Dims& dm, int k_max) {
  return dm.dtype == LUKV_DTYPE_BF16 && dm.G <= 8 && encode_fn() != nullptr &&
         dm.heads() * (int64_t)std::max(dm.T, k_max) < ((int64_t)1 << 31) &&
         dm.heads() * imp_chunks(dm, k_max) * (int64_t)imp_splits(dm, k_max) < ((int64_t)1 << 31);
}

size_t importance_tc_part_bytes(const Dims& dm, int k_max) {
  return (size_t)dm.heads() * imp_chunks(dm, k_max) * imp_splits(dm, k_max) * 128 * sizeof(float);
}

cudaError_t launch_importance_tc(const Dims& dm, int k_max, const void* q_dec, const void* k, const void* k_dec,
                                 const float* vnorm, float* part, float* importance, int32_t* status, LaunchCtx& lc) {
  return dm.d == 128 ? launch_importance_tc_t<2>(dm, k_max, q_dec, k, k_dec, vnorm, part, importance, status, lc)
                     : launch_importance_tc_t<1>(dm, k_max, q_dec, k, k_dec, vnorm, part, importance, status, lc);
}

}  // namespace lukv
