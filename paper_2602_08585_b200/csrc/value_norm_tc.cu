// Value norms of the oracle importance (Sec. 4.1, Eq. "oracle_importance"; App. E: L2 norm of the projected value),
//   vnorm[u][g][j] = || v[u][j] W_O^(g) ||_2 ,   u a KV head, g one of its G query heads, j a rankable position,
// on the tensor cores for bf16 inputs.  Per (u, g) this is a dense contraction (n x d) * (d x D_model)
// followed by a sum of squares over the D_model output columns.  The Gram matrix of the projection (value_norm_gram.cu) needs
// far fewer operations; this kernel serves narrow projections, few positions, unaligned ones, and the positions that the
// other one leaves.
//
// One persistent kernel, one CTA per SM, work items (u, g, chunk of 4096 positions).  For an item the CTA walks the
// projection in panels of 256 output columns and, per panel, the chunk's tiles of 128 positions:
//   warp 0      TMA producer: value tiles (128 positions x d channels, the layout of the key tiles of the scorer)
//   warp 1      allocates tensor memory; one lane issues the MMAs, D[position][column] = V tile * panel^T, N = 256
//   warps 2-5   epilogue: read the accumulator (a row per thread), add the squares to the row's running sum in
//               shared memory; after the last panel write the square roots
//   warps 6-9   panel writers: W_O^(g) is stored [d][D_model], the MMA wants each output column's d channels
//               contiguous, so the panel is transposed on its way into shared memory (8 loads of 4 columns -> 4 rows
//               of 8 channels, stored in the 128-byte-swizzled layout the MMA descriptor describes); a panel serves all
//               tiles of the chunk, and the next one is written while the current one is in use
// The LIST form computes the positions of a chunk that the Gram form left, as many tiles as they fill: eight more warps gather
// their rows with ordinary asynchronous copies, four to a buffer, and eight write the panels, because with few tiles there is
// little else to hide their loads behind.  Chunks of which more than three quarters are left are computed whole, as in the other
// form (a gathered tile takes 0.95 us a panel, a whole chunk's 0.75).  The chunk's positions are listed by all threads, so its
// roles meet at its ends.  256 heads x 4 query heads x 3968 positions x 4096 columns, a call of one step: nothing left 0.53 ms,
// 1 % of the positions 0.89, 9 % 1.03, 27 % 1.9, 70 % 2.9, all 3.9 (11.7 with a single gathering warp); every position in the
// other form at once 3.0 to 3.5.
// Every wait is bounded; the waits are between the warps of one CTA only.
#include "tc_ptx.cuh"

namespace lukv {
namespace {

constexpr int kVnRowTile = 128;                      // positions per MMA (M)
constexpr int kVnColTile = 256;                      // projection columns per MMA (N)
constexpr int kVnChunkTiles = 32;                    // row tiles per work item
constexpr int kVnChunkRows = kVnChunkTiles * kVnRowTile;
constexpr int kVnAHalf = kVnRowTile * 128;           // 64 channels of a value tile; d = 64 NH channels make NH of them
constexpr int kVnBHalf = kVnColTile * 128;           // 64 channels of a panel: 256 rows
__host__ __device__ constexpr int vn_writers(bool list) { return list ? 8 : 4; }
constexpr int kVnGatherPer = 4;  // LIST: gathering warps per value buffer, of two
__host__ __device__ constexpr int vn_threads(bool list) { return 32 * (6 + vn_writers(list) + (list ? 2 * kVnGatherPer : 0)); }
__host__ __device__ constexpr int vn_smem(int NH, bool list) { return 2 * NH * (kVnAHalf + kVnBHalf) + kVnChunkRows * (list ? 6 : 4) + 1024; }

enum { kVnAFull = 0, kVnAEmpty = 2, kVnBFull = 4, kVnBEmpty = 6, kVnTFull = 8, kVnTEmpty = 10, kVnBars = 12 };

struct VnArgs {
  const __nv_bfloat16* v;    // [heads][T][d]
  const __nv_bfloat16* w_o;  // [L][H*G][d][Dm]
  float* vnorm;              // [heads][G][n]
  int L, H, G, T, n, Dm;
  int chunks;                // row chunks per (u, g)
  long long items;           // heads * G * chunks
  uint32_t spin_limit;
  int32_t* status;           // where a wait that ran out is reported
  const uint32_t* left;      // [heads * G][tiles][4] a bit per position to compute (LIST)
  int tiles;                 // 128-position tiles per head
};

// Writes the panel of output columns [m0, m0 + 256) of one projection slice w [64 NH][Dm] into shared memory as 256
// rows (columns of W) of 64 NH channels, in halves of 64 channels, rows of 128 bytes, 16-byte chunk c of row m at
// chunk position c ^ (m & 7).  Columns at or beyond Dm are zero.  kThreads threads, kAhead units at a time.
template <int NH, int kThreads, int kAhead>
__device__ __forceinline__ void vn_write_panel(unsigned char* panel, const __nv_bfloat16* w, int Dm, int m0, int t,
                                               bool vec) {
  if (vec) {
    // unit = (4 columns, 8 channels): 64 x 8 NH units; lanes take consecutive column groups
    static_assert(64 * 8 * NH % (kAhead * kThreads) == 0, "every thread has as many units");
    for (int unit0 = t; unit0 < 64 * 8 * NH; unit0 += kAhead * kThreads) {
      uint2 r[kAhead][8];
#pragma unroll
      for (int h = 0; h < kAhead; ++h) {
        const int unit = unit0 + h * kThreads, m = m0 + 4 * (unit & 63), c8 = unit >> 6;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          r[h][i] = make_uint2(0u, 0u);
          if (m < Dm) r[h][i] = __ldg(reinterpret_cast<const uint2*>(w + (size_t)(8 * c8 + i) * Dm + m));
        }
      }
#pragma unroll
      for (int h = 0; h < kAhead; ++h) {
        const int unit = unit0 + h * kThreads, mq = unit & 63, c8 = unit >> 6, half = c8 >> 3, c = c8 & 7;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint4 o;
          uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const uint32_t a = k < 2 ? r[h][2 * p].x : r[h][2 * p].y, b = k < 2 ? r[h][2 * p + 1].x : r[h][2 * p + 1].y;
            ow[p] = __byte_perm(a, b, (k & 1) ? 0x7632 : 0x5410);
          }
          const int row = 4 * mq + k;
          *reinterpret_cast<uint4*>(panel + half * kVnBHalf + row * 128 + ((c ^ (row & 7)) << 4)) = o;
        }
      }
    }
  } else {
    // any Dm and alignment: one column and 8 channels per unit
    for (int unit = t; unit < 256 * 8 * NH; unit += kThreads) {
      const int row = unit & 255, c8 = unit >> 8;
      const int m = m0 + row;
      uint4 o = make_uint4(0u, 0u, 0u, 0u);
      if (m < Dm) {
        uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
        const unsigned short* ws = reinterpret_cast<const unsigned short*>(w);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const uint32_t lo = __ldg(ws + (size_t)(8 * c8 + 2 * p) * Dm + m);
          const uint32_t hi = __ldg(ws + (size_t)(8 * c8 + 2 * p + 1) * Dm + m);
          ow[p] = lo | (hi << 16);
        }
      }
      const int half = c8 >> 3, c = c8 & 7;
      *reinterpret_cast<uint4*>(panel + half * kVnBHalf + row * 128 + ((c ^ (row & 7)) << 4)) = o;
    }
  }
}

struct VnItem {
  int u, g, row0, ntiles;
  int rows;                  // positions of the chunk (LIST: those to compute)
  const __nv_bfloat16* w;
};
template <int NH>
__device__ __forceinline__ VnItem vn_item(const VnArgs& a, long long idx) {
  VnItem it;
  const int chunk = (int)(idx % a.chunks);
  const long long ug = idx / a.chunks;
  it.g = (int)(ug % a.G);
  it.u = (int)(ug / a.G);
  it.row0 = chunk * kVnChunkRows;
  it.rows = min(kVnChunkRows, a.n - it.row0);
  it.ntiles = (it.rows + kVnRowTile - 1) / kVnRowTile;
  const int layer = (it.u / a.H) % a.L, h = it.u % a.H;
  it.w = a.w_o + ((size_t)layer * a.H * a.G + (size_t)h * a.G + it.g) * (64 * NH) * a.Dm;
  return it;
}

// The bits of 32 positions from row0 + 32 i on (those past the head's end hold anything).
__device__ __forceinline__ uint32_t vn_left(const VnArgs& a, size_t ug, int row0, int i) {
  const int rest = a.n - row0 - 32 * i;
  if (rest <= 0) return 0u;
  const uint32_t bits = a.left[(ug * a.tiles + row0 / kVnRowTile) * 4 + i];
  return rest >= 32 ? bits : bits & ((1u << rest) - 1u);
}

// Lists the positions of the chunk that are left, counted from its first, in order; all threads of the CTA.
__device__ __forceinline__ int vn_list(const VnArgs& a, const VnItem& it, unsigned short* list, int* counts) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t bits = 0;
  int before = 0;
  if (warp < 4) {  // a word per thread
    bits = vn_left(a, (size_t)it.u * a.G + it.g, it.row0, threadIdx.x);
    before = __popc(bits);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, before, off);
      if (lane >= off) before += o;
    }
    if (lane == 31) counts[warp] = before;
    before -= __popc(bits);
  }
  __syncthreads();
  const int all = counts[0] + counts[1] + counts[2] + counts[3];
  if (warp < 4) {
    for (int i = 0; i < warp; ++i) before += counts[i];
    for (; bits; bits &= bits - 1) list[before++] = (unsigned short)(32 * threadIdx.x + __ffs(bits) - 1);
  }
  __syncthreads();
  return all;
}

template <int NH, bool LIST>
__global__ void __launch_bounds__(vn_threads(LIST), 1)
    value_norm_tc_kernel(const __grid_constant__ CUtensorMap v_map, const VnArgs a) {
  constexpr int kVnABytes = NH * kVnAHalf, kVnBBytes = NH * kVnBHalf, kWriters = vn_writers(LIST), kThreads = vn_threads(LIST);
  static_assert(vn_smem(NH, LIST) <= 232448 - 512, "exceeds the shared memory of one CTA");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* a_tiles = smem;                              // [2][kVnABytes]
  unsigned char* panels = smem + 2 * kVnABytes;               // [2][kVnBBytes]
  float* ssq = reinterpret_cast<float*>(panels + 2 * kVnBBytes);  // [kVnChunkRows] running sums of squares
  unsigned short* list = reinterpret_cast<unsigned short*>(ssq + kVnChunkRows);  // LIST: [kVnChunkRows]
  __shared__ __align__(8) uint64_t bars[kVnBars];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s, counts_s[4];
  volatile int* abort_flag = &abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto bar = [&](int kind, int i) { return smem_u32(&bars[kind + i]); };

  if constexpr (LIST) {  // most often nothing is left to do
    pdl_wait();
    constexpr int kWords = kVnChunkRows / 32;
    uint32_t any = 0;
    for (long long k = threadIdx.x; blockIdx.x + k / kWords * gridDim.x < a.items; k += kThreads) {
      const long long idx = blockIdx.x + k / kWords * gridDim.x;
      any |= vn_left(a, (size_t)(idx / a.chunks), (int)(idx % a.chunks) * kVnChunkRows, (int)(k % kWords));
    }
    if (!__syncthreads_or(any != 0)) return;
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(kVnAFull, i), LIST ? kVnGatherPer : 1);
      mbar_init(bar(kVnAEmpty, i), 1);
      mbar_init(bar(kVnBFull, i), kWriters);
      mbar_init(bar(kVnBEmpty, i), 1);
      mbar_init(bar(kVnTFull, i), 1);
      mbar_init(bar(kVnTEmpty, i), 4);
    }
    abort_s = 0;
    // the first kernel of the call clears the word; a wait runs out milliseconds after this, at the earliest
    if (blockIdx.x == 0 && !LIST) atomicExch(a.status, 0);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < kVnChunkRows; i += kThreads) ssq[i] = 0.f;
  if (warp == 1) tmem_alloc(smem_u32(&tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  const int npanels = (a.Dm + kVnColTile - 1) / kVnColTile;

  uint32_t tt = 0, pc = 0;  // value tiles and panels so far
  bool ok = true;
  for (long long idx = blockIdx.x; idx < a.items && ok; idx += gridDim.x) {
    VnItem it = vn_item<NH>(a, idx);
    bool whole = true;  // all positions of the chunk
    if constexpr (LIST) {
      const int rows = vn_list(a, it, list, counts_s);
      if (rows == 0) continue;
      whole = 4 * rows > 3 * it.rows;
      if (!whole) it.rows = rows, it.ntiles = (rows + kVnRowTile - 1) / kVnRowTile;
    }
    if (warp == 0) {
      // ---------------- TMA producer: the value tiles, once per panel ----------------
      if (LIST && !whole) {
        tt += npanels * it.ntiles;
      } else if (lane == 0) {
        for (int cp = 0; cp < npanels && ok; ++cp)
          for (int rt = 0; rt < it.ntiles; ++rt, ++tt) {
            const uint32_t s = tt & 1, ph = (tt >> 1) & 1;
            if (!(ok = mbar_wait(bar(kVnAEmpty, s), ph ^ 1, abort_flag, a.status, a.spin_limit))) break;
            mbar_expect_tx(bar(kVnAFull, s), kVnABytes);
            if constexpr (LIST) mbar_arrive(bar(kVnAFull, s), kVnGatherPer - 1);
            const uint32_t dst = smem_u32(a_tiles + s * kVnABytes);
            const int row = it.u * a.T + it.row0 + rt * kVnRowTile;  // rows past the head are never written back
            for (int h = 0; h < NH; ++h) tma_load_2d(dst + h * kVnAHalf, &v_map, bar(kVnAFull, s), h * 64, row);
          }
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer ----------------
      if (lane == 0) {
        constexpr uint32_t idesc = instr_desc_bf16(kVnRowTile, kVnColTile);
        for (int cp = 0; cp < npanels && ok; ++cp, ++pc) {
          const uint32_t pb = pc & 1;
          if (!(ok = mbar_wait(bar(kVnBFull, pb), (pc >> 1) & 1, abort_flag, a.status, a.spin_limit))) break;
          const uint32_t bp = smem_u32(panels + pb * kVnBBytes);
          for (int rt = 0; rt < it.ntiles; ++rt, ++tt) {
            const uint32_t s = tt & 1, ph = (tt >> 1) & 1;
            if (!(ok = mbar_wait(bar(kVnTEmpty, s), ph ^ 1, abort_flag, a.status, a.spin_limit))) break;
            if (!(ok = mbar_wait(bar(kVnAFull, s), ph, abort_flag, a.status, a.spin_limit))) break;
            tc_fence_after();
            const uint32_t at = smem_u32(a_tiles + s * kVnABytes);
#pragma unroll
            for (int ks = 0; ks < 4 * NH; ++ks) {
              const int h = ks >> 2, sub = ks & 3;
              const uint64_t da = smem_desc_sw128(at + h * kVnAHalf) + (uint64_t)(sub * 2);
              const uint64_t db = smem_desc_sw128(bp + h * kVnBHalf) + (uint64_t)(sub * 2);
              umma_bf16(tmem_base + s * kVnColTile, da, db, idesc, ks > 0);
            }
            umma_commit(bar(kVnAEmpty, s));  // the value tile may be replaced once these MMAs have read it
            umma_commit(bar(kVnTFull, s));   // the accumulator is complete
          }
          if (ok) umma_commit(bar(kVnBEmpty, pb));  // the panel may be overwritten
        }
      }
    } else if (warp < 6) {
      // ---------------- epilogue: a row per thread ----------------
      const int row = 32 * (warp & 3) + lane;  // a warp reads the TMEM lanes of its quadrant
      const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
      for (int cp = 0; cp < npanels && ok; ++cp)
        for (int rt = 0; rt < it.ntiles; ++rt, ++tt) {
          const uint32_t s = tt & 1, ph = (tt >> 1) & 1;
          if (!(ok = mbar_wait(bar(kVnTFull, s), ph, abort_flag, a.status, a.spin_limit))) break;
          tc_fence_after();
          float ss0 = 0.f, ss1 = 0.f, ss2 = 0.f, ss3 = 0.f;
#pragma unroll 1
          for (int c0 = 0; c0 < kVnColTile; c0 += 32) {
            float v[32];
            tmem_ld32(tmem_base + lane_addr + s * kVnColTile + c0, v);
            tmem_ld_wait(v);
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              ss0 = fmaf(v[i], v[i], ss0);
              ss1 = fmaf(v[i + 1], v[i + 1], ss1);
              ss2 = fmaf(v[i + 2], v[i + 2], ss2);
              ss3 = fmaf(v[i + 3], v[i + 3], ss3);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(kVnTEmpty, s), 1);
          ssq[rt * kVnRowTile + row] += (ss0 + ss1) + (ss2 + ss3);  // only this thread touches this entry
        }
      if (ok) {
        float* out = a.vnorm + ((size_t)it.u * a.G + it.g) * a.n + it.row0;
        for (int i = row; i < it.ntiles * kVnRowTile; i += kVnRowTile) {
          if (i < it.rows) out[LIST && !whole ? list[i] : i] = sqrtf(ssq[i]);
          ssq[i] = 0.f;
        }
      }
    } else if (warp < 6 + kWriters) {
      // ---------------- panel writers ----------------
      const int t = threadIdx.x - 6 * 32;
      const bool vec = (a.Dm & 3) == 0 && (reinterpret_cast<uintptr_t>(a.w_o) & 7) == 0;
      for (int cp = 0; cp < npanels; ++cp, ++pc) {
        const uint32_t pb = pc & 1;
        if (!(ok = mbar_wait(bar(kVnBEmpty, pb), ((pc >> 1) & 1) ^ 1, abort_flag, a.status, a.spin_limit))) break;
        vn_write_panel<NH, 32 * kWriters, LIST ? 2 : 1>(panels + pb * kVnBBytes, it.w, a.Dm, cp * kVnColTile, t, vec);
        // the MMA reads shared memory through the asynchronous proxy: order these writes before it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kVnBFull, pb), 1);
      }
    } else if constexpr (LIST) {
      // ---------------- gatherers: the value tiles of the list ----------------
      if (whole) {
        tt += npanels * it.ntiles;
      } else {
        const int which = (warp - 6 - kWriters) / kVnGatherPer, part = (warp - 6 - kWriters) % kVnGatherPer;
        constexpr int kRows = kVnRowTile / kVnGatherPer, kPieces = kRows * 8 * NH / 32;  // 16 bytes each, per lane
        const __nv_bfloat16* v = a.v + ((size_t)it.u * a.T + it.row0) * (64 * NH);
        for (int cp = 0; cp < npanels && ok; ++cp)
          for (int rt = 0; rt < it.ntiles; ++rt, ++tt) {
            const uint32_t s = tt & 1, ph = (tt >> 1) & 1;
            if ((int)s != which) continue;
            uint32_t src[kPieces];
#pragma unroll
            for (int i = 0; i < kPieces; ++i) {
              const int piece = lane + 32 * i, row = kRows * part + piece / (8 * NH);
              // rows past the last are never written back
              src[i] = list[min(rt * kVnRowTile + row, it.rows - 1)] * (64u * NH) + 8 * (piece % (8 * NH));
            }
            if (!(ok = mbar_wait(bar(kVnAEmpty, s), ph ^ 1, abort_flag, a.status, a.spin_limit))) break;
            const uint32_t dst = smem_u32(a_tiles + s * kVnABytes);
            int first = lane;
            asm volatile("" : "+r"(first));  // the places are worked out again: kept, they would take a register each
#pragma unroll
            for (int i = 0; i < kPieces; ++i) {
              const int piece = first + 32 * i, row = kRows * part + piece / (8 * NH), c8 = piece % (8 * NH);
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (c8 >> 3) * kVnAHalf + row * 128 +
                                                                              (((c8 & 7) ^ (row & 7)) << 4)), "l"(v + src[i])
                           : "memory");
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            // the MMA reads shared memory through the asynchronous proxy: order these copies before it
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kVnAFull, s), 1);
          }
      }
    }
    if constexpr (LIST) {
      __syncthreads();  // the list is free again
      ok = *abort_flag == 0;
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

bool value_norm_tc_supported(const Dims& dm) {
  return dm.dtype == LUKV_DTYPE_BF16 && dm.heads() * (int64_t)dm.T < ((int64_t)1 << 31);
}

template <bool LIST>
static cudaError_t launch_value_norm_t(const Dims& dm, int d_model, const void* v, const void* w_o, float* vnorm,
                                       const uint32_t* left, int32_t* status, LaunchCtx& lc) {
  CUtensorMap vm;
  if (!make_map(&vm, v, (uint64_t)dm.heads() * dm.T, dm.d)) return cudaErrorNotSupported;
  VnArgs a;
  a.v = static_cast<const __nv_bfloat16*>(v);
  a.w_o = static_cast<const __nv_bfloat16*>(w_o);
  a.vnorm = vnorm;
  a.L = dm.L, a.H = dm.H, a.G = dm.G, a.T = dm.T, a.n = dm.n, a.Dm = d_model;
  a.chunks = (dm.n + kVnChunkRows - 1) / kVnChunkRows;
  a.items = (long long)dm.heads() * dm.G * a.chunks;
  a.status = status;
  a.left = left;
  a.tiles = (dm.n + kVnRowTile - 1) / kVnRowTile;
  int drop = 0;
  score_test_hooks(&a.spin_limit, &drop);
  int sms = 0;
  cudaError_t e;
  if ((e = device_sms(&sms)) != cudaSuccess) return e;
  auto kern = dm.d == 128 ? value_norm_tc_kernel<2, LIST> : value_norm_tc_kernel<1, LIST>;
  const int smem = vn_smem(dm.d / 64, LIST);
  if ((e = allow_smem((const void*)kern, smem)) != cudaSuccess) return e;
  const long long grid = a.items < sms ? a.items : sms;  // one CTA per SM: each owns the SM's tensor memory
  e = launch_pdl(kern, dim3((unsigned)grid), dim3(vn_threads(LIST)), smem, lc.st, LIST, vm, a);
  lc.mark(LIST ? "value_norm_list" : "value_norm_tc");
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_value_norm_tc(const Dims& dm, int d_model, const void* v, const void* w_o, float* vnorm,
                                 const uint32_t* left, int32_t* status, LaunchCtx& lc) {
  return left ? launch_value_norm_t<true>(dm, d_model, v, w_o, vnorm, left, status, lc)
              : launch_value_norm_t<false>(dm, d_model, v, w_o, vnorm, nullptr, status, lc);
}

}  // namespace lukv
