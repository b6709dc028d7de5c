// Stage (a) on the 5th-generation tensor cores (bf16): one persistent kernel
// computes the un-pooled observation-window scores of every head.
//
// The window logits S = Q K^T of Eq. 1 (Sec. 3.1) come from tcgen05.mma with fp32
// accumulators in tensor memory; operands are staged in shared memory by TMA (128-byte
// swizzle, no multicast).  A row's softmax normaliser needs every key of the head before any
// probability is final, so each head is swept twice:
//   pass 1  D[query row][key]: a thread owns one query row in TMEM and folds its columns into
//           a (reference, sum-exp) pair; the partials of a work item go to global memory and
//           the CTA that delivers a head's last partial folds them into the row log-sum-exp
//   pass 2  D[key][query row] (operands swapped): a thread owns one key and adds
//           exp2(x - lse_row) over all rows in registers -> the un-pooled score of the key
// Both operand tiles are K-major, so the same shared-memory tiles serve as A or B.
//
// Work item = (head, run of at most item_tiles key tiles).  Items are dealt round-robin to a grid of
// at most one CTA per SM, launched cooperatively (all CTAs resident).  A CTA runs pass 1
// lag-1 items ahead of pass 2, so that the log-sum-exp of a head is normally complete before
// pass 2 needs it.  With small items the key tiles pass 2 re-reads are still in L2 (K crosses
// HBM once); large ones re-read K from HBM but change jobs less often (the launcher weighs it).
//
// Warp roles per CTA: 4*NQ epilogue warps in NQ quads (a warp may only read the TMEM lanes
// 32*(warp%4)..+31), then one warp each: TMA producer, MMA issuer 0 and TMEM owner, MMA issuer 1,
// helper (pass-1 partials -> global memory, head completion, -lse -> shared memory: it keeps every
// global-memory round trip off the epilogue warps).
// Every wait is bounded; a wait that runs out raises the CTA's abort flag and stores
// LUKV_ERR_TIMEOUT to the status word; the CTA then skips the remaining work and tears down
// normally.
#include <algorithm>

#include "score_chunks.cuh"

namespace lukv {
namespace {


// ---- shared-memory layout ---------------------------------------------------------------------

// NH: halves of 64 channels, d = 64 NH.
template <int MT, int NQ, int NH>
struct Plan {
  static_assert(MT == 1 || NQ == 2, "two query-row blocks are split over exactly two quads");
  // An mbarrier wait only knows the parity of the phase it waits for, so a thread must not wait for a phase whose predecessor may
  // be incomplete.  An accumulator buffer takes one row block of one key tile, buffer (tile * MT + block) % kNumBufs, and is
  // written by issuer tile % 2; see kFullSets for its readers.
  static_assert(NQ == 2 || (MT == 1 && NQ == 3), "two quads, or three that take the tiles in turn");
  static constexpr int kEpiWarps = 4 * NQ;
  // + TMA producer, two MMA issuers, helper.  The count stays a multiple of 4 warps: the register
  // file is handed out as if the CTA were rounded up to one.
  static constexpr int kThreads = (kEpiWarps + 4) * 32;
  // Key-tile ring.  The count must be even: tile t uses stage t % kStages and is issued by issuer
  // t % 2, so with an even count every stage (its "full" barrier) has one waiting thread.  With an
  // odd count the two issuers would take turns on a stage, and the one that runs ahead could wait
  // for a phase two ahead of the barrier -- which a parity wait reports as complete while the
  // previous load of that stage is still in flight.
  static constexpr int kStages = 4 * (3 - NH);
  static constexpr int kStageBytes = NH * kHalfBytes;
  static_assert(kStages % 2 == 0, "a key stage must always be consumed by the same MMA issuer");
  // Query tiles of the job in the tensor pipe and of the next one.  One slot where two of 256 rows x 128 channels would leave room
  // for two key stages only, which do not cover the latency of their loads (eight 16k sequences of 256 rows: 7690 us a call with
  // two slots and two stages, 7615 so).
  static constexpr int kQSlots = MT == 2 && NH == 2 ? 1 : 2;
  static constexpr int kQBytes = MT * kStageBytes;     // [half][MT*128 rows][128 B]
  static constexpr int kFinBufs = 1;                   // blocks of partials in flight while a head is folded
  static constexpr int kFinBytes = 16384;              // one block
  static constexpr int kFinParts = kFinBytes / (128 * MT * 4);  // items per block (one float per row and item)
  static constexpr int kKOff = kQSlots * kQBytes;
  static constexpr int kFinOff = kKOff + kStages * kStageBytes;
  static constexpr int kBarOff = kFinOff + kFinBufs * kFinBytes;
  static constexpr int kNumBufs = 4;                   // accumulator buffers in TMEM, one row block of a key tile each
  static constexpr int kBufCols = 128;
  // "Accumulator complete" barriers per buffer, used in turn, so that a quad that runs ahead waits on a barrier whose previous phase
  // is long complete.  With one row block a quad only ever reads what one issuer wrote (or, with three quads, is held back by the
  // key ring), two sets do.  With two it reads one block of every tile in pass 1 and both of every other one in pass 2: a set per
  // key stage, since a tile 2 kFullSets back that is not issued keeps the key ring from loading the tile before this one.
  static constexpr int kFullSets = MT == 2 ? kStages : 2;
  // barriers: full[kStages], empty[kStages], qfull[kQSlots], qempty[kQSlots], tfull[kFullSets][kNumBufs],
  // tempty[kNumBufs], pub_full[NQ], pub_empty[NQ], lse_full[kMaxLag], lse_empty[kMaxLag], fin[kFinBufs]
  static constexpr int kBarFull = 0, kBarEmpty = kStages, kBarQFull = 2 * kStages, kBarQEmpty = kBarQFull + kQSlots,
                       kBarTFull = kBarQEmpty + kQSlots, kBarTEmpty = kBarTFull + kFullSets * kNumBufs,
                       kBarPubFull = kBarTEmpty + kNumBufs, kBarPubEmpty = kBarPubFull + NQ,
                       kBarLseFull = kBarPubEmpty + NQ, kBarLseEmpty = kBarLseFull + kMaxLag,
                       kBarFin = kBarLseEmpty + kMaxLag, kNumBars = kBarFin + kFinBufs;
  static constexpr int kMiscOff = (kBarOff + kNumBars * 8 + 15) & ~15;  // tmem base, abort flag
  static constexpr int kPubOff = kMiscOff + 16;        // [NQ][128] (reference, sum-exp) handed to the publisher warp
  static constexpr int kLseOff = kPubOff + NQ * 128 * 8;  // [kMaxLag][256] -lse of the pass-2 jobs to come
  static_assert(kLseOff % 16 == 0, "lse rows are read with 16-byte loads");
  static constexpr int kTotal = kLseOff + kMaxLag * 256 * 4 + 1024;  // + slack for the 1024-byte alignment
  static_assert(kTotal <= 232448, "exceeds the shared memory of one CTA");
};

struct FusedArgs {
  float* stats;        // pass 1 partials: [heads][items_per_head][128*MT] log-sum-exp of the item's keys, exp2 domain
  float* lse;          // [heads][lse_rows] (row log-sum-exp in the exp2 domain, tag); zero at launch
  float* raw;          // pass 2 out: [heads][n_stride]
  int* head_cnt;       // [heads] items whose partials were delivered (zero at launch)
  int32_t* dev_status;
  int M, T, w, n;
  int lse_rows;        // M rounded up to a multiple of 4
  int nheads;
  int item_tiles, items_per_head, tiles_T, tiles_n;
  uint32_t iph_magic;  // div_magic(items_per_head)
  int adapt_items;     // host only: let the launcher pick a number of tiles from item_tiles on
  int npad;            // pass 2: query rows rounded up to a multiple of 32 (MMA N and columns read)
  int lag;             // 2..kMaxLag: pass 1 of item k+lag-1 precedes pass 2 of item k
  int l2_hints;        // 1: pass-1 key loads ask L2 to keep the lines, pass-2 loads to drop them first
  float scale_log2;
  // sequences of different lengths in one launch (RAGGED kernels): seq_T[q] = context length of sequence q,
  // seq_item0[q] = number of its first work item; heads_per_seq heads each.  The uniform fields above then hold
  // the maxima (strides and capacities).  The tables travel by value in the launch arguments.
  int seq_T[kMaxRaggedSeqs], seq_item0[kMaxRaggedSeqs], seq_iph[kMaxRaggedSeqs];
  uint32_t seq_magic[kMaxRaggedSeqs];  // div_magic(seq_iph)
  int n_seq, heads_per_seq, total_items;
  int T_stride, n_stride;  // rows between consecutive heads in K and in the raw scores
  uint32_t spin_limit; // iterations a wait may take
  int drop_item;       // test hook: this work item's partials are stored but never counted in (-1: none)
};

struct Job {
  int u;       // head
  int c;       // item of the head
  int tile0;   // first key tile
  int ntiles;  // key tiles of this job (may be 0)
  int n;       // rankable positions of the head
  int iph;     // work items of the head
  bool p2;
};

// Quotients by a number of items without a division: that would go through the special-function unit, where it would queue
// behind the exponentials of the epilogue, and every role works its job out when it changes jobs (128 heads x 157 tiles, 14 jobs a
// CTA: 367 us a call with three divisions a job, 347 with none).  Exact while dividend times divisor stays below 2^32.
__host__ __device__ inline uint32_t div_magic(int d) { return d > 1 ? (uint32_t)((1ull << 32) / (uint32_t)d) + 1u : 0u; }
__device__ __forceinline__ int div_by(int x, uint32_t magic) { return magic ? (int)__umulhi((uint32_t)x, magic) : x; }

template <bool RAGGED>
__device__ __forceinline__ Job make_job(int k, bool p2, const FusedArgs& a) {
  Job j;
  j.p2 = p2;
  const int item = (int)blockIdx.x + k * (int)gridDim.x;
  int tiles_T = a.tiles_T, tiles_n = a.tiles_n, local = item, head0 = 0;
  uint32_t magic = a.iph_magic;
  j.n = a.n;
  j.iph = a.items_per_head;
  if (RAGGED) {
    int lo = 0, hi = a.n_seq;  // the sequence whose items contain `item`
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (a.seq_item0[mid] <= item) lo = mid; else hi = mid;
    }
    j.n = a.seq_T[lo] - a.w;
    tiles_T = (a.seq_T[lo] + kTileKeys - 1) / kTileKeys;
    tiles_n = (j.n + kTileKeys - 1) / kTileKeys;
    j.iph = a.seq_iph[lo];
    magic = a.seq_magic[lo];
    local = item - a.seq_item0[lo];
    head0 = lo * a.heads_per_seq;
  }
  const int hu = div_by(local, magic);
  j.c = local - hu * j.iph;
  j.u = head0 + hu;
  int end;
  if (RAGGED) {
    // a head's items differ by one tile at most: with full items and a short last one a CTA could be dealt the long ones every
    // time (eight sequences of 1750 to 16000 keys: 1493 us a call with full items, 1438 so)
    const int base = div_by(tiles_T, magic), rest = tiles_T - base * j.iph;
    j.tile0 = j.c * base + min(j.c, rest);
    end = j.tile0 + base + (j.c < rest ? 1 : 0);
  } else {
    // where all heads are alike the short items fall to all CTAs (128 x 157 tiles: 343 us a call, 347 with equal items)
    j.tile0 = j.c * a.item_tiles;
    end = min(j.tile0 + a.item_tiles, tiles_T);
  }
  j.ntiles = max(0, (p2 ? min(end, tiles_n) : end) - j.tile0);
  return j;
}

// Job `idx` of a CTA that owns K items: lag-1 pass-1 jobs first, then pass 1 of item k+lag-1
// alternating with pass 2 of item k, then the remaining pass-2 jobs.
template <bool RAGGED>
__device__ __forceinline__ Job decode_job(int idx, int K, const FusedArgs& a) {
  const int lead = min(a.lag - 1, K);
  if (idx < lead) return make_job<RAGGED>(idx, false, a);
  const int r = idx - lead, pairs = 2 * (K - lead);
  if (r < pairs) return (r & 1) ? make_job<RAGGED>(r >> 1, true, a) : make_job<RAGGED>(lead + (r >> 1), false, a);
  return make_job<RAGGED>(K - lead + (r - pairs), true, a);
}

template <int MT, int NQ, int NH, bool RAGGED>
__global__ void __launch_bounds__(Plan<MT, NQ, NH>::kThreads, 1)
    score_fused_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                       const FusedArgs a) {
  using P = Plan<MT, NQ, NH>;
  constexpr int kStages = P::kStages, kStageBytes = P::kStageBytes;
  constexpr int kNumBufs = P::kNumBufs;
  constexpr int kEpiWarps = P::kEpiWarps;
  constexpr int kRowsPad = 128 * MT;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t q_s = sbase;
  const uint32_t k_s = sbase + P::kKOff;
  const uint32_t bars = sbase + P::kBarOff;
  auto bar = [&](int first, int i) { return bars + 8u * (uint32_t)(first + i); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + P::kMiscOff);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + P::kMiscOff + 4);
  float2* pub_s = reinterpret_cast<float2*>(smem + P::kPubOff);   // [NQ][128]
  float* nlse_s = reinterpret_cast<float*>(smem + P::kLseOff);    // [kMaxLag][256]

  pdl_launch_dependents();  // kernels that do not read the scores may start on SMs this grid leaves free
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total_items = a.total_items;
  const int K = (total_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // items of this CTA (>= 1)
  const int njobs = 2 * K;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar(P::kBarFull, s), 1);
      mbar_init(bar(P::kBarEmpty, s), 1);
    }
    for (int s = 0; s < P::kQSlots; ++s) {
      mbar_init(bar(P::kBarQFull, s), 1);
      mbar_init(bar(P::kBarQEmpty, s), 2);  // both MMA issuers
    }
    for (int b = 0; b < kNumBufs; ++b) {
      for (int f = 0; f < P::kFullSets; ++f) mbar_init(bar(P::kBarTFull, f * kNumBufs + b), 1);
      mbar_init(bar(P::kBarTEmpty, b), 4);
    }
    for (int q = 0; q < NQ; ++q) {
      mbar_init(bar(P::kBarPubFull, q), 4);
      mbar_init(bar(P::kBarPubEmpty, q), 1);
    }
    for (int s = 0; s < kMaxLag; ++s) {
      mbar_init(bar(P::kBarLseFull, s), 1);
      mbar_init(bar(P::kBarLseEmpty, s), kEpiWarps);
    }
    for (int b = 0; b < P::kFinBufs; ++b) mbar_init(bar(P::kBarFin, b), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpiWarps + 1) tmem_alloc(smem_u32((const void*)tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == kEpiWarps) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      const uint64_t keep = l2_policy_evict_last(), drop = l2_policy_evict_first();
      uint32_t tt = 0, jq = 0;
      for (int idx = 0; idx < njobs; ++idx) {
        const Job j = decode_job<RAGGED>(idx, K, a);
        if (j.ntiles == 0) continue;
        // With one slot the query tiles follow the first key tiles, which need not wait for the job before to end.
        const int q_after = P::kQSlots == 1 ? min(kStages, j.ntiles) : 0;
        bool ok = true;
        auto load_q = [&]() -> bool {
          const uint32_t slot = jq % P::kQSlots;
          if (!mbar_wait(bar(P::kBarQEmpty, slot), ((jq / P::kQSlots) & 1) ^ 1, abort_flag, a.dev_status, a.spin_limit)) return false;
          mbar_expect_tx(bar(P::kBarQFull, slot), P::kQBytes);
          const uint32_t qd = q_s + slot * P::kQBytes;
          for (int h = 0; h < NH; ++h)
            for (int mt = 0; mt < MT; ++mt) {
              const uint32_t dst = qd + h * (MT * kHalfBytes) + mt * kHalfBytes;
              if (a.l2_hints) tma_load_2d_hint(dst, &q_map, bar(P::kBarQFull, slot), h * 64, j.u * a.M + mt * 128, keep);
              else tma_load_2d(dst, &q_map, bar(P::kBarQFull, slot), h * 64, j.u * a.M + mt * 128);
            }
          ++jq;
          return true;
        };
        if (q_after == 0 && !load_q()) break;
        for (int t = 0; t < j.ntiles; ++t, ++tt) {
          const uint32_t s = tt % kStages, ph = (tt / kStages) & 1;
          if (!(ok = mbar_wait(bar(P::kBarEmpty, s), ph ^ 1, abort_flag, a.dev_status, a.spin_limit))) break;
          mbar_expect_tx(bar(P::kBarFull, s), kStageBytes);
          const int row = j.u * a.T_stride + (j.tile0 + t) * kTileKeys;
          const uint32_t dst = k_s + s * kStageBytes;
          if (a.l2_hints) {
            const uint64_t pol = j.p2 ? drop : keep;
            for (int h = 0; h < NH; ++h) tma_load_2d_hint(dst + h * kHalfBytes, &k_map, bar(P::kBarFull, s), h * 64, row, pol);
          } else {
            for (int h = 0; h < NH; ++h) tma_load_2d(dst + h * kHalfBytes, &k_map, bar(P::kBarFull, s), h * 64, row);
          }
          if (t + 1 == q_after && !(ok = load_q())) break;
        }
        if (!ok) break;
      }
    }
  } else if (warp == kEpiWarps + 1 || warp == kEpiWarps + 2) {
    // ---------------- MMA issuers ----------------
    // Two threads (in two warps) issue alternate key tiles.  A thread is held up by its waits and by
    // the tensor pipe's issue queue; with two of them one can wait while the other issues, so the
    // pipe does not idle between tiles.  Tiles that share an accumulator buffer or a key stage
    // (both have an even count) always belong to the same issuer, which keeps them in order.
    if (lane == 0) {
      const uint32_t me = warp == kEpiWarps + 1 ? 0u : 1u;
      uint32_t tt = 0, jq = 0;
      for (int idx = 0; idx < njobs; ++idx) {
        const Job j = decode_job<RAGGED>(idx, K, a);
        if (j.ntiles == 0) continue;
        const uint32_t slot = jq % P::kQSlots;
        const uint32_t qd = q_s + slot * P::kQBytes;
        bool ok = true, have_q = false;
        for (int t = 0; t < j.ntiles; ++t, ++tt) {
          if ((tt & 1) != me) continue;
          if (!have_q) {
            if (!(ok = mbar_wait(bar(P::kBarQFull, slot), (jq / P::kQSlots) & 1, abort_flag, a.dev_status, a.spin_limit))) break;
            have_q = true;
          }
          const uint32_t s = tt % kStages, ph = (tt / kStages) & 1;
          if (!(ok = mbar_wait(bar(P::kBarFull, s), ph, abort_flag, a.dev_status, a.spin_limit))) break;
          const uint32_t kt = k_s + s * kStageBytes;
          for (int mt = 0; mt < MT; ++mt) {
            const uint32_t st = tt * MT + mt, buf = st % kNumBufs, use = st / kNumBufs;
            if (!(ok = mbar_wait(bar(P::kBarTEmpty, buf), (use & 1) ^ 1, abort_flag, a.dev_status, a.spin_limit))) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + buf * P::kBufCols;
            const uint32_t qb = qd + mt * kHalfBytes;
            // pass 1: D[q row][key], A = 128 query rows, B = K tile; pass 2: D[key][q row], A = K tile, B = the query rows (up to
            // 128, padded to a multiple of 32)
            const uint32_t idesc = j.p2 ? instr_desc_bf16(128, min(128, a.npad - 128 * mt)) : instr_desc_bf16(128, kTileKeys);
#pragma unroll
            for (int ks = 0; ks < 4 * NH; ++ks) {
              const int h = ks >> 2, sub = ks & 3;
              const uint64_t dq = smem_desc_sw128(qb + h * (MT * kHalfBytes)) + (uint64_t)(sub * 2);
              const uint64_t dk = smem_desc_sw128(kt + h * kHalfBytes) + (uint64_t)(sub * 2);
              umma_bf16(d_tmem, j.p2 ? dk : dq, j.p2 ? dq : dk, idesc, ks > 0);
            }
            umma_commit(bar(P::kBarTFull, buf + kNumBufs * (use % P::kFullSets)));   // the accumulator is complete
          }
          if (!ok) break;
          umma_commit(bar(P::kBarEmpty, s));     // the stage may be refilled once these MMAs have read it
        }
        // An issuer without a tile in this job (a job of one tile) waits all the same: else it could hand the slot back twice
        // while the other issuer still works on the job before in it, which would free that job's query tiles, and its
        // next wait on this barrier would be two phases ahead, which a parity wait reports as complete.
        if (ok && !have_q) ok = mbar_wait(bar(P::kBarQFull, slot), (jq / P::kQSlots) & 1, abort_flag, a.dev_status, a.spin_limit);
        if (!ok) break;
        umma_commit(bar(P::kBarQEmpty, slot));   // this issuer's share of the job no longer needs the query tiles
        ++jq;
      }
    }
  } else if (warp == kEpiWarps + 3) {
    // ---------------- helper: everything that needs a global-memory round trip ----------------
    // publish(k): merge the quads' pass-1 partials of item k, store them, count the item in
    //   (release).  The warp that counts a head's last item folds all its partials into the row
    //   log-sum-exp and stores it as (value, tag) pairs, zero at launch.
    // prefetch(k): poll those pairs for the head of item k (polling the data itself saves a flag
    //   round trip) and put -lse into shared memory for pass 2 of item k, which the quads reach
    //   several jobs after its pass 1.
    // Both are attempted in turn without blocking, so a head that completes late does not hold up
    // the publication of this CTA's next partials.
    uint32_t fin_uses[P::kFinBufs] = {};
    constexpr int kRowsLaneP = 4 * MT;
    int kp = 0, kf = 0;
    uint32_t p2c = 0, idle = 0;
    while ((kp < K || kf < K) && !*abort_flag) {
      bool progress = false;
      if (kp < K) {
        int ready = 1;
        if (lane == 0)
          for (int q = 0; q < NQ; ++q) ready &= (int)mbar_try_wait(bar(P::kBarPubFull, q), kp & 1);
        ready = __shfl_sync(0xffffffffu, ready, 0);
        if (ready) {
          const int k = kp;
          const bool ok = true;
          const Job j1 = make_job<RAGGED>(k, false, a);
          if (ok) {
            // one value per row: the log-sum-exp of the item's keys, m + log2(l); -inf for an empty partial
            float* dst = a.stats + ((size_t)j1.u * a.items_per_head + j1.c) * kRowsPad;
#pragma unroll
            for (int rr = 0; rr < kRowsPad; rr += 32) {
              float2 v = pub_s[rr + lane];
              if (MT == 1) {
                // the quads hold partials of the same 128 rows over different key tiles: merge them
#pragma unroll
                for (int q = 1; q < NQ; ++q) {
                  const float2 o = pub_s[q * 128 + rr + lane];
                  if (o.y > 0.f) {  // an empty partial is (-inf, 0)
                    const float mn = fmaxf(v.x, o.x);
                    v.y = v.y * ex2(v.x - mn) + o.y * ex2(o.x - mn);
                    v.x = mn;
                  }
                }
              }
              dst[rr + lane] = p1_log(v.x, v.y);
            }
          }
          __syncwarp();
          if (lane == 0 && ok)
            for (int q = 0; q < NQ; ++q) mbar_arrive(bar(P::kBarPubEmpty, q), 1);
          // count the item in (release: the partials above; acquire: everybody else's)
          int last = 0;
          const bool dropped = (int)blockIdx.x + k * (int)gridDim.x == a.drop_item;
          if (lane == 0 && ok && !dropped && !*abort_flag)
            last = atom_add_acq_rel(a.head_cnt + j1.u, 1) == j1.iph - 1;
          last = __shfl_sync(0xffffffffu, last, 0);
          if (last) {
            // Fold the head's partials into lse = log2(sum_c 2^(v_c)).  The bulk-copy engine brings them
            // into shared memory (one round trip instead of one per load).  This warp competes with the
            // epilogue warps for issue slots and the head's consumers wait for the result, so the fold
            // is kept short: lane i owns rows 4i..4i+3 (one 16-byte load per item), terms are added
            // relative to the first item's value, and the exact two-sweep form (maximum first) is only
            // the fallback when that sum leaves a safe range.
            constexpr int kVecs = MT;  // float4 per lane and item
            const char* src = reinterpret_cast<const char*>(a.stats) + (size_t)j1.u * a.items_per_head * kRowsPad * 4;
            const int nblk = (j1.iph + P::kFinParts - 1) / P::kFinParts;
            auto request = [&](int blk) {  // lane 0
              const int parts = min(P::kFinParts, j1.iph - blk * P::kFinParts);
              const uint32_t bytes = (uint32_t)parts * kRowsPad * 4;
              mbar_expect_tx(bar(P::kBarFin, 0), bytes);
              bulk_load(sbase + P::kFinOff, src + (size_t)blk * P::kFinParts * kRowsPad * 4, bytes, bar(P::kBarFin, 0));
            };
            const float4* part = reinterpret_cast<const float4*>(smem + P::kFinOff);
            float ref[kVecs][4], sum[kVecs][4];
            bool fin_ok = true;
            for (int pass = 0; pass < 2 && fin_ok; ++pass) {  // pass 1 only if pass 0 left the safe range
              for (int blk = 0; blk < nblk && fin_ok; ++blk) {
                asm volatile("fence.proxy.async;" ::: "memory");
                __syncwarp();
                if (lane == 0) request(blk);
                fin_ok = mbar_wait(bar(P::kBarFin, 0), fin_uses[0] & 1, abort_flag, a.dev_status, a.spin_limit);
                ++fin_uses[0];
                if (!fin_ok) break;
                const int parts = min(P::kFinParts, j1.iph - blk * P::kFinParts);
                if (blk == 0) {
#pragma unroll
                  for (int vv = 0; vv < kVecs; ++vv) {
                    float4 r0 = part[vv * 32 + lane];
                    ref[vv][0] = r0.x, ref[vv][1] = r0.y, ref[vv][2] = r0.z, ref[vv][3] = r0.w;
                    sum[vv][0] = sum[vv][1] = sum[vv][2] = sum[vv][3] = 0.f;
                  }
                }
                if (pass == 1 && blk == 0) {
                  // the fallback needs the maximum of every row first; it is rare, so it simply reads the
                  // partials from global memory
                  const float4* g = reinterpret_cast<const float4*>(src);
                  for (int c = 0; c < j1.iph; ++c)
#pragma unroll
                    for (int vv = 0; vv < kVecs; ++vv) {
                      const float4 v = __ldcg(g + (size_t)c * (kRowsPad / 4) + vv * 32 + lane);
                      ref[vv][0] = fmaxf(ref[vv][0], v.x), ref[vv][1] = fmaxf(ref[vv][1], v.y);
                      ref[vv][2] = fmaxf(ref[vv][2], v.z), ref[vv][3] = fmaxf(ref[vv][3], v.w);
                    }
                }
                for (int c0 = 0; c0 < parts; c0 += 8)
#pragma unroll
                  for (int cc = 0; cc < 8; ++cc)
                    if (c0 + cc < parts) {
#pragma unroll
                      for (int vv = 0; vv < kVecs; ++vv) {
                        const float4 v = part[(c0 + cc) * (kRowsPad / 4) + vv * 32 + lane];
                        sum[vv][0] += ex2(v.x - ref[vv][0]);
                        sum[vv][1] += ex2(v.y - ref[vv][1]);
                        sum[vv][2] += ex2(v.z - ref[vv][2]);
                        sum[vv][3] += ex2(v.w - ref[vv][3]);
                      }
                    }
              }
              bool safe = true;
#pragma unroll
              for (int vv = 0; vv < kVecs; ++vv)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (4 * (vv * 32 + lane) + e < a.M) safe = safe && (sum[vv][e] >= 1e-30f) && (sum[vv][e] <= 1e30f);
              if (__all_sync(0xffffffffu, safe)) break;
            }
            float4* out = reinterpret_cast<float4*>(a.lse) + (size_t)j1.u * (a.lse_rows / 2);
#pragma unroll
            for (int vv = 0; vv < kVecs; ++vv) {
              const int row = 4 * (vv * 32 + lane);
              if (row < a.lse_rows && fin_ok) {
                __stcg(out + row / 2, make_float4(ref[vv][0] + log2f(sum[vv][0]), 1.f, ref[vv][1] + log2f(sum[vv][1]), 1.f));
                if (row + 2 < a.lse_rows)
                  __stcg(out + row / 2 + 1,
                         make_float4(ref[vv][2] + log2f(sum[vv][2]), 1.f, ref[vv][3] + log2f(sum[vv][3]), 1.f));
              }
            }
          }
          ++kp;
          progress = true;
        }
      }
      if (kf < kp) {
        const Job j2 = make_job<RAGGED>(kf, true, a);
        if (j2.ntiles == 0) {
          ++kf;
          progress = true;
        } else {
          const uint32_t slot = p2c % a.lag;
          int freeslot = 0;
          if (lane == 0) freeslot = (int)mbar_try_wait(bar(P::kBarLseEmpty, slot), ((p2c / a.lag) & 1) ^ 1);
          freeslot = __shfl_sync(0xffffffffu, freeslot, 0);
          if (freeslot) {
            const float2* src = reinterpret_cast<const float2*>(a.lse) + (size_t)j2.u * a.lse_rows;
            float2 v[kRowsLaneP];
            bool mine = true;
#pragma unroll
            for (int jj = 0; jj < kRowsLaneP; ++jj) {
              const int row = 32 * jj + lane;
              if (row < a.M) {
                v[jj] = ld_relaxed_f2(src + row);
                mine = mine && v[jj].y != 0.f;
              }
            }
            if (__all_sync(0xffffffffu, mine)) {
#pragma unroll
              for (int jj = 0; jj < 8; ++jj) {
                const int row = 32 * jj + lane;
                nlse_s[slot * 256 + row] = (jj < kRowsLaneP && row < a.M) ? -v[jj < kRowsLaneP ? jj : 0].x : -INFINITY;
              }
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(P::kBarLseFull, slot), 1);
              ++p2c;
              ++kf;
              progress = true;
            }
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
        if (idle > 8) __nanosleep(100);
      }
    }
  } else {
    // ---------------- epilogue quads ----------------
    const int quad = warp >> 2;
    const int qtid = threadIdx.x & 127;                          // TMEM lane of this thread
    const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
    const uint64_t sc2 = pack2(a.scale_log2, a.scale_log2);
    uint32_t tt = 0, p1c = 0, p2c = 0;
    // Row block `st` (counted over all tiles of the CTA) lies in buffer st % 4.  The waits give one answer to the whole warp, which
    // goes on to warp-wide loads.
    // (The one test ahead: a wait that may suspend the warp comes back late; 256 heads x 32768 keys 1109 us a call without it, 1093 so,
    // 1097 with 32 tests, 1107 where every wait of the kernel tests first.)
    auto full_wait = [&](uint32_t st) -> bool {
      const uint32_t buf = st % kNumBufs, use = st / kNumBufs;
      const uint32_t full = bar(P::kBarTFull, buf + kNumBufs * (use % P::kFullSets)), parity = (use / P::kFullSets) & 1;
      if (__all_sync(0xffffffffu, mbar_test_wait(full, parity))) return true;
      return __all_sync(0xffffffffu, mbar_wait(full, parity, abort_flag, a.dev_status, a.spin_limit));
    };
    auto column = [&](uint32_t st) { return tmem_base + lane_addr + (st % kNumBufs) * P::kBufCols; };
    auto release = [&](uint32_t st) {  // this warp has the last columns it needs in registers
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(P::kBarTEmpty, st % kNumBufs), 1);
    };
    float va[32], vb[32];
    for (int idx = 0; idx < njobs; ++idx) {
      const Job j = decode_job<RAGGED>(idx, K, a);
      if (j.ntiles == 0) continue;
      // The quads take the tiles in turn; with two row blocks pass 1 gives each quad one block of every tile.  Buffers of one block
      // instead of whole tiles let the MMAs of a quad's next tile start when half of this one is read, not all of it.
      const bool every = MT == 2 && !j.p2;
      const int step = every ? 1 : NQ;
      int t = every ? 0 : (int)((quad + NQ - tt % NQ) % NQ);
      if (!j.p2) {
        // ---- pass 1: (reference, sum-exp) of this thread's query row over the job's keys.  A tile is one stretch of code without a
        // branch, relative to the reference so far (the maximum of the job's first 32 keys to begin with); a sum that leaves the
        // safe range, or a tile with keys hidden from some row, is done again chunk by chunk, exactly.  The range is wide (2^80):
        // with one of 2^40, tested per chunk, outlier channels at head size 64 (logits of 23 binary orders' standard deviation)
        // sent every tenth chunk through the exact form (128 heads x 20011 keys: 345 us a call; 323 with the wide range, 305
        // tested per tile; 256 heads x 32768 keys at head size 128 1217 and 1163).
        const int r = (MT == 2 ? 128 * quad : 0) + qtid;
        const int lim = r < a.M ? j.n + (r % a.w) : -1;           // last visible key; -1: padded row
        const bool live = (r & ~31) < a.M;                        // a row of this warp is no padding
        float m = -INFINITY, l = 0.f;
        bool first = true;
        for (; t < j.ntiles; t += step) {
          const uint32_t st = MT == 2 ? 2 * (tt + t) + quad : tt + t;
          if (!full_wait(st)) continue;
          tc_fence_after();
          if (!live) {
            release(st);
            continue;
          }
          const uint32_t tcol = column(st);
          tmem_ld32(tcol, va);
          const int j0 = (j.tile0 + t) * kTileKeys;
          bool redo = true;
          if (j0 + kTileKeys <= j.n) {  // all keys are visible to all rows
            uint64_t acc0 = 0ull, acc1 = 0ull;
            float pmax = -INFINITY;
            tmem_ld_wait(va);
            tmem_ld32(tcol + 32, vb);
            if (first) m = p1_reference(va, a.scale_log2);
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
            if (p1_in_range(cs, pmax, a.scale_log2, m)) {
              l += cs;
              redo = false;
            }
          }
          first = false;
          if (__any_sync(0xffffffffu, redo && lim >= 0)) {
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              tmem_ld32(tcol + 32 * c, vb);
              tmem_ld_wait(vb);
              if (redo) p1_exact(vb, j0 + 32 * c, lim, a.scale_log2, m, l);
            }
          }
          release(st);
        }
        // hand the partial to the publisher warp
        const bool ok = mbar_wait(bar(P::kBarPubEmpty, quad), (p1c & 1) ^ 1, abort_flag, a.dev_status, a.spin_limit);
        if (ok) pub_s[quad * 128 + qtid] = lim >= 0 ? make_float2(m, l) : make_float2(-INFINITY, 0.f);
        __syncwarp();
        if (lane == 0 && ok) mbar_arrive(bar(P::kBarPubFull, quad), 1);
        ++p1c;
      } else {
        // ---- pass 2: this thread's key, summed over all query rows
        const uint32_t slot = p2c % a.lag;
        const bool have_lse = mbar_wait(bar(P::kBarLseFull, slot), (p2c / a.lag) & 1, abort_flag, a.dev_status, a.spin_limit);
        for (; t < j.ntiles; t += step) {
          uint64_t acc0 = 0ull, acc1 = 0ull;
          bool ok = true;
#pragma unroll 1
          for (int mt = 0; mt < MT; ++mt) {  // 128 rows unrolled: 7850 -> 7640 us for eight 16k sequences of 256 rows
            const uint32_t st = (tt + t) * MT + mt;
            const float* nlse = nlse_s + slot * 256 + 128 * mt;
            const uint32_t tcol = column(st);
            if (!(ok = full_wait(st))) break;
            tc_fence_after();
            tmem_ld32(tcol, va);
            const int cols = a.npad - 128 * mt;
            if (cols >= 128) {
              tmem_ld_wait(va);
              tmem_ld32(tcol + 32, vb);
              p2_chunk(va, nlse, sc2, acc0, acc1);
              tmem_ld_wait(vb);
              tmem_ld32(tcol + 64, va);
              p2_chunk(vb, nlse + 32, sc2, acc0, acc1);
              tmem_ld_wait(va);
              tmem_ld32(tcol + 96, vb);
              p2_chunk(va, nlse + 64, sc2, acc0, acc1);
              tmem_ld_wait(vb);
              release(st);
              p2_chunk(vb, nlse + 96, sc2, acc0, acc1);
            } else {
#pragma unroll 1
              for (int c = 0; c < cols; c += 32) {
                tmem_ld_wait(va);
                if (c + 32 >= cols) release(st);
                p2_chunk(va, nlse + c, sc2, acc0, acc1);
                if (c + 32 < cols) tmem_ld32(tcol + c + 32, va);
              }
            }
          }
          const int key = (j.tile0 + t) * kTileKeys + qtid;
          if (ok && key < j.n) a.raw[(size_t)j.u * a.n_stride + key] = sum4(acc0, acc1);
        }
        __syncwarp();
        if (lane == 0 && have_lse) mbar_arrive(bar(P::kBarLseEmpty, slot), 1);
        ++p2c;
      }
      tt += j.ntiles;
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  if (warp == kEpiWarps + 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ---- host side --------------------------------------------------------------------------------

// Clocks of the CTA with the most to do when the items of `groups` groups of heads (heads each, T[g] keys long, at most `it` tiles an
// item) are dealt to `ctas` CTAs in turn: `tile` a tile and kItem an item, and what pass 2 waits for the row log-sum-exps of its head.
// Those come kFold clocks after the head's last partial, and kFoldItem for each of the partials that they are put together from; pass 1
// of the next item (`sweep` clocks a tile) runs meanwhile.
double deal_cost(const int32_t* T, int groups, int heads, int it, int ctas, double tile, double sweep) {
  constexpr double kItem = 1300.0, kFold = 8000.0, kFoldItem = 130.0;
  constexpr int kMaxCtas = 256;
  double step[kMaxCtas + 1] = {};  // what a group's last, incomplete round adds: differences from CTA to CTA
  if (ctas > kMaxCtas) ctas = kMaxCtas;
  double base = 0.0;
  int first = 0;  // the CTA that gets the group's first item
  for (int g = 0; g < groups; ++g) {
    const long long tiles = (T[g] + kTileKeys - 1) / kTileKeys, per_head = (tiles + it - 1) / it, items = heads * per_head;
    const double own = (double)tiles / (double)per_head, fold = kFold + kFoldItem * (double)per_head;
    const double time = own * tile + kItem + std::max(0.0, fold - own * sweep);
    const int rest = (int)(items % ctas);
    base += time * (double)(items / ctas);
    if (rest) {
      step[first] += time;
      if (first + rest <= ctas) {
        step[first + rest] -= time;
      } else {
        step[0] += time;
        step[first + rest - ctas] -= time;
      }
      first = (first + rest) % ctas;
    }
  }
  double run = 0.0, most = 0.0;
  for (int c = 0; c < (groups > 1 ? ctas : 1); ++c) {
    run += step[c];
    if (run > most) most = run;
  }
  return base + most;
}

template <int MT, int NQ, int NH, bool RAGGED = false>
cudaError_t launch_fused(const CUtensorMap& qm, const CUtensorMap& km, FusedArgs args, int spare_sms, LaunchCtx& lc,
                         const int32_t* seq_T_host = nullptr) {
  using P = Plan<MT, NQ, NH>;
  const int smem = P::kTotal;
  auto kern = score_fused_kernel<MT, NQ, NH, RAGGED>;
  cudaError_t e;
  int sms = 0;
  if ((e = allow_smem((const void*)kern, smem)) != cudaSuccess || (e = device_sms(&sms)) != cudaSuccess) return e;
  if (spare_sms > 0 && sms > 8 * spare_sms) sms -= spare_sms;
  // A CTA runs pass 1 of later items before pass 2 of the current one, so a head's items must
  // not outnumber the CTAs (else a CTA would wait for partials that it is due to produce itself).
  if (args.adapt_items) {
    // Larger work items mean fewer job changes and fewer partials to fold per head, but coarser dealing.  A tile takes the time of
    // its arithmetic in both sweeps, or of its way out of HBM where that is longer (128 heads x 157 tiles, head size 64: 223 us of
    // scorer in items of 20 tiles, 231 in 16, 237 in 8; 2048 x 128 tiles of two row blocks 5.84 ms in 64 and 5.94 in 8).  Pass 1
    // takes a row block's time however few of its rows there are, pass 2 what its columns take.  Large items do not leave pass 2 its
    // key tiles in L2: items of up to eight tiles do, whose two sweeps' keys fit (256 heads x 256 tiles of 128 rows: 1163 us a call
    // in 64 tiles, 1172 in 32, 1176 in 12, 1143 in 10, 1129 in 8 and 9; of 64 rows 982 in 64, 980 in 32, 977 in 16, 941 in 9, 926
    // in 8); some of a cache not much larger than L2 is there in any case (32 heads x 256 tiles 181 us in 8, 174 in 29).  But a head
    // of many items has its row log-sum-exps late (8 heads x 938 tiles: 187 us a call in 53 tiles, 218 in 9).  Any number of tiles up
    // to 64 is tried: 8 heads x 64 tiles 33 us a call with 4, 37 with 6 or 8.
    constexpr double kBlock = 1290.0, kRead = 760.0 * NH;
    constexpr long long kL2Tiles = (80ll << 20) / (NH * kHalfBytes);
    const double clocks = kBlock * (MT + args.npad / 128.0);
    long long all_tiles = 0;
    for (int q = 0; q < (RAGGED ? args.n_seq : 1); ++q)
      all_tiles += (long long)(RAGGED ? args.heads_per_seq : args.nheads) * (((RAGGED ? seq_T_host[q] : args.T) + kTileKeys - 1) / kTileKeys);
    int best = args.item_tiles;
    double best_cost = 1e30;
    for (int it = args.item_tiles; it <= 64; ++it) {
      const bool twice = all_tiles > kL2Tiles && 2ll * sms * it > kL2Tiles;  // K comes out of HBM twice
      const double tile = std::max(clocks, (twice ? 2.0 - (double)kL2Tiles / (double)all_tiles : 1.0) * kRead);
      const double cost = RAGGED ? deal_cost(seq_T_host, args.n_seq, args.heads_per_seq, it, sms, tile, kBlock * MT)
                                 : deal_cost(&args.T, 1, args.nheads, it, sms, tile, kBlock * MT);
      if (cost < best_cost * 0.995) {
        best_cost = cost;
        best = it;
      }
    }
    args.item_tiles = best;
  }
  while ((args.tiles_T + args.item_tiles - 1) / args.item_tiles > sms) ++args.item_tiles;
  args.items_per_head = (args.tiles_T + args.item_tiles - 1) / args.item_tiles;
  args.iph_magic = div_magic(args.items_per_head);
  int total_items = args.nheads * args.items_per_head;
  if (RAGGED) {
    int base = 0;
    for (int q = 0; q < args.n_seq; ++q) {
      args.seq_T[q] = seq_T_host[q];
      args.seq_item0[q] = base;
      const int tiles = (seq_T_host[q] + kTileKeys - 1) / kTileKeys;
      args.seq_iph[q] = (tiles + args.item_tiles - 1) / args.item_tiles;
      args.seq_magic[q] = div_magic(args.seq_iph[q]);
      base += args.heads_per_seq * args.seq_iph[q];
    }
    total_items = base;
  }
  args.total_items = total_items;
  const int grid = total_items < sms ? total_items : sms;  // one CTA per SM: each owns the SM's tensor memory
  void* params[] = {(void*)&qm, (void*)&km, (void*)&args};
  // cooperative launch: the CTAs of a head wait for one another, so all must be resident (one per SM: the launch fails if
  // they cannot be)
  e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(P::kThreads), params, (size_t)smem,
                                  lc.st);
  lc.mark("score_fused");
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Offset of the (lse, tag) rows inside the zero-initialised block that starts with the [heads] counters and the status.
size_t score_tc_lse_offset(const Dims& dm) { return (((size_t)dm.heads() + 1) * sizeof(int) + 255) & ~(size_t)255; }

// Test hooks of the tensor-core scorers, read from the environment at every call: LUKV_TEST_SPIN_LIMIT shortens
// the limit of every device-side wait, LUKV_TEST_DROP_ITEM names one work item whose partial results never
// reach the other CTAs -- together they make a bounded wait run out without faulting anything.
void score_test_hooks(uint32_t* spin_limit, int* drop_item) {
  const char* lim = getenv("LUKV_TEST_SPIN_LIMIT");
  const char* drop = getenv("LUKV_TEST_DROP_ITEM");
  const long l = lim ? atol(lim) : 0, d = drop ? atol(drop) : -1;
  *spin_limit = (l >= 1 && l <= (1L << 30)) ? (uint32_t)l : kSpinLimit;
  *drop_item = (drop && d >= 0 && d <= (1L << 30)) ? (int)d : -1;
}

// Fewest key tiles per work item the launcher tries (it grows for very long contexts): eight, or two where items of eight
// are fewer than two per SM.  The 148 is the chip this library is built for: the workspace depends on it.
// LUKV_ITEM_TILES (1..64) overrides it for tuning runs.
static int forced_item_tiles() {
  static const int v = env_int("LUKV_ITEM_TILES", 1, 64, 0);
  return v;
}
static size_t tiles_of(const Dims& dm) { return ((size_t)dm.T + kTileKeys - 1) / kTileKeys; }
bool score_tc_small(const Dims& dm) {
  return !forced_item_tiles() && (size_t)dm.heads() * ((tiles_of(dm) + 7) / 8) < 2 * 148;
}
int score_item_tiles(const Dims& dm) { return forced_item_tiles() ? forced_item_tiles() : score_tc_small(dm) ? 2 : 8; }
// Bytes of pass-1 partials the tensor-core scorer may write for these sizes, in items of eight tiles and in a small call's of
// two.  The latter stay at the largest small call's where small calls end: a call must not need less than a smaller one.
size_t score_tc_stats_bytes(const Dims& dm) {
  const size_t least = forced_item_tiles() ? forced_item_tiles() : 8;
  return (size_t)dm.heads() * ((tiles_of(dm) + least - 1) / least) * 256 * sizeof(float);
}
size_t score_tc_small_stats_bytes(const Dims& dm) {
  if (forced_item_tiles()) return 0;
  const size_t items = (size_t)dm.heads() * ((tiles_of(dm) + 1) / 2), most = 4 * (2 * 148 - 1);  // a small call's items of two
  return (items < most ? items : most) * 256 * sizeof(float);
}
// Bytes of the block that must be zero at launch: [heads] counters, the status word, then [heads][lse_rows][2] floats.
size_t score_tc_flag_bytes(const Dims& dm) {
  // the single-sweep kernel strides the rows of a head by 128 or 256, the two-sweep kernel by M rounded up to 4
  return score_tc_lse_offset(dm) + (size_t)dm.heads() * ((dm.M + 127) & ~127) * 2 * sizeof(float);
}

bool score_tc_supported(const Dims& dm) {
  return dm.dtype == LUKV_DTYPE_BF16 && encode_fn() != nullptr;
}

cudaError_t launch_score_tc(const Dims& dm, const void* q, const void* k, const Workspace& ws, int spare_sms, LaunchCtx& lc) {
  // The two-sweep kernel below is the default.  LUKV_SCORER=onesweep selects the single-sweep kernel where the
  // shape allows it (it parks a head's exponentials in tensor memory and is bound by the latency of the
  // log-sum-exp exchange between CTAs; at long contexts the two sweeps are faster).
  const char* which = getenv("LUKV_SCORER");
  if (which && which[0] == 'o' && !dm.seq_T && score_onepass_eligible(dm)) {
    const cudaError_t e1 = launch_score_onepass(dm, q, k, ws, spare_sms, lc);
    if (e1 != cudaErrorNotSupported) return e1;
  }
  CUtensorMap qm, km;
  if (!make_map(&qm, q, (uint64_t)dm.heads() * dm.M, dm.d) || !make_map(&km, k, (uint64_t)dm.heads() * dm.T, dm.d))
    return cudaErrorInvalidValue;
  FusedArgs args;
  args.stats = ws.tc_stats;
  args.lse = reinterpret_cast<float*>(reinterpret_cast<char*>(ws.head_flags) + score_tc_lse_offset(dm));
  args.raw = ws.raw;
  args.head_cnt = ws.head_flags;
  args.dev_status = score_tc_status(dm, ws);
  args.M = dm.M;
  args.T = dm.T;
  args.w = dm.w;
  args.n = dm.n;
  args.T_stride = dm.T;
  args.n_stride = dm.raw_stride();
  args.n_seq = dm.S;
  args.heads_per_seq = dm.N;
  args.lse_rows = (dm.M + 3) & ~3;
  args.nheads = (int)dm.heads();
  args.tiles_T = (dm.T + kTileKeys - 1) / kTileKeys;
  args.item_tiles = score_item_tiles(dm);
  args.adapt_items = getenv("LUKV_ITEM_TILES") ? 0 : 1;
  args.tiles_n = (dm.n + kTileKeys - 1) / kTileKeys;
  args.items_per_head = 0;  // set by the launcher
  args.npad = (dm.M + 31) & ~31;
  static const int hints = env_int("LUKV_L2_HINTS", 0, 1, 1);
  args.l2_hints = hints;
  static const int lag = env_int("LUKV_LAG", 2, kMaxLag, 2);
  args.lag = lag;
  args.scale_log2 = dm.scale_log2;
  score_test_hooks(&args.spin_limit, &args.drop_item);
  // the per-head counters and the (value, tag) rows must start at zero; they are adjacent in the workspace
  const cudaError_t e = cudaMemsetAsync(ws.head_flags, 0, score_tc_flag_bytes(dm), lc.st);
  if (e != cudaSuccess) return e;
  if (dm.seq_T) {
    // sequences of different lengths: work items dealt per sequence
    if (dm.S > kMaxRaggedSeqs) return cudaErrorInvalidValue;
    if (dm.d == 64)
      return dm.M > 128 ? launch_fused<2, 2, 1, true>(qm, km, args, spare_sms, lc, dm.seq_T)
                        : launch_fused<1, 2, 1, true>(qm, km, args, spare_sms, lc, dm.seq_T);
    return dm.M > 128 ? launch_fused<2, 2, 2, true>(qm, km, args, spare_sms, lc, dm.seq_T)
                      : launch_fused<1, 2, 2, true>(qm, km, args, spare_sms, lc, dm.seq_T);
  }
  if (dm.d == 64)
    return dm.M > 128 ? launch_fused<2, 2, 1>(qm, km, args, spare_sms, lc) : launch_fused<1, 2, 1>(qm, km, args, spare_sms, lc);
  if (dm.M > 128) return launch_fused<2, 2, 2>(qm, km, args, spare_sms, lc);
  static const int quads = env_int("LUKV_QUADS", 2, 3, 2);
  if (quads == 3) return launch_fused<1, 3, 2>(qm, km, args, spare_sms, lc);
  return launch_fused<1, 2, 2>(qm, km, args, spare_sms, lc);
}

}  // namespace lukv
