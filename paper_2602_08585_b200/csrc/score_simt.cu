// Stage (a), general-shape scorer on the FP32 pipes (any dtype, d in {64,128}, up to 256
// score rows per head).  Two sweeps over the keys of a head:
//   sweep 1  logits of the window queries against a chunk of keys -> per-chunk row
//            (max, sum-exp) partials
//   sweep 2  the partials folded into the row log-sum-exps (by every CTA for its head), the same
//            logits again -> probabilities -> column sums over the w window rows and the G query
//            heads (the "accumulated attention" of the proxy)
// The 1-D max-pool follows, in a kernel of its own here or in the selection.  Attention weights are Eq. 1
// (Sec. 3.1) of the paper.  Logits are kept in the exp2 domain: x2 = <q,k> * scale * log2(e).
#include "simt_tile.cuh"

namespace lukv {
namespace {

constexpr int kThreads = kSimtThreads;
constexpr int kKeyTile = 64;     // keys per shared-memory tile
constexpr int kMaxChunkTiles = 16;  // tiles per CTA

// Tiles per CTA: up to 16 (the query rows are loaded once per CTA), fewer where that would leave SMs without one; 4 heads of
// 1024 keys took 37 us a sweep in 4 CTAs, 4.5 us in 64.
int chunk_tiles(const Dims& dm) {
  const long long tiles = dm.heads() * ((dm.T + kKeyTile - 1) / kKeyTile);
  const long long per = tiles / (4 * 148);
  return per < 1 ? 1 : per > kMaxChunkTiles ? kMaxChunkTiles : (int)per;
}

// Merges the (reference, sum-exp) pairs of the 16 lanes that differ in their low four bits.
__device__ __forceinline__ void fold16(float& m, float& l) {
#pragma unroll
  for (int off = 1; off < 16; off <<= 1) {
    const float mo = __shfl_xor_sync(0xffffffffu, m, off);
    const float lo = __shfl_xor_sync(0xffffffffu, l, off);
    const float mn = fmaxf(m, mo);
    if (mn > -INFINITY) {
      l = l * exp2f(m - mn) + lo * exp2f(mo - mn);
      m = mn;
    }
  }
}

// One CTA: all M rows of head u against keys [chunk*chunk_keys, +chunk_keys).
// Thread layout: kg = tid%16 owns keys {kg, kg+16, kg+32, kg+48} of a tile, rg = tid/16 owns
// rows {rg, rg+16, ...}.
template <typename TIn, int D, int RPT, bool SWEEP2>
__global__ void __launch_bounds__(kThreads) score_simt_kernel(const TIn* __restrict__ q, const TIn* __restrict__ k,
                                                              float* __restrict__ stats, float* __restrict__ raw,
                                                              int n_stride, int M, int T, int w, int chunks, int chunk_keys,
                                                              float scale_log2, SeqLens sl, int heads_per_seq) {
  constexpr int kPitch = D + 4;
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;                         // [16*RPT][kPitch]
  float* Ks = smem + 16 * RPT * kPitch;     // [kKeyTile][kPitch]
  __shared__ float colred[kThreads / 32][kKeyTile];

  const int u = blockIdx.x / chunks, chunk = blockIdx.x % chunks;
  // T is the row stride of the cache (the longest sequence); Tu the length of this head's sequence
  const int Tu = heads_per_seq > 0 ? sl.T[u / heads_per_seq] : T;
  const int n = Tu - w;
  const int tid = threadIdx.x, kg = tid & 15, rg = tid >> 4;
  const TIn* qh = q + (size_t)u * M * D;
  const TIn* kh = k + (size_t)u * T * D;

  pdl_launch_dependents();
  load_rows_f32<TIn, D>(Qs, qh, 16 * RPT, M);
  if (SWEEP2) pdl_wait();  // the partials are the first sweep's

  float row_m[RPT], row_l[RPT], row_lse[RPT];
  int row_lim[RPT];  // last visible key of the row
#pragma unroll
  for (int a = 0; a < RPT; ++a) {
    const int r = rg + 16 * a;
    row_m[a] = -INFINITY;
    row_l[a] = 0.f;
    row_lim[a] = r < M ? n + (r % w) : -1;
    row_lse[a] = 0.f;
    if (SWEEP2) {
      // the 16 threads of a row group fold the chunks' partials: m + log2(l)
      float m = -INFINITY, l = 0.f;
      for (int c = kg; c < chunks && r < M; c += 16) {
        const float2 s = *reinterpret_cast<const float2*>(stats + (((size_t)u * chunks + c) * M + r) * 2);
        const float mn = fmaxf(m, s.x);
        if (mn > -INFINITY) {
          l = l * exp2f(m - mn) + s.y * exp2f(s.x - mn);
          m = mn;
        }
      }
      fold16(m, l);
      row_lse[a] = m + log2f(l);
    }
  }

  const int key_begin = chunk * chunk_keys;
  const int key_end = min(Tu, key_begin + chunk_keys);
  for (int j0 = key_begin; j0 < key_end; j0 += kKeyTile) {
    __syncthreads();  // previous tile fully consumed (and Qs visible on the first pass)
    load_rows_f32<TIn, D>(Ks, kh + (size_t)j0 * D, kKeyTile, min(kKeyTile, Tu - j0));
    __syncthreads();

    float acc[RPT][4];
#pragma unroll
    for (int a = 0; a < RPT; ++a)
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) acc[a][kk] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      float4 kv[4];
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) kv[kk] = *reinterpret_cast<const float4*>(Ks + (kg + 16 * kk) * kPitch + c);
#pragma unroll
      for (int a = 0; a < RPT; ++a) {
        const float4 qv = *reinterpret_cast<const float4*>(Qs + (rg + 16 * a) * kPitch + c);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          acc[a][kk] = fmaf(qv.x, kv[kk].x, acc[a][kk]);
          acc[a][kk] = fmaf(qv.y, kv[kk].y, acc[a][kk]);
          acc[a][kk] = fmaf(qv.z, kv[kk].z, acc[a][kk]);
          acc[a][kk] = fmaf(qv.w, kv[kk].w, acc[a][kk]);
        }
      }
    }

    if (!SWEEP2) {
#pragma unroll
      for (int a = 0; a < RPT; ++a) {
        float x[4], tmax = -INFINITY;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int j = j0 + kg + 16 * kk;
          x[kk] = (j <= row_lim[a]) ? acc[a][kk] * scale_log2 : -INFINITY;
          tmax = fmaxf(tmax, x[kk]);
        }
        if (tmax > -INFINITY) {
          const float mn = fmaxf(row_m[a], tmax);
          float l = row_l[a] * exp2f(row_m[a] - mn);  // exp2f(-inf) = 0 on the first update
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) l += exp2f(x[kk] - mn);
          row_m[a] = mn;
          row_l[a] = l;
        }
      }
    } else {
      float cs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int a = 0; a < RPT; ++a)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int j = j0 + kg + 16 * kk;
          if (j <= row_lim[a]) cs[kk] += exp2f(fmaf(acc[a][kk], scale_log2, -row_lse[a]));
        }
      // lanes l and l^16 hold the two row groups of this warp
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) cs[kk] += __shfl_xor_sync(0xffffffffu, cs[kk], 16);
      const int warp = tid >> 5;
      if ((tid & 16) == 0)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) colred[warp][kg + 16 * kk] = cs[kk];
      __syncthreads();
      if (tid < kKeyTile) {
        float s = 0.f;
#pragma unroll
        for (int wv = 0; wv < kThreads / 32; ++wv) s += colred[wv][tid];
        const int j = j0 + tid;
        if (j < n) raw[(size_t)u * n_stride + j] = s;
      }
    }
  }

  if (!SWEEP2) {
    // fold the 16 key groups of each row (lanes differing in their low 4 bits)
#pragma unroll
    for (int a = 0; a < RPT; ++a) {
      float m = row_m[a], l = row_l[a];
      fold16(m, l);
      const int r = rg + 16 * a;
      if (kg == 0 && r < M) {
        float* o = stats + (((size_t)u * chunks + chunk) * M + r) * 2;
        o[0] = m;
        o[1] = l;
      }
    }
    pdl_wait();  // an allocation kernel that runs beside this sweep ends before it
  }
}

// The general form (windows of more than nine positions): a thread per output.
// n: rankable positions (of the longest sequence); the head's own length comes from `sl` when the
// sequences differ (heads_per_seq > 0).
__global__ void max_pool_kernel(const float* __restrict__ raw, float* __restrict__ pooled, int raw_stride, int stride, int n,
                                int half, int tiles, SeqLens sl, int heads_per_seq, int w) {
  const int u = blockIdx.x / tiles;
  const int j = (blockIdx.x % tiles) * blockDim.x + threadIdx.x;
  if (heads_per_seq > 0) n = sl.T[u / heads_per_seq] - w;
  if (j >= n) return;
  const float* r = raw + (size_t)u * raw_stride;
  const int lo = max(0, j - half), hi = min(n - 1, j + half);
  float best = r[lo];
  for (int t = lo + 1; t <= hi; ++t) best = fmaxf(best, r[t]);
  pooled[(size_t)u * stride + j] = best;
}

// Windows of at most nine positions: four outputs per thread from three 16-byte loads (the rows of the un-pooled scores are
// padded to 16 bytes): the outputs 4t..4t+3 need the inputs 4t-4..4t+7.  Positions outside [0,n) count as -inf (the window
// is clipped at the ends).
__global__ void max_pool4_kernel(const float4* __restrict__ raw, float* __restrict__ pooled, int raw_quads, int stride, int n,
                                 int half, int tiles, SeqLens sl, int heads_per_seq, int w) {
  const int u = blockIdx.x / tiles;
  const int t = (blockIdx.x % tiles) * blockDim.x + threadIdx.x;
  if (heads_per_seq > 0) n = sl.T[u / heads_per_seq] - w;
  if (4 * t >= n) return;
  const float4* r = raw + (size_t)u * raw_quads;
  float x[12];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float4 v = r[min(max(t + q - 1, 0), raw_quads - 1)];
    x[4 * q] = v.x, x[4 * q + 1] = v.y, x[4 * q + 2] = v.z, x[4 * q + 3] = v.w;
  }
#pragma unroll
  for (int i = 0; i < 12; ++i)
    if ((unsigned)(4 * t - 4 + i) >= (unsigned)n) x[i] = -INFINITY;
  float y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float best = x[4 + i];
#pragma unroll
    for (int d = 1; d <= 4; ++d)
      if (d <= half) best = fmaxf(best, fmaxf(x[4 + i - d], x[4 + i + d]));
    y[i] = best;
  }
  float* out = pooled + (size_t)u * stride + 4 * t;
  if (stride % 4 == 0 && 4 * t + 3 < n && (reinterpret_cast<uintptr_t>(pooled) & 15u) == 0) {
    *reinterpret_cast<float4*>(out) = make_float4(y[0], y[1], y[2], y[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * t + i < n) out[i] = y[i];
  }
}

template <typename TIn, int D, int RPT>
cudaError_t launch_sweeps(const Dims& dm, const void* q, const void* k, const Workspace& ws, bool overlap, LaunchCtx& lc) {
  const int chunks = score_chunks(dm), chunk_keys = chunk_tiles(dm) * kKeyTile;
  const size_t smem = (size_t)(16 * RPT + kKeyTile) * (D + 4) * sizeof(float);
  auto k1 = score_simt_kernel<TIn, D, RPT, false>;
  auto k2 = score_simt_kernel<TIn, D, RPT, true>;
  cudaError_t e;
  if ((e = allow_smem((const void*)k1, smem)) != cudaSuccess || (e = allow_smem((const void*)k2, smem)) != cudaSuccess)
    return e;
  const dim3 grid((unsigned)(dm.heads() * chunks));
  SeqLens sl = {};
  const int heads_per_seq = dm.seq_T ? dm.N : 0;
  if (dm.seq_T)
    for (int s = 0; s < dm.S; ++s) sl.T[s] = dm.seq_T[s];
  if ((e = launch_pdl(k1, grid, dim3(kThreads), smem, lc.st, overlap, (const TIn*)q, (const TIn*)k, ws.stats, (float*)nullptr,
                      dm.raw_stride(), dm.M, dm.T, dm.w, chunks, chunk_keys, dm.scale_log2, sl, heads_per_seq)) != cudaSuccess)
    return e;
  lc.mark("score_simt_sweep1");
  if ((e = launch_pdl(k2, grid, dim3(kThreads), smem, lc.st, true, (const TIn*)q, (const TIn*)k, ws.stats, ws.raw,
                      dm.raw_stride(), dm.M, dm.T, dm.w, chunks, chunk_keys, dm.scale_log2, sl, heads_per_seq)) != cudaSuccess)
    return e;
  lc.mark("score_simt_sweep2");
  return cudaGetLastError();
}

template <typename TIn, int D>
cudaError_t dispatch_rows(const Dims& dm, const void* q, const void* k, const Workspace& ws, bool overlap, LaunchCtx& lc) {
  const int rpt = (dm.M + 15) / 16;
  if (rpt <= 1) return launch_sweeps<TIn, D, 1>(dm, q, k, ws, overlap, lc);
  if (rpt <= 2) return launch_sweeps<TIn, D, 2>(dm, q, k, ws, overlap, lc);
  if (rpt <= 4) return launch_sweeps<TIn, D, 4>(dm, q, k, ws, overlap, lc);
  if (rpt <= 8) return launch_sweeps<TIn, D, 8>(dm, q, k, ws, overlap, lc);
  return launch_sweeps<TIn, D, 16>(dm, q, k, ws, overlap, lc);
}

}  // namespace

int score_chunks(const Dims& dm) {
  const int keys = chunk_tiles(dm) * kKeyTile;
  return (dm.T + keys - 1) / keys;
}

cudaError_t launch_score_simt(const Dims& dm, const void* q, const void* k, const Workspace& ws, bool overlap,
                              LaunchCtx& lc) {
  if (dm.dtype == LUKV_DTYPE_BF16) {
    if (dm.d == 64) return dispatch_rows<__nv_bfloat16, 64>(dm, q, k, ws, overlap, lc);
    return dispatch_rows<__nv_bfloat16, 128>(dm, q, k, ws, overlap, lc);
  }
  if (dm.d == 64) return dispatch_rows<float, 64>(dm, q, k, ws, overlap, lc);
  return dispatch_rows<float, 128>(dm, q, k, ws, overlap, lc);
}

cudaError_t launch_pool(const Dims& dm, const float* raw, float* pooled, int stride, LaunchCtx& lc) {
  const int half = dm.kp / 2, hps = dm.seq_T ? dm.N : 0;
  SeqLens sl = {};
  if (dm.seq_T)
    for (int q = 0; q < dm.S; ++q) sl.T[q] = dm.seq_T[q];
  if (half <= 4) {
    const int quads = dm.raw_stride() / 4, tiles = (quads + 255) / 256;
    max_pool4_kernel<<<(unsigned)(dm.heads() * tiles), 256, 0, lc.st>>>(reinterpret_cast<const float4*>(raw), pooled, quads,
                                                                       stride, dm.n, half, tiles, sl, hps, dm.w);
  } else {
    const int tiles = (dm.n + 255) / 256;
    max_pool_kernel<<<(unsigned)(dm.heads() * tiles), 256, 0, lc.st>>>(raw, pooled, dm.raw_stride(), stride, dm.n, half,
                                                                      tiles, sl, hps, dm.w);
  }
  lc.mark("max_pool");
  return cudaGetLastError();
}

}  // namespace lukv
