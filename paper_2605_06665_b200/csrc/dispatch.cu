// Token permute into expert-contiguous order and its inverse (combine), forward
// and backward.  All data movement is in 16-byte vectors; one warp moves one row.
#include <atomic>

#include "common.cuh"

namespace unipool {

// ---------------------------------------------------------------- maps
// Chunk c holds tokens [c*CH, (c+1)*CH); a block of the placing kernel owns one chunk, warp w of it the
// tokens [w*CH/8, (w+1)*CH/8) of those: the stable (token-major) order is chunk order, then warp order,
// then lane order inside a warp.
constexpr int kDispatchWarps = 8;
constexpr int kHistWarps = kDispatchSuperChunks;   // a block of the histogram kernel counts this many chunks, a warp each
static_assert(kHistWarps == 16, "a group's counts of one expert are two 16-byte stores");

// Where the histogram kernel leaves its counts (S = groups of 16 chunks):
//   pre16 [S][M][16]  assignments to the expert in the chunks of the group before the chunk
//                     (at most 15 * 256 * 8: 16 bits)
//   super [M][S]      assignments to the expert in the whole group
// so that a block of the placing kernel sums S + 1 numbers per expert instead of one per chunk: the
// placing kernel went from 34 to 29 us at 16384 tokens, k = 2, 96 experts and from 81 to 62 us at k = 8,
// 384 experts, where every block had read 98 / 393 KB of counts.
struct ChunkCounts { uint16_t* pre16; int32_t* super; int n_chunks, n_super; };

static ChunkCounts chunk_counts(void* base, int n_chunks, int M) {
  ChunkCounts c;
  c.n_chunks = n_chunks;
  c.n_super = (n_chunks + kDispatchSuperChunks - 1) / kDispatchSuperChunks;
  c.pre16 = static_cast<uint16_t*>(base);
  c.super = reinterpret_cast<int32_t*>(c.pre16 + (int64_t)c.n_super * M * kDispatchSuperChunks);
  return c;
}

// An expert index outside [0, M) is a corrupt routing entry: recorded in `status` (may be NULL), dropped.
__device__ __forceinline__ bool routed(int e, int M, int32_t* status) {
  if (e >= 0 && e < M) return true;
  if (status != nullptr && atomicCAS(status, 0, kStatusCheck) == 0) { status[1] = 10; status[2] = e; }
  return false;
}

__global__ void __launch_bounds__(kHistWarps * 32)
dispatch_hist_kernel(const int32_t* __restrict__ idx, int T, int k, int M, int chunk, ChunkCounts cc,
                     int32_t* __restrict__ status) {
  grid_wait(idx);
  extern __shared__ int hist[];                      // [kHistWarps][M]
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int i = threadIdx.x; i < kHistWarps * M; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  const int c = (int)blockIdx.x * kHistWarps + warp;
  const int64_t total = (int64_t)T * k;
  const int64_t a_begin = min(total, (int64_t)c * chunk * k), a_end = min(total, a_begin + (int64_t)chunk * k);
  // few blocks (one per 16 chunks), so each lane keeps kAhead indices in flight
  constexpr int kAhead = 8;
  for (int64_t a0 = a_begin + lane; a0 < a_end; a0 += 32 * kAhead) {
    int e[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) e[q] = a0 + 32 * q < a_end ? __ldg(idx + a0 + 32 * q) : 0;
#pragma unroll
    for (int q = 0; q < kAhead; ++q)
      if (a0 + 32 * q < a_end && routed(e[q], M, status)) atomicAdd(&hist[warp * M + e[q]], 1);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < M; e += blockDim.x) {
    int run = 0;
    uint32_t pre[kHistWarps / 2];
#pragma unroll
    for (int w = 0; w < kHistWarps; ++w) {
      pre[w / 2] = (w & 1) ? pre[w / 2] | ((uint32_t)run << 16) : (uint32_t)run;
      run += hist[w * M + e];
    }
    uint4* out = reinterpret_cast<uint4*>(cc.pre16 + ((int64_t)blockIdx.x * M + e) * kHistWarps);
    out[0] = make_uint4(pre[0], pre[1], pre[2], pre[3]);
    out[1] = make_uint4(pre[4], pre[5], pre[6], pre[7]);
    cc.super[(int64_t)e * cc.n_super + blockIdx.x] = run;
  }
}

// Second (and last) kernel of the permute.  Block b owns the tokens of chunk b.  From the histograms of
// the first kernel every block derives, for itself, the padded group starts (sums over all chunks,
// exclusive scan over the experts) and the rows its own chunk starts at (sums over the chunks before
// it); it then ranks its assignments (block, warp, lane order = token order, so the permutation is
// stable), writes row_of / token_of and moves its tokens: a token's row is read once and written to each
// of its k rows.  All blocks share the bookkeeping: pad rows (token_of = -1, zeros in Xp), the
// tile -> expert table, the rows behind the last group.  Blocks behind the last chunk do only that.
// Small batches (cc.n_super == 0): no histogram kernel, every block counts all T*k indices itself.
constexpr int kPlaceTokens = 8;          // tokens a warp has in flight while moving rows
constexpr int kVpl = 3;                  // 16-byte vectors per lane and pass of the row movers
constexpr int kPlaceExperts = 4;         // experts whose counts a warp sums at a time: independent loads

__global__ void __launch_bounds__(kDispatchWarps * 32)
dispatch_place_kernel(const int32_t* __restrict__ idx, int T, int k, int M, int chunk, ChunkCounts cc,
                      int32_t* __restrict__ status, const uint4* __restrict__ x,
                      int row_vecs, int row_capacity, int32_t* __restrict__ offsets,
                      int32_t* __restrict__ row_of, int32_t* __restrict__ token_of,
                      int32_t* __restrict__ tile_expert, int32_t* __restrict__ group_rows, uint4* __restrict__ Xp) {
  grid_wait(idx, x);
  extern __shared__ int sm[];
  int* hist = sm;                                   // [8][M] per-warp histograms, then per-warp next rows
  int* start = hist + kDispatchWarps * M;           // [M + 1] group starts
  int* total = start + M + 1;                       // [M] assignments per expert, all chunks
  int* before = total + M;                          // [M] assignments per expert in the chunks before this one
  int* rows_s = before + M;                         // [chunk * k] row of each assignment of this chunk
  __shared__ int warp_sum[kDispatchWarps];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int me = (int)blockIdx.x;
  const int64_t n_assign = (int64_t)T * k;
  const int64_t chunk_a0 = min(n_assign, (int64_t)me * chunk * k);
  const int n_tok = (int)min((int64_t)chunk, max((int64_t)0, (int64_t)T - (int64_t)me * chunk));
  const int warp_tokens = chunk / kDispatchWarps;
  const int64_t a_begin = min(n_assign, ((int64_t)me * chunk + (int64_t)warp * warp_tokens) * k);
  const int64_t a_end = min(n_assign, a_begin + (int64_t)warp_tokens * k);

  for (int i = threadIdx.x; i < kDispatchWarps * M; i += blockDim.x) hist[i] = 0;
  // (a) per expert: assignments in all chunks, and in the chunks before this block's
  if (cc.n_super > 0) {
    const int my_super = me / kDispatchSuperChunks;
    for (int e0 = warp * kPlaceExperts; e0 < M; e0 += kDispatchWarps * kPlaceExperts) {
      int tot[kPlaceExperts], bef[kPlaceExperts];
#pragma unroll
      for (int q = 0; q < kPlaceExperts; ++q) {
        const int e = e0 + q;
        tot[q] = 0;
        bef[q] = (e < M && lane == 0 && me < cc.n_chunks)
                     ? (int)cc.pre16[((int64_t)my_super * M + e) * kDispatchSuperChunks + me % kDispatchSuperChunks] : 0;
      }
      for (int b = lane; b < cc.n_super; b += 32) {
#pragma unroll
        for (int q = 0; q < kPlaceExperts; ++q) {
          const int v = e0 + q < M ? cc.super[(int64_t)(e0 + q) * cc.n_super + b] : 0;
          tot[q] += v;
          bef[q] += b < my_super ? v : 0;
        }
      }
#pragma unroll
      for (int q = 0; q < kPlaceExperts; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          tot[q] += __shfl_xor_sync(0xffffffffu, tot[q], o);
          bef[q] += __shfl_xor_sync(0xffffffffu, bef[q], o);
        }
        if (lane == 0 && e0 + q < M) { total[e0 + q] = tot[q]; before[e0 + q] = bef[q]; }
      }
    }
  } else {
    for (int i = threadIdx.x; i < 2 * M; i += blockDim.x) total[i] = 0;       // total and before
    __syncthreads();
    for (int64_t a = threadIdx.x; a < n_assign; a += blockDim.x) {
      const int e = __ldg(idx + a);
      if (!routed(e, M, me == 0 ? status : nullptr)) continue;
      atomicAdd(&total[e], 1);
      if (a < chunk_a0) atomicAdd(&before[e], 1);
    }
  }
  __syncthreads();
  // (b) exclusive scan of the padded totals: a thread takes a run of experts, warps and the block scan the runs
  {
    const int per = (M + (int)blockDim.x - 1) / (int)blockDim.x;
    const int e0 = threadIdx.x * per;
    int mine = 0;
    for (int i = 0; i < per; ++i)
      if (e0 + i < M) mine += (total[e0 + i] + UNIPOOL_ROW_ALIGN - 1) / UNIPOOL_ROW_ALIGN * UNIPOOL_ROW_ALIGN;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int base = 0;
    for (int w = 0; w < warp; ++w) base += warp_sum[w];
    int run = base + incl - mine;
    for (int i = 0; i < per; ++i)
      if (e0 + i < M) {
        start[e0 + i] = run;
        run += (total[e0 + i] + UNIPOOL_ROW_ALIGN - 1) / UNIPOOL_ROW_ALIGN * UNIPOOL_ROW_ALIGN;
      }
    if (threadIdx.x == blockDim.x - 1) start[M] = run;   // the last thread's run ends the last group
  }
  __syncthreads();
  // (c) this chunk's per-warp histograms -> first row of every warp per expert
  if (n_tok > 0) {
    for (int64_t a = a_begin + lane; a < a_end; a += 32) {
      const int e = __ldg(idx + a);
      if (e >= 0 && e < M) atomicAdd(&hist[warp * M + e], 1);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < M; e += blockDim.x) {
      int run = start[e] + before[e];
#pragma unroll
      for (int w = 0; w < kDispatchWarps; ++w) {
        const int n = hist[w * M + e];
        hist[w * M + e] = run;
        run += n;
      }
    }
    __syncthreads();
    // (d) ranks: every warp walks its assignments in lane order
    int* next_row = hist + warp * M;
    for (int64_t a0 = a_begin; a0 < a_end; a0 += 32) {
      const int64_t a = a0 + lane;
      const bool live = a < a_end;
      int e = live ? __ldg(idx + a) : -1;
      const bool ok = live && e >= 0 && e < M;
      if (!ok) e = -1 - lane;                                  // unique key: matches nobody
      const unsigned peers = __match_any_sync(0xffffffffu, e);
      const int rank = __popc(peers & ((1u << lane) - 1u));
      int row = -1;
      if (ok) row = next_row[e] + rank;
      __syncwarp();
      if (ok && rank == 0) next_row[e] += __popc(peers);       // leader = lowest lane of the peer set
      __syncwarp();
      if (live) { row_of[a] = row; rows_s[a - chunk_a0] = row; }
      if (ok) token_of[row] = (int)((uint32_t)a / (uint32_t)k);   // T * k < 2^30
    }
    __syncwarp();
    // (e) every warp moves its own tokens, kPlaceTokens rows of x in flight
    const int t0 = me * chunk;
    const int w_begin = warp * warp_tokens, w_end = min(n_tok, w_begin + warp_tokens);
    for (int v0 = lane; v0 < row_vecs; v0 += 32 * kVpl) {
      for (int tt = w_begin; tt < w_end; tt += kPlaceTokens) {
        uint4 buf[kPlaceTokens][kVpl];
#pragma unroll
        for (int q = 0; q < kPlaceTokens; ++q)
#pragma unroll
          for (int i = 0; i < kVpl; ++i) {
            const int v = v0 + 32 * i;
            buf[q][i] = (tt + q < w_end && v < row_vecs) ? __ldg(x + (int64_t)(t0 + tt + q) * row_vecs + v)
                                                         : make_uint4(0, 0, 0, 0);
          }
#pragma unroll
        for (int q = 0; q < kPlaceTokens; ++q) {
          if (tt + q >= w_end) break;
          for (int j = 0; j < k; ++j) {
            const int row = rows_s[(tt + q) * k + j];
            if (row < 0) continue;
            uint4* dst = Xp + (int64_t)row * row_vecs;
#pragma unroll
            for (int i = 0; i < kVpl; ++i) {
              const int v = v0 + 32 * i;
              if (v < row_vecs) dst[v] = buf[q][i];
            }
          }
        }
      }
    }
  }
  // (f) bookkeeping, shared out over the blocks
  if (me == 0)
    for (int e = threadIdx.x; e <= M; e += blockDim.x) {
      offsets[e] = start[e];
      if (group_rows != nullptr && e < M) group_rows[e] = total[e];
    }
  for (int p = me * kDispatchWarps + warp; p < M * UNIPOOL_ROW_ALIGN; p += (int)gridDim.x * kDispatchWarps) {
    const int e = p / UNIPOOL_ROW_ALIGN;                                   // pad row p % 128 of expert e, if it has so many
    const int r = start[e] + total[e] + p % UNIPOOL_ROW_ALIGN;
    if (r >= start[e + 1]) continue;
    if (lane == 0) token_of[r] = -1;                                       // no token, zeros
    uint4* dst = Xp + (int64_t)r * row_vecs;
    for (int v = lane; v < row_vecs; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
  }
  for (int e = me; e < M; e += gridDim.x)
    for (int tl = start[e] / UNIPOOL_ROW_ALIGN + threadIdx.x; tl < start[e + 1] / UNIPOOL_ROW_ALIGN; tl += blockDim.x)
      tile_expert[tl] = e;
  const int used = start[M];
  const int gid = me * (int)blockDim.x + threadIdx.x, gstride = (int)(gridDim.x * blockDim.x);
  for (int r = used + gid; r < row_capacity; r += gstride) token_of[r] = -1;
  for (int tl = used / UNIPOOL_ROW_ALIGN + gid; tl < row_capacity / UNIPOOL_ROW_ALIGN; tl += gstride) tile_expert[tl] = -1;
}

template <typename T> struct Vec16;
template <> struct Vec16<float> {
  static constexpr int N = 4;
  __device__ static void unpack(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
  __device__ static uint4 pack(const float* f) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
  }
};
template <> struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void unpack(const uint4& v, float* f) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  __device__ static uint4 pack(const float* f) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<uint32_t*>(&p);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};

// y[t] = (residual[t]) + sum_j gate[t,j] * Yp[row_of[t,j]]   (gate == NULL: unit weights)
// KT = compile-time bound of k (registers for the rows in flight), V = 16-byte vectors of a row per lane and pass.
template <typename T, int KT, int V>
__global__ void __launch_bounds__(256, V > 1 ? 1 : sizeof(T) == 2 ? 4 : 3)
combine_kernel(const uint4* __restrict__ Yp, const int32_t* __restrict__ row_of,
               const float* __restrict__ gate, const uint4* __restrict__ residual,
               uint4* __restrict__ y, int n_tokens, int k, int row_vecs) {
  grid_wait(Yp, row_of, gate, residual);
  constexpr int N = Vec16<T>::N;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int t = blockIdx.x * 8 + warp; t < n_tokens; t += gridDim.x * 8) {
    int rows[KT];
    float g[KT];
#pragma unroll
    for (int j = 0; j < KT; ++j) {
      rows[j] = j < k ? __ldg(row_of + (int64_t)t * k + j) : -1;
      g[j] = (j < k && gate) ? __ldg(gate + (int64_t)t * k + j) : 1.f;
    }
    for (int v0 = lane; v0 < row_vecs; v0 += 32 * V) {
      uint4 rv[V], yv[KT][V];
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int v = v0 + 32 * i;
        rv[i] = (residual && v < row_vecs) ? __ldg(residual + (int64_t)t * row_vecs + v) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < KT; ++j)
          yv[j][i] = (rows[j] >= 0 && v < row_vecs) ? __ldg(Yp + (int64_t)rows[j] * row_vecs + v)
                                                    : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int v = v0 + 32 * i;
        if (v >= row_vecs) continue;
        float acc[N];
        if (residual) {
          Vec16<T>::unpack(rv[i], acc);
        } else {
#pragma unroll
          for (int q = 0; q < N; ++q) acc[q] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < KT; ++j) {
          if (rows[j] < 0) continue;
          float fv[N];
          Vec16<T>::unpack(yv[j][i], fv);
#pragma unroll
          for (int q = 0; q < N; ++q) acc[q] = fmaf(g[j], fv[q], acc[q]);
        }
        y[(int64_t)t * row_vecs + v] = Vec16<T>::pack(acc);
      }
    }
  }
}

// Backward of the combine, token-major: for token t and slot j with row r = row_of[t,j]
//   dgate[t,j] = <dy[t], Yp[r]>,   dYp[r] = gate[t,j] * dy[t];
// the pad rows (token_of < 0) below offsets[M] are zeroed afterwards; with group_rows, by further warps beside the
// tokens', only those up to the next multiple of pad_step rows, and the group sizes are counted in token_of and
// written there: what the array holds on entry may belong to another permute.  A warp takes KT slots of one
// token; with k > KT the token's slots are split over ceil(k / KT) warps (each re-reads dy[t], which
// keeps the registers per thread low enough for four resident blocks per SM).
template <typename T, int KT>
__global__ void __launch_bounds__(256, 4)
combine_bwd_kernel(const uint4* __restrict__ dy, const uint4* __restrict__ Yp,
                   const int32_t* __restrict__ row_of, const float* __restrict__ gate,
                   const int32_t* __restrict__ token_of, const int32_t* __restrict__ offsets,
                   int32_t* __restrict__ group_rows, int pad_step, int M, uint4* __restrict__ dYp,
                   float* __restrict__ dgate, int n_tokens, int k, int row_vecs) {
  grid_wait(dy, Yp, row_of, gate, token_of, offsets);
  constexpr int N = Vec16<T>::N;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int groups = (k + KT - 1) / KT;
  const int n_items = n_tokens * groups;                 // < 2^30: T * k is
  const int n_pads = group_rows != nullptr ? M * pad_step : 0;
  for (int item = blockIdx.x * 8 + warp; item < n_items + n_pads; item += gridDim.x * 8) {
    if (item >= n_items) {
      const int p = item - n_items, e = p / pad_step, i = p % pad_step, end = __ldg(offsets + e + 1);
      int n = end - __ldg(offsets + e);                          // the padding lies in the group's last 128 rows
      if (n > 0) {
        const int32_t* tail = token_of + end - UNIPOOL_ROW_ALIGN;
        n -= UNIPOOL_ROW_ALIGN;
#pragma unroll
        for (int q = 0; q < UNIPOOL_ROW_ALIGN / 32; ++q) n += __popc(__ballot_sync(0xffffffffu, __ldg(tail + 32 * q + lane) >= 0));
      }
      if (i == 0 && lane == 0) group_rows[e] = n;
      if (i >= (-n & (pad_step - 1))) continue;
      uint4* dst = dYp + (int64_t)(offsets[e] + n + i) * row_vecs;
      for (int v = lane; v < row_vecs; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
      continue;
    }
    const int t = groups == 1 ? item : item / groups, j0 = groups == 1 ? 0 : (item % groups) * KT;
    int rows[KT];
    float g[KT], dot[KT];
#pragma unroll
    for (int j = 0; j < KT; ++j) {
      rows[j] = j0 + j < k ? __ldg(row_of + (int64_t)t * k + j0 + j) : -1;
      g[j] = j0 + j < k ? __ldg(gate + (int64_t)t * k + j0 + j) : 0.f;
      dot[j] = 0.f;
    }
    for (int v0 = lane; v0 < row_vecs; v0 += 32 * kVpl) {
      uint4 dv[kVpl], yv[KT][kVpl];
#pragma unroll
      for (int i = 0; i < kVpl; ++i) {
        const int v = v0 + 32 * i;
        dv[i] = v < row_vecs ? __ldg(dy + (int64_t)t * row_vecs + v) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < KT; ++j)
          yv[j][i] = (rows[j] >= 0 && v < row_vecs) ? __ldg(Yp + (int64_t)rows[j] * row_vecs + v)
                                                    : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int i = 0; i < kVpl; ++i) {
        const int v = v0 + 32 * i;
        if (v >= row_vecs) continue;
        float a[N];
        Vec16<T>::unpack(dv[i], a);
#pragma unroll
        for (int j = 0; j < KT; ++j) {
          if (rows[j] < 0) continue;
          float fv[N], o[N];
          Vec16<T>::unpack(yv[j][i], fv);
#pragma unroll
          for (int q = 0; q < N; ++q) {
            dot[j] = fmaf(a[q], fv[q], dot[j]);
            o[q] = g[j] * a[q];
          }
          dYp[(int64_t)rows[j] * row_vecs + v] = Vec16<T>::pack(o);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < KT; ++j) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dot[j] += __shfl_xor_sync(0xffffffffu, dot[j], o);
      if (lane == 0 && j0 + j < k) dgate[(int64_t)t * k + j0 + j] = dot[j];
    }
  }
  if (group_rows != nullptr) return;
  const int used = offsets[M];
  for (int r = blockIdx.x * 8 + warp; r < used; r += gridDim.x * 8) {
    if (token_of[r] >= 0) continue;
    uint4* dst = dYp + (int64_t)r * row_vecs;
    for (int v = lane; v < row_vecs; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
  }
}

__global__ void dispatch_empty_kernel(int32_t* offsets, int32_t* token_of, int32_t* tile_expert, int32_t* group_rows,
                                      int M, int row_capacity) {
  grid_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (group_rows != nullptr && i < M) group_rows[i] = 0;
  if (i <= M) offsets[i] = 0;
  if (i < row_capacity) token_of[i] = -1;
  if (i < row_capacity / UNIPOOL_ROW_ALIGN) tile_expert[i] = -1;
}

static size_t place_smem_bytes(int M, int k, int chunk) {
  return ((size_t)kDispatchWarps * M + (M + 1) + 2 * (size_t)M + (size_t)chunk * k) * sizeof(int);
}

// Tokens per chunk (= per block of the placing kernel): the largest of 256 .. 16 that still gives every SM a
// block - a block moves its own tokens, and an SM alone pulls well under its share of the memory bandwidth.
static int dispatch_chunk_tokens(int T, int sm_count) {
  if (sm_count > kDispatchMaxSms) sm_count = kDispatchMaxSms;
  for (int chunk = kDispatchChunkTokens; chunk > kDispatchMinChunkTokens; chunk /= 2)
    if ((T + chunk - 1) / chunk >= sm_count) return chunk;
  return kDispatchMinChunkTokens;
}

// Up to this many assignments every block counts all of them itself (16 per thread) instead of waiting for a
// histogram kernel.
constexpr int64_t kSelfCountAssignments = 4096;

// The two launches of the permute (T > 0).  counts: scratch, 36 bytes per (16 chunks, expert).
static int permute_launch(unipool_ctx* prof, const void* x, int T, int k, const int32_t* idx, int M, int chunk,
                          int sm_count, void* counts, int32_t* status, int row_vecs, int cap, int32_t* offsets,
                          int32_t* row_of, int32_t* token_of, int32_t* tile_expert, int32_t* rows, void* Xp,
                          cudaStream_t s) {
  const int n_chunks = (T + chunk - 1) / chunk;
  ChunkCounts cc = chunk_counts(counts, n_chunks, M);
  if ((int64_t)T * k <= kSelfCountAssignments) {
    cc.n_super = 0;
  } else {
    PhaseTimer pt(prof, UNIPOOL_PH_DISPATCH_MAPS, 1, s);
    UP_KERNEL(dispatch_hist_kernel, cc.n_super, kHistWarps * 32, kHistWarps * M * sizeof(int), s, idx, T, k, M, chunk, cc, status);
  }
  PhaseTimer pt(prof, UNIPOOL_PH_DISPATCH_GATHER, 1, s);
  // A small batch has few chunks but as many pad rows as a large one: blocks without a chunk share those.
  const int grid = n_chunks > sm_count ? n_chunks : sm_count;
  UP_KERNEL(dispatch_place_kernel, grid, kDispatchWarps * 32, place_smem_bytes(M, k, chunk), s, idx, T, k, M, chunk, cc, status, static_cast<const uint4*>(x), row_vecs, cap, offsets, row_of, token_of, tile_expert,
      rows, static_cast<uint4*>(Xp));
  return UNIPOOL_OK;
}

static int row_mover_grid(const unipool_ctx* ctx, int64_t rows) {
  int64_t want = (rows + 7) / 8;
  int64_t cap = (int64_t)ctx->sm_count * 8;      // 8 resident 256-thread blocks per SM
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

int dispatch_launch(unipool_ctx* ctx, const void* x, int T, const int32_t* idx, int M,
                    int32_t* offsets, int32_t* row_of, int32_t* token_of, int32_t* tile_expert,
                    int32_t* rows, void* Xp, cudaStream_t s) {
  const int k = ctx->cfg.top_k, d = ctx->cfg.d_model;
  const int cap = (int)ctx->row_capacity;
  if (T == 0) {
    UP_KERNEL(dispatch_empty_kernel, (cap + 255) / 256, 256, 0, s, offsets, token_of, tile_expert, rows, M, cap);
    return UNIPOOL_OK;
  }
  return permute_launch(ctx, x, T, k, idx, M, dispatch_chunk_tokens(T, ctx->sm_count), ctx->sm_count, ctx->ws.block_hist,
                        ctx->ws.status, (int)((size_t)d * ctx->elem_bytes / 16), cap, offsets, row_of, token_of,
                        tile_expert, rows, Xp, s);
}

// With up to eight rows in flight three vectors a pass leave an SM one block (176 registers), one vector four (in 64
// registers, 48 bytes of the bf16 form spilled; three in fp32).  A token's passes follow one another, so few tokens want
// few passes; as soon as a second round of one-block SMs is needed, more blocks are worth more.  us, three vectors / one:
//   bf16, top-8   200 tokens of 768 3.6 / 5.3, 1184 5.3 / 6.6, 1185 6.9 / 6.5, 1500 8.0 / 6.9, 4096 15.9 / 12.3, 16384 51 / 44
//                 1184 of 2944 13.8 / 18.4, 1500 22.0 / 21.8, 2000 24.9 / 24.5, 2400 33.9 / 29.1; 2000 of 384 6.5 / 5.7
//   fp32, top-8   1184 of 256 4.0 / 5.0, 1500 5.7 / 5.2; 1184 of 768 7.4 / 10.9, 1500 10.3 / 11.6, 2000 11.9 / 13.0, 2600 15.8 / 15.3
// (One vector at k = 3, 4, where three leave two blocks: top-4, 2000 tokens of 2944 11.3 -> 14.3, 16384 of 768 27.1 -> 26.8.)
static bool combine_in_few_passes(const unipool_ctx* ctx, int n_tokens, int row_vecs) {
  const int rounds = ctx->cfg.dtype == UNIPOOL_FP32 && row_vecs > 32 * kVpl ? 2 : 1;
  return n_tokens <= 8 * rounds * ctx->sm_count;
}

template <typename T>
static int combine_dispatch_k(const unipool_ctx* ctx, int grid, cudaStream_t s, int k, const void* Yp, const int32_t* row_of,
                              const float* gate, const void* residual, void* y, int n_tokens, int row_vecs) {
  auto Y = static_cast<const uint4*>(Yp);
  auto R = static_cast<const uint4*>(residual);
  auto O = static_cast<uint4*>(y);
  auto kern = k <= 1 ? combine_kernel<T, 1, kVpl> : k <= 2 ? combine_kernel<T, 2, kVpl> : k <= 4 ? combine_kernel<T, 4, kVpl>
              : combine_in_few_passes(ctx, n_tokens, row_vecs) ? combine_kernel<T, 8, kVpl> : combine_kernel<T, 8, 1>;
  UP_KERNEL(kern, grid, 256, 0, s, Y, row_of, gate, R, O, n_tokens, k, row_vecs);
  return UNIPOOL_OK;
}

static int combine_phase(unipool_ctx* ctx, int phase, const void* Yp, const int32_t* row_of,
                         const float* gate, int T, const void* residual, void* y, cudaStream_t s) {
  if (T == 0) return UNIPOOL_OK;
  PhaseTimer pt(ctx, phase, 1, s);
  const int k = ctx->cfg.top_k;
  const int row_vecs = (int)((size_t)ctx->cfg.d_model * ctx->elem_bytes / 16);
  const int grid = row_mover_grid(ctx, T);
  if (ctx->cfg.dtype == UNIPOOL_BF16)
    return combine_dispatch_k<__nv_bfloat16>(ctx, grid, s, k, Yp, row_of, gate, residual, y, T, row_vecs);
  return combine_dispatch_k<float>(ctx, grid, s, k, Yp, row_of, gate, residual, y, T, row_vecs);
}

int combine_launch(unipool_ctx* ctx, const void* Yp, const int32_t* row_of, const float* gate, int T,
                   const void* residual, void* y, cudaStream_t s) {
  return combine_phase(ctx, UNIPOOL_PH_COMBINE, Yp, row_of, gate, T, residual, y, s);
}

template <typename T>
static int combine_bwd_dispatch_k(int grid, cudaStream_t s, int k, const void* dy, const void* Yp,
                                  const int32_t* row_of, const float* gate, const int32_t* token_of,
                                  const int32_t* offsets, int32_t* rows, int M, void* dYp, float* dgate,
                                  int n_tokens, int row_vecs) {
  constexpr int step = sizeof(T) == 2 ? kRowStep : UNIPOOL_ROW_ALIGN;       // (the fp32 kernels read whole groups)
  auto D = static_cast<const uint4*>(dy);
  auto Y = static_cast<const uint4*>(Yp);
  auto O = static_cast<uint4*>(dYp);
  UP_KERNEL((k <= 1 ? combine_bwd_kernel<T, 1> : combine_bwd_kernel<T, 2>), grid, 256, 0, s, D, Y, row_of, gate, token_of, offsets, rows,
            step, M, O, dgate, n_tokens, k, row_vecs);
  return UNIPOOL_OK;
}

int combine_bwd_launch(unipool_ctx* ctx, const void* dy, int T, const int32_t* row_of,
                       const float* gate, const int32_t* token_of, const int32_t* offsets, int32_t* rows, int M,
                       const void* Yp, void* dYp, float* dgate, cudaStream_t s) {
  if (T == 0) return UNIPOOL_OK;
  const int k = ctx->cfg.top_k;
  const int row_vecs = (int)((size_t)ctx->cfg.d_model * ctx->elem_bytes / 16);
  // one warp per token and pair of slots, and per pad row that is to be looked at
  const int64_t pads = rows == nullptr ? 0 : (int64_t)M * (ctx->cfg.dtype == UNIPOOL_BF16 ? kRowStep : UNIPOOL_ROW_ALIGN);
  const int grid = row_mover_grid(ctx, (int64_t)T * ((k + 1) / 2) + pads);
  PhaseTimer pt(ctx, UNIPOOL_PH_BWD_SCALE_GATHER, 1, s);
  if (ctx->cfg.dtype == UNIPOOL_BF16)
    return combine_bwd_dispatch_k<__nv_bfloat16>(grid, s, k, dy, Yp, row_of, gate, token_of, offsets, rows, M, dYp, dgate, T, row_vecs);
  return combine_bwd_dispatch_k<float>(grid, s, k, dy, Yp, row_of, gate, token_of, offsets, rows, M, dYp, dgate, T, row_vecs);
}

int unpermute_sum_launch(unipool_ctx* ctx, const void* dXp, const int32_t* row_of, int T,
                         const void* residual, void* dx, cudaStream_t s) {
  // dx_t = residual_t + sum_j dXp[row_of[t,j]]: the combine kernel with unit weights
  return combine_phase(ctx, UNIPOOL_PH_UNPERMUTE_SUM, dXp, row_of, nullptr, T, residual, dx, s);
}

}  // namespace unipool

// ---------------------------------------------------------------- dispatch without a workspace
// Scratch of unipool_dispatch_static: the per-chunk histograms of the map kernels plus a status
// word, held in the library's own device image.  Every GPU that loads the library carries these
// 2 MiB until the process exits.  All calls share them.
namespace {
constexpr int64_t kStaticHistInts = 1024 * 512 - 64;      // chunks x experts accepted: 36 / 16 bytes each and one group rounded up
static __device__ __align__(256) int32_t g_dispatch_scratch[1024 * 512];
constexpr int kMaxDevices = 64;
// per device: the array's address there, looked up by the first call on that device.
// Host threads may race on the first call: the entry is complete before its address becomes visible.
struct ScratchInfo { int32_t* addr; };
std::atomic<const ScratchInfo*> g_scratch[kMaxDevices];
ScratchInfo g_scratch_slots[kMaxDevices][2];
std::atomic<int> g_scratch_next[kMaxDevices];
}  // namespace

extern "C" int unipool_dispatch_static(const void* x, int32_t T, int32_t d_model, int32_t dtype, int32_t top_k,
                                       const int32_t* idx, int32_t n_experts, int64_t row_capacity,
                                       int32_t* offsets, int32_t* row_of, int32_t* token_of,
                                       int32_t* tile_expert, void* Xp, unipool_stream stream) {
  using namespace unipool;
  UP_REQUIRE(x && idx && offsets && row_of && token_of && tile_expert && Xp, UNIPOOL_ERR_INVALID_ARG,
             "dispatch_static: a tensor pointer is NULL");
  UP_REQUIRE(dtype == UNIPOOL_FP32 || dtype == UNIPOOL_BF16, UNIPOOL_ERR_INVALID_ARG, "dispatch_static: bad dtype %d", dtype);
  const size_t eb = dtype == UNIPOOL_BF16 ? 2 : 4;
  UP_REQUIRE(d_model > 0 && ((size_t)d_model * eb) % 16 == 0, UNIPOOL_ERR_UNSUPPORTED,
             "dispatch_static: a row of %d elements is not a whole number of 16-byte vectors", d_model);
  UP_REQUIRE(n_experts >= 1 && n_experts <= UNIPOOL_MAX_EXPERTS && top_k >= 1 && top_k <= UNIPOOL_MAX_TOPK &&
                 top_k <= n_experts, UNIPOOL_ERR_UNSUPPORTED, "dispatch_static: bad (n_experts, top_k) = (%d, %d)",
             n_experts, top_k);
  UP_REQUIRE(T >= 0 && (int64_t)T * top_k < (1ll << 30), UNIPOOL_ERR_UNSUPPORTED, "dispatch_static: bad T = %d", T);
  const int64_t need_rows = ((int64_t)T * top_k + (int64_t)n_experts * (UNIPOOL_ROW_ALIGN - 1) + UNIPOOL_ROW_ALIGN - 1) /
                            UNIPOOL_ROW_ALIGN * UNIPOOL_ROW_ALIGN;
  UP_REQUIRE(row_capacity % UNIPOOL_ROW_ALIGN == 0 && row_capacity >= need_rows && row_capacity < (1ll << 31),
             UNIPOOL_ERR_INVALID_ARG, "dispatch_static: row_capacity %lld, need a multiple of %d >= %lld",
             (long long)row_capacity, UNIPOOL_ROW_ALIGN, (long long)need_rows);
  const int n_blocks = (T + kDispatchChunkTokens - 1) / kDispatchChunkTokens;
  UP_REQUIRE((int64_t)n_blocks * n_experts <= kStaticHistInts, UNIPOOL_ERR_WORKSPACE,
             "dispatch_static: ceil(T/%d) * n_experts = %lld exceeds the built-in scratch of %lld entries "
             "(use unipool_dispatch with a workspace)", kDispatchChunkTokens, (long long)n_blocks * n_experts,
             (long long)kStaticHistInts);
  int dev = 0;
  UP_CUDA(cudaGetDevice(&dev));
  UP_REQUIRE(dev >= 0 && dev < kMaxDevices, UNIPOOL_ERR_UNSUPPORTED, "dispatch_static: device ordinal %d", dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const ScratchInfo* info = g_scratch[dev].load(std::memory_order_acquire);
  if (info == nullptr) {
    // Once per device, with that device current: in host code the array's name is only a handle,
    // the kernels need the address it has on THIS device.  Two threads that both get here look up the
    // same values; each fills a slot of its own and publishes it.
    int32_t* ptr = nullptr;
    UP_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_dispatch_scratch));
    UP_REQUIRE(ptr != nullptr, UNIPOOL_ERR_CUDA, "dispatch_static: no address for the built-in scratch");
    const int slot = g_scratch_next[dev].fetch_add(1) & 1;
    g_scratch_slots[dev][slot] = ScratchInfo{ptr};
    g_scratch[dev].store(&g_scratch_slots[dev][slot], std::memory_order_release);
    info = &g_scratch_slots[dev][slot];
  }
  int32_t* status = info->addr;                            // [0, 64): status word (+ spare)
  int32_t* counts = info->addr + 64;
  const int cap = (int)row_capacity;
  if (T == 0) {
    UP_KERNEL(dispatch_empty_kernel, (cap + 255) / 256, 256, 0, s, offsets, token_of, tile_expert, nullptr, n_experts, cap);
    return UNIPOOL_OK;
  }
  // the counts are fully rewritten by the first kernel for the chunks of this call; nothing else in the
  // array has to start at zero
  int sm_count = 0;
  UP_CUDA(cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev));
  return permute_launch(nullptr, x, T, top_k, idx, n_experts, kDispatchChunkTokens, sm_count, counts, status,
                        (int)((size_t)d_model * eb / 16), cap, offsets, row_of, token_of, tile_expert, nullptr, Xp, s);
}
