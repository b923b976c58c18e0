// Router forward (NormRouter, Eq. 7, or softmax; top-k, Sec. 4.3) and backward.
#include <cfloat>

#include "common.cuh"
#include "simt_gemm.cuh"

namespace unipool {

// ---------------------------------------------------------------- logits  z = x W_r^T (+ bias)
// Eight warps share a tile of 32 tokens and 64 experts while every tile has an SM to itself; of more tiles, with four warps
// to each, an SM takes three.  us of the router with eight / four: 512 tokens, 16 experts of 256 11.9 / 12.8; 1024, 384 of 256 (192
// tiles) 22.8 / 20.5; 8192, 16 of 256 (256) 23.3 / 21.0; 16384, 96 of 768 123 / 108.  (Eight: 255 registers, 44 bytes spilled.)
template <typename RouterTile>
__global__ void __launch_bounds__(RouterTile::kThreads, RouterTile::kBlocks)
router_logits_kernel(const float* __restrict__ x, const float* __restrict__ W_r,
                     const float* __restrict__ bias, float* __restrict__ z, int T, int M, int d, bool vec) {
  grid_wait(x, W_r, bias);
  extern __shared__ float4 smem_raw[];
  typename RouterTile::Smem& sm = *reinterpret_cast<typename RouterTile::Smem*>(smem_raw);
  const int m0 = blockIdx.x * kSimtM, n0 = blockIdx.y * kSimtN;
  RouterTile::template run<kAlongK, kAlongK>(
      sm, d / kSimtKC, vec, vec, x, [](int) {},
      [&](int c, int i, int k) { return m0 + i < T ? x + (int64_t)(m0 + i) * d + c * kSimtKC + k : nullptr; },
      [&](int c, int i, int k) { return n0 + i < M ? W_r + (int64_t)(n0 + i) * d + c * kSimtKC + k : nullptr; });
  for (int q = threadIdx.x; q < kSimtM * kSimtN; q += RouterTile::kThreads) {
    const int tok = m0 + q / kSimtN, e = n0 + q % kSimtN;
    if (tok < T && e < M) z[(int64_t)tok * M + e] = RouterTile::value(sm, q / kSimtN, q % kSimtN) + (bias ? bias[e] : 0.f);
  }
}

template <typename RouterTile>
static int router_logits_as(const float* x, const float* W_r, const float* bias, float* z, int T, int M, int d, cudaStream_t s) {
  auto kern = router_logits_kernel<RouterTile>;
  constexpr int smem = (int)sizeof(typename RouterTile::Smem);
  UP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  UP_KERNEL(kern, dim3((T + kSimtM - 1) / kSimtM, (M + kSimtN - 1) / kSimtN), RouterTile::kThreads, smem, s, x, W_r, bias, z, T, M, d,
            aligned16(x, W_r));
  return UNIPOOL_OK;
}

// ---------------------------------------------------------------- scores, top-k, statistics
// One warp per token.  Lane l holds experts l, l+32, ...  Selection key: score
// descending, expert index ascending.
constexpr int kRouteWarps = 8;

template <bool SOFTMAX, int kPerWarp>
__global__ void __launch_bounds__(kRouteWarps * 32)
router_select_kernel(const float* __restrict__ z, int T, int M, int k, float sigma_c, float eps,
                     int32_t* __restrict__ idx, float* __restrict__ gate, float* __restrict__ znorm,
                     int32_t* __restrict__ counts_out, float* __restrict__ sum_out,
                     int32_t* __restrict__ acc_counts, double* __restrict__ acc_sums,
                     uint32_t* __restrict__ ticket) {
  extern __shared__ float smem[];
  float* sc = smem;                                           // [warps][M] scores of the current token
  float* wsum = smem + kRouteWarps * M;                       // [warps][M] per-warp score sums
  int* hist = reinterpret_cast<int*>(wsum + kRouteWarps * M); // [M]
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int i = threadIdx.x; i < M; i += blockDim.x) hist[i] = 0;
  for (int i = lane; i < M; i += 32) wsum[warp * M + i] = 0.f;
  grid_wait(z);
  __syncthreads();

  float* my = sc + warp * M;
  const int t_begin = (blockIdx.x * kRouteWarps + warp) * kPerWarp;
  for (int tt = 0; tt < kPerWarp; ++tt) {
    const int t = t_begin + tt;
    if (t >= T) break;
    const float* zr = z + (int64_t)t * M;
    if (SOFTMAX) {
      // s = exp(z - max) / sum exp(z - max); the log-sum-exp goes where the NormRouter keeps ||z||
      float mx = -INFINITY;
      for (int i = lane; i < M; i += 32) {
        float v = __ldg(zr + i);
        my[i] = v;
        mx = fmaxf(mx, v);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float tot = 0.f;
      for (int i = lane; i < M; i += 32) {
        float e = expf(my[i] - mx);
        my[i] = e;
        tot += e;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      for (int i = lane; i < M; i += 32) {
        float s = my[i] / tot;
        my[i] = s;
        wsum[warp * M + i] += s;
      }
      if (lane == 0) znorm[t] = mx + logf(tot);
    } else {
      float ss = 0.f;
      for (int i = lane; i < M; i += 32) {
        float v = __ldg(zr + i);
        my[i] = v;
        ss = fmaf(v, v, ss);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      const float n = sqrtf(ss);
      const float den = n + eps;
      for (int i = lane; i < M; i += 32) {
        float s = sigma_c * fmaxf(0.f, my[i] / den);
        my[i] = s;
        wsum[warp * M + i] += s;
      }
      if (lane == 0) znorm[t] = n;
    }
    __syncwarp();
    for (int j = 0; j < k; ++j) {
      float bv = -INFINITY;
      int bi = INT_MAX;
      for (int i = lane; i < M; i += 32) {
        float v = my[i];
        if (v != -INFINITY && !(v == v)) v = -FLT_MAX;       // NaN scores sort last but stay selectable
        if (v > bv) { bv = v; bi = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
      }
      if (lane == 0) {
        idx[(int64_t)t * k + j] = bi;
        gate[(int64_t)t * k + j] = my[bi];
        atomicAdd(&hist[bi], 1);
        my[bi] = -INFINITY;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  // block totals -> global accumulators (integer counts exact; score sums in double)
  for (int i = threadIdx.x; i < M; i += blockDim.x) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kRouteWarps; ++w) s += wsum[w * M + i];
    if (hist[i]) atomicAdd(&acc_counts[i], hist[i]);
    if (s != 0.f) atomicAdd(&acc_sums[i], (double)s);
  }
  __threadfence();
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last) {                       // the block that arrives last publishes and resets
    __threadfence();
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
      counts_out[i] = __ldcg(&acc_counts[i]);
      sum_out[i] = (float)__ldcg(&acc_sums[i]);
      acc_counts[i] = 0;
      acc_sums[i] = 0.0;
    }
    if (threadIdx.x == 0) *ticket = 0u;
  }
}

__global__ void zero_stats_kernel(int32_t* counts, float* sums, int M) {
  grid_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < M) { counts[i] = 0; sums[i] = 0.f; }
}

int route_launch(unipool_ctx* ctx, const void* x, int T, const float* W_r, float sigma,
                 const float* bias, int M, int32_t* idx, float* gate, int32_t* counts,
                 float* score_sum, float* znorm, float* z_saved, cudaStream_t s) {
  const int d = ctx->cfg.d_model, k = ctx->cfg.top_k;
  if (T == 0) {
    UP_KERNEL(zero_stats_kernel, (M + 127) / 128, 128, 0, s, counts, score_sum, M);
    return UNIPOOL_OK;
  }
  if (ctx->cfg.dtype == UNIPOOL_BF16)
    return (route_on_few(ctx, W_r, T, M) ? route_few_launch : route_tc_launch)(ctx, x, T, W_r, sigma, bias, M, idx, gate, counts,
                                                                         score_sum, znorm, z_saved, s);
  {
    PhaseTimer pt(ctx, UNIPOOL_PH_ROUTE_LOGITS, 1, s);
    const int64_t tiles = (int64_t)((T + kSimtM - 1) / kSimtM) * ((M + kSimtN - 1) / kSimtN);
    const int rc = (tiles <= ctx->sm_count ? router_logits_as<SimtTile<8>> : router_logits_as<SimtTile<4>>)(
        static_cast<const float*>(x), W_r, bias, z_saved, T, M, d, s);
    if (rc != UNIPOOL_OK) return rc;
  }
  PhaseTimer pt(ctx, UNIPOOL_PH_ROUTE_SELECT, 1, s);
  // A token to a warp, or four one after the other: more blocks hide more latency, but each adds its totals of all experts by
  // atomics.  us of the router with one / four (experts of 256): 512 tokens, 16 experts 12.1 / 15.5; 4800, 16 18.1 / 20.2; 8192, 16
  // 20.4 / 21.2; 4736, 64 17.4 / 17.7; 9000, 64 25.3 / 22.7; 2400, 96 20.7 / 22.0; 3552, 96 23.5 / 22.3; 4736, 96 25.9 / 23.3;
  // 2400, 384 33.4 / 37.7; 4736, 512 56.3 / 57.1.
  const int most = M <= 32 ? 8 : M <= 64 ? 4 : 3;              // blocks to an SM
  const int per_warp = T <= most * kRouteWarps * ctx->sm_count ? 1 : 4, per_block = kRouteWarps * per_warp;
  const int blocks = (T + per_block - 1) / per_block;
  const size_t smem = (size_t)(2 * kRouteWarps * M) * sizeof(float) + (size_t)M * sizeof(int);
  static_assert((2 * kRouteWarps + 1) * UNIPOOL_MAX_EXPERTS * 4 <= 48 * 1024, "no opt-in to more shared memory");
  const bool softmax = ctx->cfg.router_mode == UNIPOOL_ROUTER_SOFTMAX;
  auto kern = per_warp == 1 ? (softmax ? router_select_kernel<true, 1> : router_select_kernel<false, 1>)
                            : (softmax ? router_select_kernel<true, 4> : router_select_kernel<false, 4>);
  UP_KERNEL(kern, blocks, kRouteWarps * 32, smem, s, z_saved, T, M, k, sigma * ctx->cfg.c, ctx->cfg.eps, idx, gate, znorm,
            counts, score_sum, ctx->ws.route_counts, ctx->ws.route_sums, ctx->ws.tickets + 0);
  return UNIPOOL_OK;
}

// ---------------------------------------------------------------- backward
// dz from (z, n, idx, dgate, coef); one warp per token.
template <bool SOFTMAX>
__global__ void __launch_bounds__(256)
router_dz_kernel(const float* __restrict__ z, const float* __restrict__ znorm,
                 const int32_t* __restrict__ idx, const float* __restrict__ dgate,
                 const float* __restrict__ coef, int T, int M, int k, float sigma, float c, float eps,
                 float* __restrict__ dz, float* __restrict__ dsigma, double* __restrict__ acc,
                 uint32_t* __restrict__ ticket) {
  grid_wait(z, znorm, idx, dgate, coef);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int t = blockIdx.x * (blockDim.x / 32) + warp;
  float dsig_part = 0.f;
  if (t < T) {
    const float* zr = z + (int64_t)t * M;
    int my_idx = -1;
    float my_dg = 0.f;
    if (lane < k) { my_idx = __ldg(idx + (int64_t)t * k + lane); my_dg = __ldg(dgate + (int64_t)t * k + lane); }
    const float n = __ldg(znorm + t);
    const float ne = n + eps;
    float q = 0.f;
    // pass 1: q = sum_i ds_i * max(z_i, 0)
    for (int i0 = 0; i0 < M; i0 += 32) {
      int i = i0 + lane;
      float ds = (i < M && coef) ? __ldg(coef + i) : 0.f;
      for (int j = 0; j < k; ++j) {
        int ej = __shfl_sync(0xffffffffu, my_idx, j);
        float dj = __shfl_sync(0xffffffffu, my_dg, j);
        if (ej == i) ds += dj;
      }
      if (i < M) q = fmaf(ds, SOFTMAX ? expf(__ldg(zr + i) - n) : fmaxf(__ldg(zr + i), 0.f), q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    const float scale = sigma * c;
    const float qn = n > 0.f ? q / (n * ne * ne) : 0.f;
    for (int i0 = 0; i0 < M; i0 += 32) {
      int i = i0 + lane;
      float ds = (i < M && coef) ? __ldg(coef + i) : 0.f;
      for (int j = 0; j < k; ++j) {
        int ej = __shfl_sync(0xffffffffu, my_idx, j);
        float dj = __shfl_sync(0xffffffffu, my_dg, j);
        if (ej == i) ds += dj;
      }
      if (i < M) {
        float zi = __ldg(zr + i);
        float v = n > 0.f ? scale * ((zi > 0.f ? ds / ne : 0.f) - zi * qn) : 0.f;
        if (SOFTMAX) v = expf(zi - n) * (ds - q);          // n holds log sum exp(z)
        dz[(int64_t)t * M + i] = v;
      }
    }
    dsig_part = SOFTMAX ? 0.f : c * q / ne;
  }
  __shared__ float part[8];
  if (lane == 0) part[warp] = dsig_part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) s += (double)part[w];
    atomicAdd(acc, s);
    __threadfence();
    if (atomicAdd(ticket, 1u) == gridDim.x - 1) {
      __threadfence();
      *dsigma += (float)__ldcg(acc);
      *acc = 0.0;
      *ticket = 0u;
    }
  }
}

// dx[t,:] += dz[t,:] W_r     (K = M)
using RouterDxTile = SimtTile<4>;

__global__ void __launch_bounds__(RouterDxTile::kThreads, RouterDxTile::kBlocks)
router_dx_kernel(const float* __restrict__ dz, const float* __restrict__ W_r, float* __restrict__ dx,
                 int T, int M, int d, bool vec, bool vec_dx) {
  grid_wait(dz, W_r);
  extern __shared__ float4 smem_raw[];
  RouterDxTile::Smem& sm = *reinterpret_cast<RouterDxTile::Smem*>(smem_raw);
  const int m0 = blockIdx.x * kSimtM, n0 = blockIdx.y * kSimtN;
  RouterDxTile::run<kAlongK, kAcrossK>(
      sm, (M + kSimtKC - 1) / kSimtKC, (M & 3) == 0, vec, dz, [](int) {},     // dz is a workspace array of rows of M
      [&](int c, int i, int k) {
        const int kk = c * kSimtKC + k;
        return m0 + i < T && kk < M ? dz + (int64_t)(m0 + i) * M + kk : nullptr;
      },
      [&](int c, int i, int k) {
        const int kk = c * kSimtKC + k;
        return kk < M ? W_r + (int64_t)kk * d + n0 + i : nullptr;
      });
  constexpr int kMine = kSimtM * kSimtN / 4 / RouterDxTile::kThreads;
  float4 old[kMine];
#pragma unroll
  for (int u = 0; u < kMine; ++u) {
    const int q = u * RouterDxTile::kThreads + threadIdx.x, tok = m0 + q / (kSimtN / 4);
    const float* o = dx + (int64_t)tok * d + n0 + q % (kSimtN / 4) * 4;
    if (tok < T) old[u] = vec_dx ? *reinterpret_cast<const float4*>(o) : make_float4(o[0], o[1], o[2], o[3]);
  }
#pragma unroll
  for (int u = 0; u < kMine; ++u) {
    const int q = u * RouterDxTile::kThreads + threadIdx.x, tok = m0 + q / (kSimtN / 4), j = q % (kSimtN / 4) * 4;
    if (tok >= T) continue;
    const float4 v = RouterDxTile::value4(sm, q / (kSimtN / 4), j);
    st4(dx + (int64_t)tok * d + n0 + j, make_float4(old[u].x + v.x, old[u].y + v.y, old[u].z + v.z, old[u].w + v.w), vec_dx);
  }
}

// dW_r[m,:] += sum_t dz[t,m] x[t,:]   (K = T, cut into runs of k_len tokens over blockIdx.z: one run adds in
// place, several by atomics)
using RouterDwTile = SimtTile<8>;

__global__ void __launch_bounds__(RouterDwTile::kThreads, RouterDwTile::kBlocks)
router_dw_kernel(const float* __restrict__ dz, const float* __restrict__ x, float* __restrict__ dW_r,
                 int T, int M, int d, int k_len, bool vec) {
  grid_wait(dz, x);
  extern __shared__ float4 smem_raw[];
  RouterDwTile::Smem& sm = *reinterpret_cast<RouterDwTile::Smem*>(smem_raw);
  const int m0 = blockIdx.x * kSimtM, n0 = blockIdx.y * kSimtN;
  const int k_begin = blockIdx.z * k_len, k_end = min(T, k_begin + k_len);
  RouterDwTile::run<kAcrossK, kAcrossK>(
      sm, (k_end - k_begin + kSimtKC - 1) / kSimtKC, (M & 3) == 0, vec, dz, [](int) {},
      [&](int c, int i, int k) {
        const int tok = k_begin + c * kSimtKC + k;
        return tok < k_end && m0 + i < M ? dz + (int64_t)tok * M + m0 + i : nullptr;
      },
      [&](int c, int i, int k) {
        const int tok = k_begin + c * kSimtKC + k;
        return tok < k_end ? x + (int64_t)tok * d + n0 + i : nullptr;
      });
  for (int q = threadIdx.x; q < kSimtM * kSimtN; q += RouterDwTile::kThreads) {
    const int m = m0 + q / kSimtN;
    if (m >= M) continue;
    float* o = dW_r + (int64_t)m * d + n0 + q % kSimtN;
    const float v = RouterDwTile::value(sm, q / kSimtN, q % kSimtN);
    if (gridDim.z == 1) *o += v;
    else atomicAdd(o, v);
  }
}

int route_bwd_launch(unipool_ctx* ctx, const void* x, int T, const float* W_r, float sigma, int M,
                     const float* znorm, const float* z_saved, const int32_t* idx,
                     const float* dgate, const float* coef, void* dx, float* dW_r, float* dsigma,
                     cudaStream_t s) {
  if (T == 0) return UNIPOOL_OK;
  if (ctx->cfg.dtype == UNIPOOL_BF16)
    return route_bwd_tc_launch(ctx, x, T, W_r, sigma, M, znorm, z_saved, idx, dgate, coef, dx, dW_r, dsigma, s);
  const int d = ctx->cfg.d_model, k = ctx->cfg.top_k;
  float* dz = ctx->ws.dz;
  {
  PhaseTimer pt(ctx, UNIPOOL_PH_ROUTE_BWD_DZ, 1, s);
  auto kern = ctx->cfg.router_mode == UNIPOOL_ROUTER_SOFTMAX ? router_dz_kernel<true> : router_dz_kernel<false>;
  UP_KERNEL(kern, (T + 7) / 8, 256, 0, s, z_saved, znorm, idx, dgate, coef, T, M, k, sigma, ctx->cfg.c,
            ctx->cfg.eps, dz, dsigma, ctx->ws.dsigma_acc, ctx->ws.tickets + 1);
  }
  {
    PhaseTimer pt(ctx, UNIPOOL_PH_ROUTE_BWD_DX, 1, s);
    UP_CUDA(cudaFuncSetAttribute(router_dx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RouterDxTile::Smem)));
    UP_KERNEL(router_dx_kernel, dim3((T + 31) / 32, d / 64), RouterDxTile::kThreads, sizeof(RouterDxTile::Smem), s,
              dz, W_r, static_cast<float*>(dx), T, M, d, aligned16(W_r), aligned16(dx));
  }
  PhaseTimer pt(ctx, UNIPOOL_PH_ROUTE_BWD_DW, 1, s);
  const int k_len = 1024;
  UP_CUDA(cudaFuncSetAttribute(router_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RouterDwTile::Smem)));
  UP_KERNEL(router_dw_kernel, dim3((M + 31) / 32, d / 64, (T + k_len - 1) / k_len), RouterDwTile::kThreads,
            sizeof(RouterDwTile::Smem), s, dz, static_cast<const float*>(x), dW_r, T, M, d, k_len, aligned16(x));
  return UNIPOOL_OK;
}

}  // namespace unipool
