// Router forward for few tokens in bf16 mode: logits on CUDA cores, selection and statistics, one launch.
//
// Bound by latency.  On the tensor cores (route_tc.cu) a CTA pair scores 256 tokens whatever their number: 33 tokens
// are one pair that loads, multiplies and selects one step after the other while 146 SMs idle.  Here a cluster of eight
// blocks takes kTok tokens.  A block multiplies them, out of shared memory, with an eighth of the experts' weights,
// read in fp32 as they are: a warp takes four experts and eight tokens, the lanes along the width, and adds up over the
// lanes by recursive halving.  Every logit is sent to the block of the cluster that owns its token; there a warp selects.
#include <cooperative_groups.h>

#include <cfloat>
#include <climits>

#include "common.cuh"
#include "route_stats.cuh"
#include "simt_gemm.cuh"

namespace unipool {

namespace cg = cooperative_groups;

namespace {

constexpr int kFewWarps = 8;
constexpr int kFewCluster = 8;                 // blocks that share their tokens' experts
constexpr int kFewExperts = 4, kFewTokens = 8; // experts and tokens a warp multiplies at a time
constexpr int kFewAhead = 2;                   // 128-wide steps of the weights fetched ahead of their use
static_assert(kFewExperts * kFewTokens == 32, "a sum per lane");

struct FewParams {
  const __nv_bfloat16* x; const float* W_r; const float* bias;
  int T, M, d, k;
  float sigma_c, eps;
  int32_t* idx; float* gate; float* znorm; float* z_saved;
  RouteTotals totals;
  bool vec;                                    // W_r is 16-byte aligned
};

template <int kTok, bool SOFTMAX>
__global__ void __cluster_dims__(kFewCluster, 1, 1) __launch_bounds__(kFewWarps * 32, 2)
route_few_kernel(FewParams p) {
  extern __shared__ float4 smem_raw[];
  constexpr int kOwn = kTok / kFewCluster;                    // tokens that a block selects for
  const int M = p.M, d = p.d;
  float* xs = reinterpret_cast<float*>(smem_raw);             // [kTok][d] the cluster's tokens
  float* zs = xs + kTok * d;                                  // [kOwn][M] logits of the block's own, then scores
  int* hist = reinterpret_cast<int*>(zs + kOwn * M);          // [M]
  __shared__ bool last;
  cg::cluster_group cluster = cg::this_cluster();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = (int)cluster.block_rank();
  const int tc0 = (int)(blockIdx.x / kFewCluster) * kTok, t0 = tc0 + rank * kOwn;
  for (int i = threadIdx.x; i < M; i += blockDim.x) hist[i] = 0;
  grid_wait(p.x, p.W_r, p.bias);
  for (int i = 8 * threadIdx.x; i < kTok * d; i += 8 * blockDim.x) {
    const int t = tc0 + i / d;
    uint4 w = make_uint4(0, 0, 0, 0);
    if (t < p.T) w = __ldg(reinterpret_cast<const uint4*>(p.x + (int64_t)t * d + i % d));
    float4* dst = reinterpret_cast<float4*>(xs + i);
    dst[0] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                         __uint_as_float(w.y & 0xffff0000u));
    dst[1] = make_float4(__uint_as_float(w.z << 16), __uint_as_float(w.z & 0xffff0000u), __uint_as_float(w.w << 16),
                         __uint_as_float(w.w & 0xffff0000u));
  }
  cluster.sync();                                             // the tokens are staged, and all blocks have started

  constexpr int kGroups = kTok / kFewTokens;
  const int slice = ((M + kFewCluster - 1) / kFewCluster + kFewExperts - 1) / kFewExperts * kFewExperts;
  const int e_end = min(M, (rank + 1) * slice);
  for (int item = warp; item < slice / kFewExperts * kGroups; item += kFewWarps) {
    const int e0 = rank * slice + item / kGroups * kFewExperts, g = item % kGroups;
    if (e0 >= e_end) continue;
    float acc[kFewExperts * kFewTokens];
#pragma unroll
    for (int i = 0; i < kFewExperts * kFewTokens; ++i) acc[i] = 0.f;
    const float* w_e[kFewExperts];
#pragma unroll
    for (int q = 0; q < kFewExperts; ++q) w_e[q] = p.W_r + (int64_t)min(e0 + q, e_end - 1) * d;
    float4 next[kFewAhead][kFewExperts];
    auto load = [&](int c) {
#pragma unroll
      for (int a = 0; a < kFewAhead; ++a)
#pragma unroll
        for (int q = 0; q < kFewExperts; ++q)
          next[a][q] = c + 128 * a < d ? ld4(w_e[q] + c + 128 * a, p.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    load(4 * lane);
    for (int c0 = 0; c0 < d; c0 += 128 * kFewAhead) {
      float4 w[kFewAhead][kFewExperts];
#pragma unroll
      for (int a = 0; a < kFewAhead; ++a)
#pragma unroll
        for (int q = 0; q < kFewExperts; ++q) w[a][q] = next[a][q];
      load(c0 + 128 * kFewAhead + 4 * lane);
#pragma unroll
      for (int a = 0; a < kFewAhead; ++a) {
        const int c = c0 + 128 * a + 4 * lane;
        if (c < d) {
#pragma unroll
          for (int t = 0; t < kFewTokens; ++t) {
            const float4 v = *reinterpret_cast<const float4*>(xs + (g * kFewTokens + t) * d + c);
#pragma unroll
            for (int q = 0; q < kFewExperts; ++q) {
              float& s = acc[q * kFewTokens + t];
              s = fmaf(w[a][q].x, v.x, s);
              s = fmaf(w[a][q].y, v.y, s);
              s = fmaf(w[a][q].z, v.z, s);
              s = fmaf(w[a][q].w, v.w, s);
            }
          }
        }
      }
    }
    sum_over_lanes(acc, lane);                                // lane l holds expert l / 8, token l % 8
    const int e = e0 + lane / kFewTokens, t = g * kFewTokens + lane % kFewTokens;
    if (e < e_end) cluster.map_shared_rank(zs, t / kOwn)[t % kOwn * M + e] = acc[0] + (p.bias ? p.bias[e] : 0.f);
  }
  cluster.sync();                                             // the logits have arrived

  // a warp per token: norm (softmax: maximum and sum of exponentials), selection, scores
  if (warp < kOwn && t0 + warp < p.T) {
    const int t = t0 + warp;
    float* z = zs + warp * M;
    float ss = 0.f, mx = -INFINITY;
    if (SOFTMAX) {
      for (int i = lane; i < M; i += 32) mx = fmaxf(mx, z[i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    for (int i = lane; i < M; i += 32) {
      const float v = z[i];
      p.z_saved[(int64_t)t * M + i] = v;
      ss = SOFTMAX ? ss + expf(v - mx) : fmaf(v, v, ss);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float n = SOFTMAX ? mx + logf(ss) : sqrtf(ss);       // softmax keeps log sum exp(z) here
    // NormRouter: a zero logit vector scores zero.  Softmax: 1 / sum of exponentials.
    const float scale = SOFTMAX ? 1.f / ss : (ss > 0.f ? p.sigma_c / (n + p.eps) : 0.f);
    if (lane == 0) p.znorm[t] = n;
    // the order of the scores is the order of max(z, 0) (of z for the softmax); equal keys: the lower expert first
    uint32_t taken = 0;                                        // bit i: expert lane + 32 i
    for (int j = 0; j < p.k; ++j) {
      float bv = -INFINITY;
      int bi = INT_MAX;
      for (int i = lane, b = 0; i < M; i += 32, ++b) {
        const float u = SOFTMAX ? z[i] : fmaxf(z[i], 0.f);
        const float key = u == u ? u : -FLT_MAX;               // NaN logits sort last but stay selectable
        if (!(taken >> b & 1u) && key > bv) { bv = key; bi = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
      }
      if (bi != INT_MAX && bi % 32 == lane) taken |= 1u << (bi / 32);
      if (lane == 0) {
        const float g = SOFTMAX ? scale * expf(bv - mx) : scale * bv;
        p.idx[(int64_t)t * p.k + j] = bi == INT_MAX ? -1 : bi;
        p.gate[(int64_t)t * p.k + j] = bv == -FLT_MAX ? __int_as_float(0x7fc00000) : g;
        if (bi != INT_MAX) atomicAdd(&hist[bi], 1);
      }
    }
    for (int i = lane; i < M; i += 32) z[i] = scale * (SOFTMAX ? expf(z[i] - mx) : fmaxf(z[i], 0.f));
  }
  __syncthreads();
  const int live = min(kOwn, p.T - t0);
  for (int i = threadIdx.x; i < M; i += blockDim.x) {
    float sum = 0.f;
    for (int t = 0; t < live; ++t) sum += zs[t * M + i];
    add_route_total(p.totals, i, hist[i], sum);
  }
  __threadfence();
  __syncthreads();
  uint32_t* ticket = p.totals.ticket;
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();                       // the block that arrives last publishes the totals and clears the accumulators
  const bool bad = __ldcg(ticket + 1) != 0u;
  for (int i = threadIdx.x; i < M; i += blockDim.x) publish_route_total(p.totals, i, bad);
  __syncthreads();
  if (threadIdx.x == 0) { ticket[0] = 0u; ticket[1] = 0u; }
}

constexpr size_t kFewSmemMax = 100 * 1024;     // two blocks to an SM

size_t few_smem(int tok, int M, int d) { return ((size_t)tok * d + tok / kFewCluster * M + M) * sizeof(float); }

template <int kTok>
int few_launch(const unipool_ctx* ctx, const FewParams& p, cudaStream_t s) {
  auto kern = ctx->cfg.router_mode == UNIPOOL_ROUTER_SOFTMAX ? route_few_kernel<kTok, true> : route_few_kernel<kTok, false>;
  UP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmemMax));
  UP_KERNEL(kern, (p.T + kTok - 1) / kTok * kFewCluster, kFewWarps * 32, few_smem(kTok, p.M, p.d), s, p);
  return UNIPOOL_OK;
}

// Tokens to a cluster: the fewest with which all clusters run at a time (an SM takes two blocks, a GPC of 16 to 18 SMs
// four clusters; 29 of them run beside one another, of 37 some come second), 0 where that needs more than 16, and where 16
// of them do not pay: their products grow with M d, the other router's chain with d / 64, and with bf16 weights (one term;
// three otherwise) that is soon the shorter one.  Norm router, weights read from HBM, us, tensor cores with bf16 weights ->
// here (tensor cores with fp32 weights):
//   tokens         33                   150              232 / 240       464
//   64 x 512       12.0 -> 7.7 (17)     12.1 -> 8.2      12.1 -> 8.8     12.1 -> 9.9
//   96 x 768       15.6 -> 9.5 (23)     15.7 -> 10.9     15.4 -> 12.3    15.4 -> 14.2
//   384 x 768      30 -> 14.8 (41)      30 -> 16.4       30 -> 21.7      30 -> 25.7
//   192 x 1536     22.8 -> 14.5 (37)    22.7 -> 16.6     22.7 -> 18.0    22.8 [27.2 with 16 tokens to a cluster]
//   24 x 2048      18.3 -> 14.3 (38)    18.3 -> 14.7
// and at 464 tokens, 16 to a cluster, as shares of the other router's time with bf16 weights (with fp32 weights 0.5 .. 0.75):
//   width       64 experts   96     128    160    192    256    384    512
//   768         0.90         0.92   0.90   0.97   0.95   0.89   0.87   0.81
//   896         0.95         0.95   0.93   1.03   1.02   0.94   0.95   0.91
//   1024        0.95         0.96   0.95   1.05   1.05   0.98   0.98   0.96
//   1152        1.00         0.99   0.98   1.13   1.12   1.04   1.05   1.02
//   1472        1.02         1.04   1.05   1.23   1.22   1.18   1.17   1.16
// (0.02 to 0.03 less since the kernel's pointers come out of its wait; at the line, 128 x 1408 and 160, 192 x 960 measure 1.00.)
// The logits' error against 64 bits is 1.1e-7 instead of 7e-7 / 3.8e-6 (one rounding a product, no truncated sums).
int few_tokens(const unipool_ctx* ctx, int T, int M) {
  const int d = ctx->cfg.d_model, clusters = ctx->sm_count / 5;
  const int tok = T <= 8 * clusters ? 8 : T <= 16 * clusters && d <= (M <= 128 ? 1408 : 960) ? 16 : 0;
  return few_smem(tok, M, d) <= kFewSmemMax ? tok : 0;
}

}  // namespace

// (prepared weights count as they were: of those without a copy the other router has the terms)
bool route_on_few(const unipool_ctx* ctx, const float* W_r, int T, int M) {
  return few_tokens(ctx, T, M) > 0 && (ctx->prepared_now || ctx->prepared_copied || prepared_layer(ctx, W_r, M) < 0);
}

int route_few_launch(unipool_ctx* ctx, const void* x, int T, const float* W_r, float sigma, const float* bias, int M,
                     int32_t* idx, float* gate, int32_t* counts, float* score_sum, float* znorm, float* z_saved,
                     cudaStream_t s) {
  // what the tensor maps of the other router ask for, whatever the number of tokens
  UP_REQUIRE(aligned16(x) && ((M & 3) != 0 || aligned16(z_saved)), UNIPOOL_ERR_INVALID_ARG,
             "tensor base %p is not 16-byte aligned", aligned16(x) ? static_cast<const void*>(z_saved) : x);
  const int layer = ctx->prepared_now ? -1 : prepared_layer(ctx, W_r, M);
  if (layer >= 0) {
    W_r = ctx->ws.w_copy + (int64_t)layer * M * ctx->cfg.d_model;
    ctx->copy_read = true;
  }
  FewParams p{};
  p.x = static_cast<const __nv_bfloat16*>(x); p.W_r = W_r; p.bias = bias;
  p.T = T; p.M = M; p.d = ctx->cfg.d_model; p.k = ctx->cfg.top_k;
  p.sigma_c = sigma * ctx->cfg.c; p.eps = ctx->cfg.eps;
  p.idx = idx; p.gate = gate; p.znorm = znorm; p.z_saved = z_saved;
  p.totals = {counts, score_sum, ctx->ws.route_counts, reinterpret_cast<long long*>(ctx->ws.route_sums), ctx->ws.tickets + 2};
  p.vec = aligned16(W_r);
  PhaseTimer pt(ctx, UNIPOOL_PH_ROUTE_SELECT, 1, s);
  return few_tokens(ctx, T, M) == 8 ? few_launch<8>(ctx, p, s) : few_launch<16>(ctx, p, s);
}

}  // namespace unipool
