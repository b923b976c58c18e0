// Grouped SwiGLU expert FFN on CUDA cores with exact fp32 accumulation: the arithmetic path of the fp32 mode
// (parity bound 1e-5, which TF32 tensor-core products cannot meet).
#include "common.cuh"
#include "simt_gemm.cuh"

namespace unipool {

namespace {

struct RowGemm {
  const float* A; int64_t lda;                      // [rows, K]
  const float* B; int64_t b_expert, ldb;            // expert's weights: along K [N, K], across K [K, N]
  const int32_t* tile_expert; const int32_t* offsets; const int32_t* rows;   // rows: true group sizes or NULL
  int expert_base;
  float *C, *C2;
  const float* GU;
  int N, K, f, n_row_tiles;
  bool vec;                                         // every pointer is 16-byte aligned (row lengths are multiples of 64)
};

enum RowEpilogue {
  kStore,      // C [rows, N]
  kSwiglu,     // the tile is TN/2 gate and the same TN/2 up columns: GU -> C [rows, 2f], A = silu(G) U -> C2 [rows, f]
  kSwigluBwd,  // the tile is dA: dG = dA U silu'(G), dU = dA silu(G) -> C [rows, 2f], G and U from GU
};

// C = A B_e for every TM-row tile of the permuted row space; the tile's expert selects B.  Tiles at and beyond
// offsets[n_experts] are skipped (tile_expert < 0); tiles behind a group's last token hold zeros and get zeros.
template <int TM, int KG, Major BM, RowEpilogue EPI>
__global__ void __launch_bounds__(SimtTile<TM, KG>::kThreads)
grouped_rows_gemm_kernel(const RowGemm p) {
  using T = SimtTile<TM, KG>;
  constexpr int TN = kSimtN;
  extern __shared__ float4 smem_raw[];
  typename T::Smem& sm = *reinterpret_cast<typename T::Smem*>(smem_raw);
  grid_wait();
  const int n0 = blockIdx.x * (EPI == kSwiglu ? TN / 2 : TN);
  for (int rt = blockIdx.y; rt < p.n_row_tiles; rt += gridDim.y) {
    const int m0 = rt * TM;
    const int e = p.tile_expert[m0 / UNIPOOL_ROW_ALIGN];
    if (e < 0) continue;                            // uniform over the block
    const bool empty = p.rows != nullptr && m0 - p.offsets[e] >= p.rows[e];
    const float* B = p.B + (int64_t)(p.expert_base + e) * p.b_expert;
    T t;
    t.template run<kAlongK, BM>(
        sm, empty ? 0 : p.K / kSimtKC,
        [&](int c, int i, int k) { return ld4(p.A + (int64_t)(m0 + i) * p.lda + c * kSimtKC + k, p.vec); },
        [&](int c, int i, int k) {
          if (EPI == kSwiglu) i = i < TN / 2 ? n0 + i : p.f + n0 + i - TN / 2;
          else i += n0;
          const int kk = c * kSimtKC + k;
          return ld4(BM == kAlongK ? B + (int64_t)i * p.ldb + kk : B + (int64_t)kk * p.ldb + i, p.vec);
        });
    if (threadIdx.x < kSimtGroup) {
#pragma unroll
      for (int i = 0; i < T::MR; ++i) {
        const int64_t r = m0 + T::row(i);
        if constexpr (EPI == kStore) {
#pragma unroll
          for (int j = 0; j < T::NR; j += 4)
            st4(p.C + r * p.N + n0 + T::col(j),
                make_float4(t.value(i, j), t.value(i, j + 1), t.value(i, j + 2), t.value(i, j + 3)), p.vec);
        } else if constexpr (EPI == kSwiglu) {
          float g[4], u[4], a[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) { g[j] = t.value(i, j); u[j] = t.value(i, j + 4); a[j] = silu_f(g[j]) * u[j]; }
          const int n = n0 + T::col(0);
          st4(p.C + r * 2 * p.f + n, make_float4(g[0], g[1], g[2], g[3]), p.vec);
          st4(p.C + r * 2 * p.f + p.f + n, make_float4(u[0], u[1], u[2], u[3]), p.vec);
          st4(p.C2 + r * p.f + n, make_float4(a[0], a[1], a[2], a[3]), p.vec);
        } else {
#pragma unroll
          for (int j = 0; j < T::NR; j += 4) {
            const int n = n0 + T::col(j);
            const float4 g4 = ld4(p.GU + r * 2 * p.f + n, p.vec);
            const float4 u4 = ld4(p.GU + r * 2 * p.f + p.f + n, p.vec);
            const float g[4] = {g4.x, g4.y, g4.z, g4.w}, u[4] = {u4.x, u4.y, u4.z, u4.w};
            float dg[4], du[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float dA = t.value(i, j + q);
              dg[q] = dA * u[q] * silu_grad_f(g[q]);
              du[q] = dA * silu_f(g[q]);
            }
            st4(p.C + r * 2 * p.f + n, make_float4(dg[0], dg[1], dg[2], dg[3]), p.vec);
            st4(p.C + r * 2 * p.f + p.f + n, make_float4(du[0], du[1], du[2], du[3]), p.vec);
          }
        }
      }
    }
    if (gridDim.y < p.n_row_tiles) __syncthreads();  // the next tile reuses the buffers
  }
}

// dW[e][m, n] (+)= sum over the rows r of group e (of every listed layer) of P[r, m] * Q[r, n].
struct PoolGemm {
  const float* P; int ldp; const float* Q; int ldq;
  const int32_t* offsets; const int32_t* rows;      // rows [n_layers, n_experts] or NULL
  int n_experts, expert_base, n_layers; int64_t layer_stride_rows;
  float* dW; int Mdim, Ndim; bool overwrite, vec;
};

__global__ void __launch_bounds__(SimtTile<64, 2>::kThreads)
grouped_k_gemm_kernel(const PoolGemm p) {
  using T = SimtTile<64, 2>;
  __shared__ typename T::Smem sm;
  grid_wait();
  const int m0 = blockIdx.x * 64, n0 = blockIdx.y * 64, e = blockIdx.z;
  auto rows_of = [&](int l) {
    const int32_t* off = p.offsets + (int64_t)l * (p.n_experts + 1) + e;
    return p.rows ? min(p.rows[(int64_t)l * p.n_experts + e], off[1] - off[0]) : off[1] - off[0];
  };
  int n_chunks = 0;
  for (int l = 0; l < p.n_layers; ++l) n_chunks += (rows_of(l) + kSimtKC - 1) / kSimtKC;
  // the chunk being fetched: rows [row0, row0 + left) of its layer are still to come (a group asks for its chunks in order)
  int layer = -1, at = -1, left = 0;
  int64_t row0 = 0;
  auto seek = [&](int c) {
    for (; at < c; ++at) {
      row0 += kSimtKC;
      left -= kSimtKC;
      while (left <= 0) {
        ++layer;
        left = rows_of(layer);
        row0 = layer * p.layer_stride_rows + p.offsets[(int64_t)layer * (p.n_experts + 1) + e];
      }
    }
  };
  T t;
  t.template run<kAcrossK, kAcrossK>(
      sm, n_chunks,
      [&](int c, int i, int k) {
        seek(c);
        return k < left ? ld4(p.P + (row0 + k) * p.ldp + m0 + i, p.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      },
      [&](int c, int i, int k) {
        return k < left ? ld4(p.Q + (row0 + k) * p.ldq + n0 + i, p.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      });
  if (threadIdx.x >= kSimtGroup) return;
  float* out = p.dW + (int64_t)(p.expert_base + e) * p.Mdim * p.Ndim;
#pragma unroll
  for (int i = 0; i < T::MR; ++i)
#pragma unroll
    for (int j = 0; j < T::NR; j += 4) {
      float* o = out + (int64_t)(m0 + T::row(i)) * p.Ndim + n0 + T::col(j);
      float4 v = make_float4(t.value(i, j), t.value(i, j + 1), t.value(i, j + 2), t.value(i, j + 3));
      if (!p.overwrite) {
        v = make_float4(v.x + o[0], v.y + o[1], v.z + o[2], v.w + o[3]);
      }
      st4(o, v, p.vec);
    }
}

template <int TM, int KG, Major BM, RowEpilogue EPI>
int rows_gemm_as(const unipool_ctx* ctx, RowGemm p, cudaStream_t s) {
  auto kern = grouped_rows_gemm_kernel<TM, KG, BM, EPI>;
  constexpr int smem = (int)sizeof(typename SimtTile<TM, KG>::Smem);
  if (smem > 48 * 1024) UP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  p.n_row_tiles = (int)(ctx->row_capacity / TM);
  const int gy = p.n_row_tiles < 8192 ? p.n_row_tiles : 8192;
  UP_KERNEL(kern, dim3(p.N / (EPI == kSwiglu ? kSimtN / 2 : kSimtN), gy), (SimtTile<TM, KG>::kThreads), smem, s, p);
  return UNIPOOL_OK;
}

template <Major BM, RowEpilogue EPI>
int rows_gemm(unipool_ctx* ctx, RowGemm p, int n_experts, cudaStream_t s) {
  p.vec = aligned16(p.A, p.B, p.C, p.C2, p.GU);    // those that the epilogue has not are NULL
  // 64 x 64 tiles of a full batch (a group ends on half a tile).  Many: whole tiles, one group of threads on each, two
  // on a long contraction; fewer: two groups, and half tiles where the weights are read across K; few: half tiles,
  // two or four groups.  In us, TM = 64 with 1 / 2 / 4 groups, 32 with 1 / 2 / 4 (16 experts of 256 x 512, 64 rows each):
  // gate/up (384 tiles) 46/41/57, 45/41/44; down (96) 44/29/27, 35/30/27; dgrad down (192) 48/45/63, 39/36/42; dgrad
  // gate/up (96) 82/48/40, 63/49/44; 24 experts of 384 x 768, 250 rows: 2544 tiles 208/210/345, 252/255/279; 636 tiles
  // 137/119/167, 156/155/141; 1272 tiles 145/157/303, 153/154/201.
  const int64_t tiles = ((int64_t)ctx->cfg.max_tokens * ctx->cfg.top_k / 64 + n_experts / 2) *
                        (p.N / (EPI == kSwiglu ? kSimtN / 2 : kSimtN));
  if (tiles >= 600)
    return p.K >= 768 ? rows_gemm_as<64, 2, BM, EPI>(ctx, p, s) : rows_gemm_as<64, 1, BM, EPI>(ctx, p, s);
  if (tiles >= 350 && BM == kAlongK) return rows_gemm_as<64, 2, BM, EPI>(ctx, p, s);
  return p.K >= 512 ? rows_gemm_as<32, 4, BM, EPI>(ctx, p, s) : rows_gemm_as<32, 2, BM, EPI>(ctx, p, s);
}

template <typename Args>
RowGemm row_gemm(const unipool_ctx* ctx, const Args& a) {
  RowGemm p{};
  p.tile_expert = a.tile_expert;
  p.offsets = a.offsets;
  p.rows = a.rows;
  p.expert_base = a.expert_base;
  p.f = ctx->cfg.d_ff;
  p.b_expert = (int64_t)ctx->cfg.d_model * ctx->cfg.d_ff;
  return p;
}

}  // namespace

int expert_fwd_simt(unipool_ctx* ctx, const ExpertFwdArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff;
  {
    PhaseTimer pt(ctx, UNIPOOL_PH_EXPERT_FWD_GU, 1, s);
    RowGemm p = row_gemm(ctx, a);                    // GU = Xp W_gu[e]^T, A = silu(G) U
    p.A = static_cast<const float*>(a.Xp); p.lda = d; p.K = d;
    p.B = static_cast<const float*>(a.W_gu); p.b_expert *= 2; p.ldb = d; p.N = f;
    p.C = static_cast<float*>(a.GU); p.C2 = static_cast<float*>(a.A);
    const int rc = rows_gemm<kAlongK, kSwiglu>(ctx, p, a.n_experts, s);
    if (rc != UNIPOOL_OK) return rc;
  }
  PhaseTimer pt(ctx, UNIPOOL_PH_EXPERT_FWD_DOWN, 1, s);
  RowGemm p = row_gemm(ctx, a);                      // Yp = A W_down[e]^T
  p.A = static_cast<const float*>(a.A); p.lda = f; p.K = f;
  p.B = static_cast<const float*>(a.W_down); p.ldb = f; p.N = d;
  p.C = static_cast<float*>(a.Yp);
  return rows_gemm<kAlongK, kStore>(ctx, p, a.n_experts, s);
}

int pool_wgrad_simt(unipool_ctx* ctx, const PoolWgradArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff;
  PoolGemm p{};
  p.offsets = a.offsets; p.rows = a.rows;
  p.n_experts = a.n_experts; p.expert_base = a.expert_base;
  p.n_layers = a.n_layers; p.layer_stride_rows = a.layer_stride_rows;
  p.overwrite = a.overwrite;
  if (a.dW_down != nullptr) {                        // dW_down[e] [d, f] (+)= dYp_e^T A_e
    PhaseTimer pt(ctx, UNIPOOL_PH_WGRAD_DOWN, 1, s);
    p.P = static_cast<const float*>(a.dYp); p.ldp = d;
    p.Q = static_cast<const float*>(a.A); p.ldq = f;
    p.dW = a.dW_down; p.Mdim = d; p.Ndim = f; p.vec = aligned16(p.P, p.Q, p.dW);
    UP_KERNEL(grouped_k_gemm_kernel, dim3(d / 64, f / 64, a.n_experts), (SimtTile<64, 2>::kThreads), 0, s, p);
  }
  if (a.dW_gu == nullptr) return UNIPOOL_OK;
  PhaseTimer pt(ctx, UNIPOOL_PH_WGRAD_GU, 1, s);     // dW_gu[e] [2f, d] (+)= dGU_e^T Xp_e
  p.P = static_cast<const float*>(a.dGU); p.ldp = 2 * f;
  p.Q = static_cast<const float*>(a.Xp); p.ldq = d;
  p.dW = a.dW_gu; p.Mdim = 2 * f; p.Ndim = d; p.vec = aligned16(p.P, p.Q, p.dW);
  UP_KERNEL(grouped_k_gemm_kernel, dim3(2 * f / 64, d / 64, a.n_experts), (SimtTile<64, 2>::kThreads), 0, s, p);
  return UNIPOOL_OK;
}

int expert_bwd_simt(unipool_ctx* ctx, const ExpertBwdArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff;
  {
    PhaseTimer pt(ctx, UNIPOOL_PH_DGRAD_DOWN, 1, s);
    RowGemm p = row_gemm(ctx, a);                    // dA = dYp W_down[e], then dG, dU
    p.A = static_cast<const float*>(a.dYp); p.lda = d; p.K = d;
    p.B = static_cast<const float*>(a.W_down); p.ldb = f; p.N = f;
    p.C = static_cast<float*>(a.dGU); p.GU = static_cast<const float*>(a.GU);
    const int rc = rows_gemm<kAcrossK, kSwigluBwd>(ctx, p, a.n_experts, s);
    if (rc != UNIPOOL_OK) return rc;
  }
  {
    PhaseTimer pt(ctx, UNIPOOL_PH_DGRAD_GU, 1, s);
    RowGemm p = row_gemm(ctx, a);                    // dXp = dGU W_gu[e]
    p.A = static_cast<const float*>(a.dGU); p.lda = 2 * f; p.K = 2 * f;
    p.B = static_cast<const float*>(a.W_gu); p.b_expert *= 2; p.ldb = d; p.N = d;
    p.C = static_cast<float*>(a.dXp);
    const int rc = rows_gemm<kAcrossK, kStore>(ctx, p, a.n_experts, s);
    if (rc != UNIPOOL_OK) return rc;
  }
  if (!a.wgrad) return UNIPOOL_OK;
  PoolWgradArgs w{1, 0, a.offsets, a.Xp, a.A, a.dYp, a.dGU, a.expert_base, a.n_experts, a.dW_gu, a.dW_down,
                  a.overwrite, a.rows};
  return pool_wgrad_simt(ctx, w, s);
}

}  // namespace unipool
