// Grouped SwiGLU expert FFN on CUDA cores with exact fp32 accumulation: the arithmetic path of the fp32 mode
// (parity bound 1e-5, which TF32 tensor-core products cannot meet).
#include "common.cuh"
#include "simt_gemm.cuh"

namespace unipool {

namespace {

struct RowGemm {
  const float* A; int64_t lda;                      // [rows, K]
  const float* B; int64_t b_expert, ldb;            // expert's weights: along K [N, K], across K [K, N]
  const int32_t* offsets; const int32_t* rows;      // [n_experts + 1]; [n_experts] true group sizes or NULL
  int n_experts, expert_base;
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

// The expert and first row of row tile t, and whether it lies behind the group's last token; false: no such tile.  Tiles
// with tokens are numbered first, so that the blocks that have work, one after the other, fall evenly on the SMs: numbered
// as they lie in memory, with the tiles of the 128-row padding between them, some SMs had three blocks with work and some
// none (SMs active for half of the 39 us of dgrad gate/up, 16 experts of 256 x 512, 64 rows each).
template <int kRows>
__device__ __forceinline__ bool find_row_tile(const RowGemm& p, int t, int* expert, int* row, bool* empty) {
  const int lane = threadIdx.x % 32;
  auto search = [&](bool pads, int base) {            // every warp for itself; returns the tiles counted
    for (int e0 = 0; e0 < p.n_experts; e0 += 32) {
      const int e = e0 + lane;
      int first = 0, n = 0;
      if (e < p.n_experts) {
        first = p.offsets[e];
        const int all = (p.offsets[e + 1] - first) / kRows;
        const int live = p.rows ? min((max(p.rows[e], 0) + kRows - 1) / kRows, all) : all;
        n = pads ? all - live : live;
        if (pads) first += live * kRows;
      }
      int upto = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += v;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, t < base + upto);
      if (hit != 0) {
        const int src = __ffs(hit) - 1;
        *expert = e0 + src;
        *row = __shfl_sync(0xffffffffu, first + (t - base - (upto - n)) * kRows, src);
        *empty = pads;
        return -1;
      }
      base += __shfl_sync(0xffffffffu, upto, 31);
    }
    return base;
  };
  const int live = search(false, 0);
  return live < 0 || search(true, live) < 0;
}

// C = A B_e for every row tile of the groups; tiles behind a group's last token hold zeros and get zeros.
template <typename T, Major BM, RowEpilogue EPI>
__global__ void __launch_bounds__(T::kThreads, T::kBlocks)
grouped_rows_gemm_kernel(RowGemm p) {
  grid_wait(p.A, p.B, p.GU);
  constexpr int TN = kSimtN, kHalf = TN / 2;
  extern __shared__ float4 smem_raw[];
  typename T::Smem& sm = *reinterpret_cast<typename T::Smem*>(smem_raw);
  const int n0 = blockIdx.x * (EPI == kSwiglu ? kHalf : TN);
  for (int rt = blockIdx.y; rt < p.n_row_tiles; rt += gridDim.y) {
    int e, m0;
    bool empty;
    if (!find_row_tile<T::kRows>(p, rt, &e, &m0, &empty)) break;   // uniform over the block
    const float* B = p.B + (int64_t)(p.expert_base + e) * p.b_expert;
    T t;
    t.template run<kAlongK, BM>(
        sm, empty ? 0 : p.K / kSimtKC, p.vec, p.vec, p.A, [](int) {},
        [&](int c, int i, int k) { return p.A + (int64_t)(m0 + i) * p.lda + c * kSimtKC + k; },
        [&](int c, int i, int k) {
          if (EPI == kSwiglu) i = i < kHalf ? n0 + i : p.f + n0 + i - kHalf;
          else i += n0;
          const int kk = c * kSimtKC + k;
          return BM == kAlongK ? B + (int64_t)i * p.ldb + kk : B + (int64_t)kk * p.ldb + i;
        });
    if constexpr (EPI == kStore) {
      t.each4(sm, [&](int i, int j, float4 v) { st4(p.C + (int64_t)(m0 + i) * p.N + n0 + j, v, p.vec); });
    } else if constexpr (EPI == kSwiglu) {
      t.each4_halves(sm, [&](int i, int j, float4 v, float4 u) {
        const int64_t r = m0 + i;
        const int n = n0 + j;
        st4(p.C + r * 2 * p.f + n, v, p.vec);
        st4(p.C + r * 2 * p.f + p.f + n, u, p.vec);
        st4(p.C2 + r * p.f + n, make_float4(silu_f(v.x) * u.x, silu_f(v.y) * u.y, silu_f(v.z) * u.z, silu_f(v.w) * u.w), p.vec);
      });
    } else {
      t.each4(sm, [&](int i, int j, float4 v) {
        const int64_t r = m0 + i;
        const int n = n0 + j;
        const float4 g = ld4(p.GU + r * 2 * p.f + n, p.vec), u = ld4(p.GU + r * 2 * p.f + p.f + n, p.vec);
        st4(p.C + r * 2 * p.f + n,
            make_float4(v.x * u.x * silu_grad_f(g.x), v.y * u.y * silu_grad_f(g.y), v.z * u.z * silu_grad_f(g.z),
                        v.w * u.w * silu_grad_f(g.w)), p.vec);
        st4(p.C + r * 2 * p.f + p.f + n,
            make_float4(v.x * silu_f(g.x), v.y * silu_f(g.y), v.z * silu_f(g.z), v.w * silu_f(g.w)), p.vec);
      });
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

// Tiles of 64 x 64, two groups to each.  us of dW_down, dW_gu with warp tiles of two warps / block tiles: 16 experts of 256 x
// 512, 64 rows 19/19, 29/25; 24 of 384 x 768, 250 rows 103/93, 195/174, very uneven groups 178/159, 306/220; 96 of 768 x 2048,
// 341 rows 2590/2290, 5150/4560; misaligned, 24 of 384 x 768 155/101, 297/192.  (One group: a quarter slower where an expert has
// many rows and few tiles.)
using WgradTile = SimtBlockTile<2>;

__global__ void __launch_bounds__(WgradTile::kThreads, WgradTile::kBlocks)
grouped_k_gemm_kernel(PoolGemm p) {
  grid_wait(p.P, p.Q);
  using T = WgradTile;
  extern __shared__ float4 smem_raw[];
  T::Smem& sm = *reinterpret_cast<T::Smem*>(smem_raw);
  const int m0 = blockIdx.x * T::kRows, n0 = blockIdx.y * kSimtN, e = blockIdx.z;
  auto rows_of = [&](int l) {
    const int32_t* off = p.offsets + (int64_t)l * (p.n_experts + 1) + e;
    return p.rows ? min(p.rows[(int64_t)l * p.n_experts + e], off[1] - off[0]) : off[1] - off[0];
  };
  int n_chunks = 0;
  for (int l = 0; l < p.n_layers; ++l) n_chunks += (rows_of(l) + kSimtKC - 1) / kSimtKC;
  // the chunk being fetched: rows [row0, row0 + left) of its layer are still to come (a warp asks for its chunks in order)
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
  t.run<kAcrossK, kAcrossK>(
      sm, n_chunks, p.vec, p.vec, p.P, seek,
      [&](int, int i, int k) -> const float* { return k < left ? p.P + (row0 + k) * p.ldp + m0 + i : nullptr; },
      [&](int, int i, int k) -> const float* { return k < left ? p.Q + (row0 + k) * p.ldq + n0 + i : nullptr; });
  float* out = p.dW + (int64_t)(p.expert_base + e) * p.Mdim * p.Ndim;
  t.each4(sm, [&](int i, int j, float4 v) {
    float* o = out + (int64_t)(m0 + i) * p.Ndim + n0 + j;
    if (!p.overwrite) {
      const float4 w = p.vec ? *reinterpret_cast<const float4*>(o) : make_float4(o[0], o[1], o[2], o[3]);
      v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
    }
    st4(o, v, p.vec);
  });
}

template <typename T, Major BM, RowEpilogue EPI>
int rows_gemm_as(const unipool_ctx* ctx, RowGemm p, cudaStream_t s) {
  auto kern = grouped_rows_gemm_kernel<T, BM, EPI>;
  constexpr int smem = (int)sizeof(typename T::Smem);
  UP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  p.n_row_tiles = (int)(ctx->row_capacity / T::kRows);
  const int gy = p.n_row_tiles < 8192 ? p.n_row_tiles : 8192;
  UP_KERNEL(kern, dim3(p.N / (EPI == kSwiglu ? kSimtN / 2 : kSimtN), gy), T::kThreads, smem, s, p);
  return UNIPOOL_OK;
}

template <Major BM, RowEpilogue EPI>
int rows_gemm(unipool_ctx* ctx, RowGemm p, int n_experts, cudaStream_t s) {
  p.vec = aligned16(p.A, p.B, p.C, p.C2, p.GU);    // those that the epilogue has not are NULL
  const int64_t rows = (int64_t)ctx->cfg.max_tokens * ctx->cfg.top_k;
  const int64_t tiles = (rows / kSimtM + n_experts / 2) * (p.N / (EPI == kSwiglu ? kSimtN / 2 : kSimtN));
  // Block tiles, by the tiles (of 32 rows) of a full batch, where groups average at least three of them: of fewer rows the
  // 64-row tiles multiply a third more padding.  From a contraction of 768 on (256 where nothing but it is left to share)
  // two groups share a tile.  Misaligned operands earlier and whatever the rows: they cost 4-byte copies.  us, warp tiles
  // (by the rule below) / block tiles with one / two groups:
  //   16 of 512 x 1024, 512 rows    gate/up (8448 tiles) 459/406/428   down (2112) 249/227/227   dgrad down (4224) 264/242/259   dgrad gate/up (2112) 461/441/431
  //   96 of 768 x 2048, 341 rows    (68608) 5130/4751/5010   (12864) 2520/2370/2460   (34304) 2940/2420/2650   (12864) 5220/4640/4680
  //   24 of 384 x 768, 250 rows     (4776) 219/194/195   (1194) 113/126/112   (2388) 129/134/148   (1194) 213/246/208
  //   32 of 192 x 768, 500 rows     (12384) 270/243/263   (1548) 140/132/133   (6192) 196/178/238   (1548) 259/252/248
  //   96 of 768 x 2048, 85 rows     (19456) 1470/1640/1730   (3648) 707/844/858   (9728) 886/861/957   (3648) 1460/1670/1650
  //   misaligned, 24 of 384 x 768   (4776) 343/257/250   (1194) 170/142/140   (2388) 166/155/164   (1194) 285/267/239
  const bool large = tiles >= (EPI == kSwigluBwd ? (p.vec ? 3000 : 2000) : EPI == kSwiglu || p.vec ? 1500 : 700);
  if (large && (!p.vec || rows >= (int64_t)3 * kSimtM * n_experts))
    return p.K >= (EPI == kStore ? 256 : 768) ? rows_gemm_as<SimtBlockTile<2>, BM, EPI>(ctx, p, s)
                                              : rows_gemm_as<SimtBlockTile<1>, BM, EPI>(ctx, p, s);
  // Warps to a warp tile (a contraction of 768 and more is at least two sums).  us with 1 / 2 / 4 / 8 warps, and with 64 x 64
  // tiles of two groups:
  //   16 experts of 256 x 512, 64 rows      gate/up (640 tiles) 39/31/29/38, 35  down (160) 39/23/21/19, 23
  //                                         dgrad down (320) 44/29/22/25, 32     dgrad gate/up (160) 75/40/36/32, 39
  //   32 of 256 x 704, 14 rows              (660) 43/41/45/74, 71   (120) 52/30/27/19, 33   (330) 45/38/39/53, 54   (120) 102/54/47/28, 56
  //   15 of 384 x 512, 91 rows              (800) 56/45/46/53, 56   (300) 40/35/28/28, 31   (400) 52/38/27/32, 41   (300) 76/66/50/48, 53
  //   64 of 192 x 128, 250 rows             dgrad down (1064) 53/53/47/56, 67
  // Eight against four over ten more stacks of 8 to 40 experts: 0.59 to 0.99 of the time at 114 to 153 tiles and K from 256, 0.98 to 1.06
  // from 165 tiles on.  Two against four in gate/up of 820 to 1820 tiles, K < 256: 0.91 to 1.01.
  if (10 * tiles <= 11 * ctx->sm_count && p.K >= (tiles <= ctx->sm_count ? 256 : 512))
    return rows_gemm_as<SimtTile<8>, BM, EPI>(ctx, p, s);
  if constexpr (BM == kAlongK) {
    if (tiles >= 1500 && p.K < 768) return rows_gemm_as<SimtTile<1>, BM, EPI>(ctx, p, s);
    if (tiles >= 1500 || (tiles >= 600 && (p.K < 256 || rows < (int64_t)kSimtM * n_experts)))
      return rows_gemm_as<SimtTile<2>, BM, EPI>(ctx, p, s);
  }
  return rows_gemm_as<SimtTile<4>, BM, EPI>(ctx, p, s);
}

int k_gemm(const PoolGemm& p, cudaStream_t s) {
  UP_CUDA(cudaFuncSetAttribute(grouped_k_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WgradTile::Smem)));
  UP_KERNEL(grouped_k_gemm_kernel, dim3(p.Mdim / WgradTile::kRows, p.Ndim / kSimtN, p.n_experts), WgradTile::kThreads,
            sizeof(WgradTile::Smem), s, p);
  return UNIPOOL_OK;
}

template <typename Args>
RowGemm row_gemm(const unipool_ctx* ctx, const Args& a) {
  RowGemm p{};
  p.offsets = a.offsets;
  p.rows = a.rows;
  p.n_experts = a.n_experts;
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
    const int rc = k_gemm(p, s);
    if (rc != UNIPOOL_OK) return rc;
  }
  if (a.dW_gu == nullptr) return UNIPOOL_OK;
  PhaseTimer pt(ctx, UNIPOOL_PH_WGRAD_GU, 1, s);     // dW_gu[e] [2f, d] (+)= dGU_e^T Xp_e
  p.P = static_cast<const float*>(a.dGU); p.ldp = 2 * f;
  p.Q = static_cast<const float*>(a.Xp); p.ldq = d;
  p.dW = a.dW_gu; p.Mdim = 2 * f; p.Ndim = d; p.vec = aligned16(p.P, p.Q, p.dW);
  return k_gemm(p, s);
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
