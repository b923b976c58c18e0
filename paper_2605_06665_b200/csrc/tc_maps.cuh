// Grouped-GEMM modes and the tensor maps of the tcgen05 kernels (defined in expert_tc.cu).
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace unipool {

enum Mode : int {
  kFwd1 = 0,    // GU = Xp W_gu^T, A = silu(G)*U        A K-major, B K-major (3-D map), row tiles
  kFwd2 = 1,    // Yp = A W_down^T                      A K-major, B K-major,           row tiles
  kDgrad1 = 2,  // dGU = swiglu'(dYp W_down, GU)        A K-major, B MN-major,          row tiles
  kDgrad2 = 3,  // dXp = dGU W_gu                       A K-major, B MN-major,          row tiles
  kWgrad = 4,   // dW[e] (+)= P_e^T Q_e                 A MN-major, B MN-major,         ragged K
};

constexpr int kWmMaxExperts = 400;        // experts of a launch of the weights-on-M kernels (their shared-memory table)

enum MapKind { kMapOperand, kMapBf16Chunk, kMapF32Chunk };
int make_tmap(const unipool_ctx* ctx, CUtensorMap* out, MapKind kind, const void* base, int rank,
              const uint64_t* dims, const uint64_t* strides_elems, const uint32_t* box);
int map_2d(const unipool_ctx* ctx, CUtensorMap* out, const void* base, uint64_t cols, uint64_t rows,
           uint32_t box_cols, uint32_t box_rows, MapKind kind = kMapOperand);
int map_mn(const unipool_ctx* ctx, CUtensorMap* out, const void* base, uint64_t n_cols, uint64_t k_rows,
           uint32_t blocks, uint32_t k_box = 64);

}  // namespace unipool
