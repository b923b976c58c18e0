// CUDA-core tiled GEMM building block with fp32 accumulation, for the fp32 mode of the library (its 1e-5
// parity bound rules out TF32).
//
// Bound by the FMA pipe (72 TFLOP/s at 1.9 GHz) and the register side of shared memory where there are many tiles
// (40 TFLOP/s in the weight gradient of 24 experts of 384 x 768), by latency and synchronisation below that.  A group
// of 64 threads owns a TM x 64 tile, TM / 8 x 8 results per thread, multiplied with packed fma.rn.f32x2 (each half an
// IEEE fp32 fma: half the instructions for the same sums); chunks of 16 of the contraction go through
// double-buffered shared memory, fetched into registers one chunk ahead with 16-byte loads, and the operands of
// step k + 1 are read while step k is multiplied.  KG such groups in a block share a tile by taking every KG-th
// chunk and add up at the end: a long contraction over few tiles then still fills the chip.  (Both operands along K
// in shared memory, pairs along K, saves the duplication of a: no faster, and slower by a third where a weight is
// read across K.)
#pragma once

#include "common.cuh"

namespace unipool {

constexpr int kSimtKC = 16;        // k-chunk staged in shared memory
constexpr int kSimtGroup = 64;     // threads of a k-group: 8 x 8
constexpr int kSimtN = 64;         // columns of a tile

// How an operand lies in memory: kAlongK element (i, k) = p[i * ld + k], kAcrossK element (i, k) = p[k * ld + i].
enum Major { kAlongK, kAcrossK };

// Four floats at p; `vec`: p is 16-byte aligned.
__device__ __forceinline__ float4 ld4(const float* p, bool vec) {
  return vec ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
__device__ __forceinline__ void st4(float* p, float4 v, bool vec) {
  if (vec) { *reinterpret_cast<float4*>(p) = v; return; }
  p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w;
}
// The first n (<= 4, may be negative) floats at p, zeros for the rest.
__device__ __forceinline__ float4 ld4(const float* p, bool vec, int n) {
  if (n >= 4) return ld4(p, vec);
  return make_float4(n > 0 ? __ldg(p) : 0.f, n > 1 ? __ldg(p + 1) : 0.f, n > 2 ? __ldg(p + 2) : 0.f, 0.f);
}
template <typename... P> inline bool aligned16(P... p) { return ((... | reinterpret_cast<uintptr_t>(p)) & 15) == 0; }

template <int TM, int KG>
struct SimtTile {
  static constexpr int TN = kSimtN, MR = TM / 8, NR = 8, kThreads = KG * kSimtGroup;
  static constexpr int kA4 = TM * kSimtKC / 4 / kSimtGroup, kB4 = TN * kSimtKC / 4 / kSimtGroup;   // float4 per thread
  static_assert(MR == 8 || MR == 4, "result tile of a thread");
  struct Smem {
    float a[KG][2][kSimtKC][TM + 4];
    float b[KG][2][kSimtKC][TN + 4];
  };
  unsigned long long acc[MR][NR / 2];

  // results of this thread: row(i), column(j) inside the tile
  __device__ static int ty() { return (threadIdx.x % kSimtGroup) / 8; }
  __device__ static int tx() { return threadIdx.x % 8; }
  __device__ static int row(int i) { return i < 4 ? ty() * 4 + i : TM / 2 + ty() * 4 + i - 4; }
  __device__ static int col(int j) { return j < 4 ? tx() * 4 + j : TN / 2 + tx() * 4 + j - 4; }
  __device__ float value(int i, int j) const {
    const unsigned long long v = acc[i][j / 2];
    return __uint_as_float(j & 1 ? (uint32_t)(v >> 32) : (uint32_t)v);
  }

  // One operand's chunk: registers <- memory (fetch: float4 at (i, k) for this thread's pieces) and shared
  // memory <- registers.
  template <Major MJ, int T, int N4, typename F>
  __device__ static void fetch(float4 (&r)[N4], F at) {
#pragma unroll
    for (int q = 0; q < N4; ++q) {
      const int p = threadIdx.x % kSimtGroup + q * kSimtGroup;
      r[q] = MJ == kAlongK ? at(p / (kSimtKC / 4), p % (kSimtKC / 4) * 4) : at(p % (T / 4) * 4, p / (T / 4));
    }
  }
  template <Major MJ, int T, int N4>
  __device__ static void stash(float (*s)[T + 4], const float4 (&r)[N4]) {
#pragma unroll
    for (int q = 0; q < N4; ++q) {
      const int p = threadIdx.x % kSimtGroup + q * kSimtGroup;
      if (MJ == kAlongK) {
        const int i = p / (kSimtKC / 4), k = p % (kSimtKC / 4) * 4;
        s[k][i] = r[q].x; s[k + 1][i] = r[q].y; s[k + 2][i] = r[q].z; s[k + 3][i] = r[q].w;
      } else {
        *reinterpret_cast<float4*>(&s[p / (T / 4)][p % (T / 4) * 4]) = r[q];
      }
    }
  }
  struct Frag { float a[MR]; unsigned long long b[NR / 2]; };
  __device__ static void read(Frag& f, const float (*sa)[TM + 4], const float (*sb)[TN + 4], int k) {
#pragma unroll
    for (int h = 0; h < MR / 4; ++h) {
      const float4 v = *reinterpret_cast<const float4*>(&sa[k][h * (TM / 2) + ty() * 4]);
      f.a[4 * h] = v.x; f.a[4 * h + 1] = v.y; f.a[4 * h + 2] = v.z; f.a[4 * h + 3] = v.w;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&sb[k][h * (TN / 2) + tx() * 4]);
      f.b[2 * h] = v.x; f.b[2 * h + 1] = v.y;
    }
  }

  // The tile's sums over n_chunks chunks.  a_at / b_at(chunk, i, k): the float4 of the operand that starts at tile
  // row (column) i and position k of the chunk, zeros outside - four along K or four along i by its Major.
  // On return group 0 holds the sums of all groups (the others may leave).
  template <Major AM, Major BM, typename FA, typename FB>
  __device__ void run(Smem& s, int n_chunks, FA a_at, FB b_at) {
    const int g = threadIdx.x / kSimtGroup;
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
      for (int j = 0; j < NR / 2; ++j) acc[i][j] = 0ull;
    const int n_it = (n_chunks + KG - 1) / KG;
    float4 ra[kA4], rb[kB4];
    auto load = [&](int it) {
      const int c = it * KG + g;
      if (c < n_chunks) {
        fetch<AM, TM>(ra, [&](int i, int k) { return a_at(c, i, k); });
        fetch<BM, TN>(rb, [&](int i, int k) { return b_at(c, i, k); });
      } else {
#pragma unroll
        for (int q = 0; q < kA4; ++q) ra[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < kB4; ++q) rb[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    if (n_it > 0) load(0);
    for (int it = 0; it < n_it; ++it) {
      float (*sa)[TM + 4] = s.a[g][it & 1];
      float (*sb)[TN + 4] = s.b[g][it & 1];
      stash<AM, TM>(sa, ra);
      stash<BM, TN>(sb, rb);
      __syncthreads();                             // also: everyone is done with the buffer the next chunk goes to
      if (it + 1 < n_it) load(it + 1);
      Frag f[2];
      read(f[0], sa, sb, 0);
#pragma unroll
      for (int k = 0; k < kSimtKC; ++k) {
        if (k + 1 < kSimtKC) read(f[(k + 1) & 1], sa, sb, k + 1);
        const Frag& c = f[k & 1];
#pragma unroll
        for (int i = 0; i < MR; ++i) {
          unsigned long long aa;
          asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(c.a[i]));
#pragma unroll
          for (int j = 0; j < NR / 2; ++j) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(aa), "l"(c.b[j]));
        }
      }
    }
    if constexpr (KG > 1) {                        // groups 1 .. KG-1 hand their sums over through shared memory
      __syncthreads();
      constexpr int kSums = MR * NR / 2;
      unsigned long long* x = reinterpret_cast<unsigned long long*>(&s);
      static_assert(sizeof(Smem) >= (KG - 1) * kSums * kSimtGroup * 8, "room for the groups' sums");
      const int t = threadIdx.x % kSimtGroup;
      if (g > 0) {
#pragma unroll
        for (int q = 0; q < kSums; ++q) x[((g - 1) * kSums + q) * kSimtGroup + t] = acc[q / (NR / 2)][q % (NR / 2)];
      }
      __syncthreads();
      if (g == 0) {
        for (int o = 0; o < KG - 1; ++o)
#pragma unroll
          for (int q = 0; q < kSums; ++q)
            asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[q / (NR / 2)][q % (NR / 2)]) : "l"(x[(o * kSums + q) * kSimtGroup + t]));
      }
    }
  }
};

}  // namespace unipool
