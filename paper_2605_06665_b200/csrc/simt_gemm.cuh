// CUDA-core tiled GEMM building block with fp32 accumulation, for the fp32 mode of the library (its 1e-5
// parity bound rules out TF32).
//
// A warp owns a 32 x 64 tile, 8 x 8 results per lane, and works on its own: its chunks of 16 positions of the contraction
// come by cp.async into shared memory of its own, so that nothing in the loop waits for another warp.  An operand lies
// there as in memory, so that all copies and loads are 16 bytes wide.  KG warps share a tile by taking every KG-th
// chunk; their sums meet in shared memory, and all of them write.
// Bound by the FMA pipe and, as high, the register side of shared memory (8 x 8 results: 64 bytes a lane for 64 products,
// 128 bytes a clock), in fact by how few warps a launch of the fp32 sizes gives a scheduler: one alone issues in 57 % of
// its clocks, three in 72 %, three quarters of it FMAs.  Four positions unrolled twice: all sixteen miss the instruction
// cache, and their loads, moved up, take 255 registers.  Plain FMAs: packed ones (fma.rn.f32x2) keep the pipe twice as long
// and cost about one register move each, which pays only where issue slots run out (the block tile below).  32 x 128 tiles
// load less per product, and were no faster for their fewer warps.
#pragma once

#include "common.cuh"

namespace unipool {

constexpr int kSimtKC = 16;                   // positions of a chunk
constexpr int kSimtM = 32, kSimtN = 64;       // rows and columns of a tile
constexpr int kSimtLd = kSimtN + 8;           // row stride of the sums in shared memory

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
template <typename... P> inline bool aligned16(P... p) { return ((... | reinterpret_cast<uintptr_t>(p)) & 15) == 0; }

// kBytes at `src` into shared memory, zeros where src is NULL (`any`: some readable address).
template <int kBytes>
__device__ __forceinline__ void copy_async(uint32_t dst, const float* src, const float* any) {
  const float* from = src ? src : any;
  const int n = src ? kBytes : 0;
  if constexpr (kBytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" : : "r"(dst), "l"(from), "r"(n) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" : : "r"(dst), "l"(from), "r"(n) : "memory");
}

// Twelve warps on an SM.  (168 registers: the forward GEMMs of one to four warps spill 12 to 28 bytes.)
template <int KG>
struct SimtTile {
  static constexpr int kStages = 3;                // chunks in shared memory
  static constexpr int kRows = kSimtM, kThreads = KG * 32, kBlocks = 12 / KG;
  struct Stage { float a[kSimtM * kSimtKC], b[kSimtN * kSimtKC]; };
  union Warp { Stage stage[kStages]; float sums[kSimtM * kSimtLd]; };
  struct Smem { Warp w[KG]; };

  // Byte offset of element (i, k) of an operand of T rows.  Along K: rows of 64 bytes, their 16-byte pieces exchanged so
  // that eight rows' pieces of one k lie in different banks.
  template <Major MJ, int T> __device__ static uint32_t at(int i, int k) {
    return MJ == kAlongK ? (uint32_t)(i * 64 + (((k >> 2) ^ (i >> 1)) & 3) * 16 + (k & 3) * 4) : (uint32_t)(k * T + i) * 4;
  }
  // Row (column) j of a lane's eight; u: ty (tx), of kLanes.
  template <Major MJ, int kLanes> __device__ static int own(int u, int j) {
    return MJ == kAlongK ? u + kLanes * j : u * 4 + (j & 3) + (j >> 2) * 4 * kLanes;
  }

  // A chunk of one operand of T rows.  src(i, k): the address of its element, NULL outside; with `vec` that of four, along
  // K or along the rows as memory has them.
  template <Major MJ, int T, typename F>
  __device__ static void fetch(uint32_t dst, bool vec, const float* any, F src) {
    const int lane = threadIdx.x % 32;
    if (vec) {
#pragma unroll
      for (int q = 0; q < T / 8; ++q) {
        const int v = q * 32 + lane, i = MJ == kAlongK ? v / 4 : v % (T / 4) * 4, k = MJ == kAlongK ? v % 4 * 4 : v / (T / 4);
        copy_async<16>(dst + at<MJ, T>(i, k), src(i, k), any);
      }
    } else {
      for (int q = 0; q < T / 2; ++q) {
        const int v = q * 32 + lane, i = MJ == kAlongK ? v / kSimtKC : v % T, k = MJ == kAlongK ? v % kSimtKC : v / T;
        copy_async<4>(dst + at<MJ, T>(i, k), src(i, k), any);
      }
    }
  }

  // The tile's sums over n_chunks chunks.  begin(chunk) is called in front of a chunk's a_at / b_at(chunk, i, k), the
  // addresses of element i of the tile's rows (columns), position k of the chunk; NULL: zero.
  // On return (of all threads) value4 gives the sums.
  template <Major AM, Major BM, typename FB0, typename FA, typename FB>
  __device__ static void run(Smem& s, int n_chunks, bool vec_a, bool vec_b, const float* any, FB0 begin, FA a_at, FB b_at) {
    static_assert(AM == kAlongK || BM == kAcrossK, "not used");
    const int g = threadIdx.x / 32, lane = threadIdx.x % 32, ty = lane / 8, tx = lane % 8;
    Warp& w = s.w[g];
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    const int n = (n_chunks - g + KG - 1) / KG;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(&w));
    auto load = [&](int it, int stage) {
      if (it < n) {
        const int c = it * KG + g;
        begin(c);
        const uint32_t dst = base + (uint32_t)(stage * sizeof(Stage));
        fetch<AM, kSimtM>(dst, vec_a, any, [&](int i, int k) { return a_at(c, i, k); });
        fetch<BM, kSimtN>(dst + (uint32_t)sizeof(float) * kSimtM * kSimtKC, vec_b, any, [&](int i, int k) { return b_at(c, i, k); });
      }
      asm volatile("cp.async.commit_group;" : : : "memory");
    };
#pragma unroll
    for (int it = 0; it < kStages - 1; ++it) load(it, it);
    int stage = 0;
    for (int it = 0; it < n; ++it) {
      asm volatile("cp.async.wait_group %0;" : : "n"(kStages - 2) : "memory");
      __syncwarp();                                // the chunk is there, and all lanes are done with the one before it
      load(it + kStages - 1, stage == 0 ? kStages - 1 : stage - 1);
      const char* sa = reinterpret_cast<const char*>(w.stage[stage].a);
      const char* sb = reinterpret_cast<const char*>(w.stage[stage].b);
      if (++stage == kStages) stage = 0;
      auto four = [](const char* p, float (&v)[4]) {
        const float4 f = *reinterpret_cast<const float4*>(p);
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
      };
#pragma unroll 2
      for (int k = 0; k < kSimtKC; k += 4) {
        float a[8][4];                             // along K: [row][position], across K: [2 position + half][row]
        if (AM == kAlongK) {
#pragma unroll
          for (int i = 0; i < 8; ++i) four(sa + at<AM, kSimtM>(own<AM, 4>(ty, i), k), a[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) four(sa + at<AM, kSimtM>(own<AM, 4>(ty, i % 2 * 4), k + i / 2), a[i]);
        }
        if (BM == kAlongK) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float b[4];
            four(sb + at<BM, kSimtN>(own<BM, 8>(tx, j), k), b);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
              for (int i = 0; i < 8; ++i) acc[i][j] = fmaf(a[i][q], b[q], acc[i][j]);
          }
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float b[4];
              four(sb + at<BM, kSimtN>(own<BM, 8>(tx, 4 * h), k + q), b);
#pragma unroll
              for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  const float av = AM == kAlongK ? a[i][q] : a[2 * q + i / 4][i % 4];
                  acc[i][4 * h + j] = fmaf(av, b[j], acc[i][4 * h + j]);
                }
            }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" : : : "memory");
    __syncwarp();                                  // the stages are free
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) w.sums[own<AM, 4>(ty, i) * kSimtLd + own<BM, 8>(tx, j)] = acc[i][j];
    __syncthreads();
  }

  // Row r, columns c .. c + 3 of the tile (c a multiple of 4): the warps' sums added up, in their order.
  __device__ static float4 value4(const Smem& s, int r, int c) {
    float4 v = *reinterpret_cast<const float4*>(&s.w[0].sums[r * kSimtLd + c]);
#pragma unroll
    for (int g = 1; g < KG; ++g) {
      const float4 o = *reinterpret_cast<const float4*>(&s.w[g].sums[r * kSimtLd + c]);
      v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
    }
    return v;
  }
  __device__ static float value(const Smem& s, int r, int c) {
    float v = s.w[0].sums[r * kSimtLd + c];
#pragma unroll
    for (int g = 1; g < KG; ++g) v += s.w[g].sums[r * kSimtLd + c];
    return v;
  }
  // put(r, c, sums of columns c .. c + 3) for the thread's share of the tile; put2(r, c, those, the same 32 columns on).
  template <typename F> __device__ static void each4(const Smem& s, F put) {
#pragma unroll
    for (int u = 0; u < kRows * kSimtN / 4 / kThreads; ++u) {
      const int q = u * kThreads + threadIdx.x, r = q / (kSimtN / 4), c = q % (kSimtN / 4) * 4;
      put(r, c, value4(s, r, c));
    }
  }
  template <typename F> __device__ static void each4_halves(const Smem& s, F put2) {
#pragma unroll
    for (int u = 0; u < kRows * kSimtN / 8 / kThreads; ++u) {
      const int q = u * kThreads + threadIdx.x, r = q / (kSimtN / 8), c = q % (kSimtN / 8) * 4;
      put2(r, c, value4(s, r, c), value4(s, r, c + kSimtN / 2));
    }
  }
};

// The tile of batches that fill the chip several times over: 64 x 64, shared by all threads of a block.  A group of 64
// threads keeps 8 x 8 results each, packed in pairs (fma.rn.f32x2: each half an IEEE fp32 fma); chunks go through
// double-buffered shared memory, fetched into registers one chunk ahead with 16-byte loads (four of 4 bytes where an operand
// misses that alignment: an eighth of the instructions that 4-byte cp.async would take), and the operands of step k + 1
// are read while step k is multiplied.  KG groups share a tile by taking every KG-th chunk.
// Its packed products take half the issue slots, which is what counts once every scheduler has warps enough: 16 experts of
// 512 x 1024, 512 rows each, FMA pipe busy 60 to 66 % of the time in 51 to 54 % of the issue slots, against 54 to 61 % in 68 to 81
// % with warp tiles (gate/up 482 -> 405 us under the profiler; the rule and more figures: expert_simt.cu).  Twelve warps on an SM,
// 160 to 168 registers.
template <int KG>
struct SimtBlockTile {
  static constexpr int kGroup = 64, kRows = 64, kThreads = KG * kGroup, kBlocks = 6 / KG, MR = 8, NR = 8;
  static constexpr int kA4 = kRows * kSimtKC / 4 / kGroup, kB4 = kSimtN * kSimtKC / 4 / kGroup;   // float4 per thread
  struct Smem {
    float a[KG][2][kSimtKC][kRows + 4];
    float b[KG][2][kSimtKC][kSimtN + 4];
  };
  unsigned long long acc[MR][NR / 2];

  // results of this thread: row(i), column(j) inside the tile
  __device__ static int row(int i) { return i % 4 + i / 4 * (kRows / 2) + threadIdx.x % kGroup / 8 * 4; }
  __device__ static int col(int j) { return j % 4 + j / 4 * (kSimtN / 2) + threadIdx.x % 8 * 4; }
  __device__ float value(int i, int j) const {
    const unsigned long long v = acc[i][j / 2];
    return __uint_as_float(j & 1 ? (uint32_t)(v >> 32) : (uint32_t)v);
  }
  __device__ float4 value4(int i, int j) const { return make_float4(value(i, j), value(i, j + 1), value(i, j + 2), value(i, j + 3)); }

  // One operand's chunk: registers <- memory and shared memory <- registers.
  template <Major MJ, int N4, typename F>
  __device__ static void fetch(float4 (&r)[N4], bool vec, F src) {
#pragma unroll
    for (int q = 0; q < N4; ++q) {
      const int v = threadIdx.x % kGroup + q * kGroup;
      const float* p = MJ == kAlongK ? src(v / (kSimtKC / 4), v % (kSimtKC / 4) * 4) : src(v % 16 * 4, v / 16);
      r[q] = p ? ld4(p, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  template <Major MJ, int N4>
  __device__ static void stash(float (*s)[kSimtN + 4], const float4 (&r)[N4]) {
    static_assert(kRows == kSimtN, "both operands have rows of 64");
#pragma unroll
    for (int q = 0; q < N4; ++q) {
      const int v = threadIdx.x % kGroup + q * kGroup;
      if (MJ == kAlongK) {
        const int i = v / (kSimtKC / 4), k = v % (kSimtKC / 4) * 4;
        s[k][i] = r[q].x; s[k + 1][i] = r[q].y; s[k + 2][i] = r[q].z; s[k + 3][i] = r[q].w;
      } else {
        *reinterpret_cast<float4*>(&s[v / 16][v % 16 * 4]) = r[q];
      }
    }
  }
  struct Frag { float a[MR]; unsigned long long b[NR / 2]; };
  __device__ static void read(Frag& f, const float (*sa)[kRows + 4], const float (*sb)[kSimtN + 4], int k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 v = *reinterpret_cast<const float4*>(&sa[k][row(4 * h)]);
      f.a[4 * h] = v.x; f.a[4 * h + 1] = v.y; f.a[4 * h + 2] = v.z; f.a[4 * h + 3] = v.w;
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&sb[k][col(4 * h)]);
      f.b[2 * h] = w.x; f.b[2 * h + 1] = w.y;
    }
  }

  // As SimtTile::run; on return the first group of threads holds the sums.
  template <Major AM, Major BM, typename FB0, typename FA, typename FB>
  __device__ void run(Smem& s, int n_chunks, bool vec_a, bool vec_b, const float*, FB0 begin, FA a_at, FB b_at) {
    const int g = threadIdx.x / kGroup;
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
      for (int j = 0; j < NR / 2; ++j) acc[i][j] = 0ull;
    const int n_it = (n_chunks + KG - 1) / KG;
    float4 ra[kA4], rb[kB4];
    auto load = [&](int it) {
      const int c = it * KG + g;
      const bool some = c < n_chunks;
      if (some) begin(c);
      fetch<AM>(ra, vec_a, [&](int i, int k) -> const float* { return some ? a_at(c, i, k) : nullptr; });
      fetch<BM>(rb, vec_b, [&](int i, int k) -> const float* { return some ? b_at(c, i, k) : nullptr; });
    };
    if (n_it > 0) load(0);
    for (int it = 0; it < n_it; ++it) {
      float (*sa)[kRows + 4] = s.a[g][it & 1];
      float (*sb)[kSimtN + 4] = s.b[g][it & 1];
      stash<AM>(sa, ra);
      stash<BM>(sb, rb);
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
    if constexpr (KG > 1) {                        // the other groups hand their sums over through shared memory
      __syncthreads();
      constexpr int kSums = MR * NR / 2;
      unsigned long long* x = reinterpret_cast<unsigned long long*>(&s);
      static_assert(sizeof(Smem) >= (KG - 1) * kSums * kGroup * 8, "room for the groups' sums");
      const int t = threadIdx.x % kGroup;
      if (g > 0) {
#pragma unroll
        for (int q = 0; q < kSums; ++q) x[((g - 1) * kSums + q) * kGroup + t] = acc[q / (NR / 2)][q % (NR / 2)];
      }
      __syncthreads();
      if (g == 0) {
        for (int o = 0; o < KG - 1; ++o)
#pragma unroll
          for (int q = 0; q < kSums; ++q)
            asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[q / (NR / 2)][q % (NR / 2)]) : "l"(x[(o * kSums + q) * kGroup + t]));
      }
    }
  }

  template <typename F> __device__ void each4(const Smem&, F put) const {
    if (threadIdx.x >= kGroup) return;
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
      for (int j = 0; j < NR; j += 4) put(row(i), col(j), value4(i, j));
  }
  template <typename F> __device__ void each4_halves(const Smem&, F put2) const {
    if (threadIdx.x >= kGroup) return;
#pragma unroll
    for (int i = 0; i < MR; ++i) put2(row(i), col(0), value4(i, 0), value4(i, 4));
  }
};

}  // namespace unipool
