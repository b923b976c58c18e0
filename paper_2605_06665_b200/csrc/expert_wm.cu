// The four row GEMMs of the expert FFN with the WEIGHTS on the M side of the tensor-core instruction.
//
// With tokens on the M side (expert_tc.cu) a group of 341 rows is three 128-row tiles, 11 % of them
// padding, and each tile streams its expert's weights through the SM again.  Here a CTA pair (cta_group::2,
// M = 256) holds 256 rows of an expert's weights and ALL of the group's tokens up to 384 on the N side, in
// steps of 16: a weight is read once per group and the tokens need no 128-row padding.
//
// The nearest limit is shared-memory bandwidth, 128 bytes per SM clock, beside the 1 kW power cap.  Counters of gate/up /
// down / dgrad down on 24 experts of 1536 x 4096, 341 rows each, at 1.59 .. 1.68 GHz, in % of the elapsed cycles: tensor
// core's operand reads 38 / 34 / 24, TMA writes 30 / 24 / 28, epilogue 9 / 2 / 13 (of one port: 77 / 60 / 65); tensor pipe
// 60 / 56 / 40, DRAM 56 / 50 / 55; 7 / 21 / 9 % of the SM time is the last deal of units.  Per k-block and CTA
// (operands written by TMA + read by the tensor core, a CTA reading its half of the tokens):
//   token tile 128 x 256, one CTA      48 + 48 KB            768 clocks for 512 of the tensor core
//   341 tokens here, two MMAs          38 + 54 KB            736 clocks for 704
//   gate/up, 176 tokens, two MMAs      43 + 54 KB + 11..22 KB of results     864..950 clocks for 704
//   dgrad down, 176 tokens             27 + 27 KB + 15..30 KB of G, U, dG, dU    552..672 clocks for 352
// Measured 769 / 806 (second dgrad at K = 8192 / 4096), 983 / 1225, 719 / 930.  Per launch against the token-major
// kernels, interleaved: 192 experts of 1536 x 4096, 341 rows each: gate/up 1995 -> 1757, down 900 -> 806, dgrad
// down 1329 -> 1238, dgrad gate/up 1698 -> 1569 us; 96 experts of 768 x 2048: 271 -> 266, 132 -> 123, 201 -> 193,
// 240 -> 212 us.
//
//   unit     = (expert, chunk of <= 384 of its tokens, 256 weight rows); chunk fastest, so that the chunks
//              of a large group read a weight tile at the same time
//   TMEM     the accumulator is [128 weight rows = lanes][tokens = columns] per CTA; up to 256 columns it is
//              double-buffered, above that the next unit waits for the epilogue (its operands are already
//              in the stages)
//   two MMAs a chunk of more than 256 tokens is two instructions of N <= 192 on the same weight tile; the
//              gate/up projection instead runs a gate tile and an up tile over one chunk of <= 192
//              tokens, so that G and U of an element meet in one thread
//   epilogue the accumulator is transposed on its way out: tcgen05.ld.16x256b leaves a warp with 8 x 8
//              fragments (weight row x token), stmatrix.trans writes them token-major into a 32 x 32 tile,
//              a TMA store moves the tile
#include <cuda.h>

#include "common.cuh"
#include "tc_maps.cuh"
#include "tc_ptx.cuh"

namespace unipool {

namespace {

constexpr int kBK = 64;                       // k-block: 64 bf16 = one 128-byte swizzle row
constexpr int kTok = 32;                      // tokens and features of one epilogue block
constexpr uint32_t kTileBytes = 32 * 32 * 2;  // such a block in bf16: 64-byte rows, 64-byte swizzle
constexpr uint32_t kMnBlock = 64 * kBK * 2;   // one 64 (M) x 64 (K) box of weights read along M
constexpr int kBoxes = 12;                    // token boxes of 16, 32 .. 192 rows
constexpr int kEpi = 8;                       // epilogue warps: two per TMEM lane quarter, alternate blocks
constexpr int kSecond = 192;                  // column of a wide unit's second accumulator (of a narrow one: 128)
constexpr uint32_t kSmemMax = 227 * 1024;

template <int MODE> struct Wm {
  static constexpr bool kDual = MODE == kFwd1;                  // gate and up weights, two accumulators
  static constexpr bool kIo = MODE == kDgrad1;                  // the epilogue also reads G and U
  static constexpr bool kAMn = MODE == kDgrad1 || MODE == kDgrad2;
  static constexpr int kMaxTok = kDual ? 192 : kIo ? 256 : 384; // tokens of a unit
  static constexpr uint32_t kABytes = kDual ? 2 * 16384 : 16384;
  // Room for the operands of four or five k-blocks of the largest unit.  A launch whose largest unit is smaller divides
  // it into more, and the plain GEMMs take two k-blocks a stage where that leaves three stages: with few tokens the
  // launch streams weights, and waits, barriers and TMA issues per 16 KB were what held it back (31 rows of
  // 768 x 2048, five stages of one k-block / ten / five of two: down 70 / 66 / 66 us, dgrad gate/up 113 / 113 / 111;
  // 64 rows of 1536 x 4096: down 337 / 322 / 305, dgrad gate/up 609 / 595 / 535).
  static constexpr uint32_t kStageRoom = (kDual ? 4 : 5) * (kABytes + kMaxTok / 2 * 128);
  static constexpr int kMaxStages = kDual ? 5 : kIo ? 8 : 11;
  // gate/up: the epilogue warps keep a unit's last two blocks of both accumulators in registers (see there), so
  // they are two warpgroups of their own that take over the registers of the first (setmaxnreg)
  static constexpr int kEpiBase = kDual ? 4 : 2;                // first epilogue warp
  static constexpr int kThreads = 32 * (kEpiBase + kEpi) + (kIo ? 128 : 0);
  static constexpr uint32_t kStaging = kStageRoom;
  static constexpr int kRing = 4;                               // dgrad1: (G, U) blocks in flight per lane quarter
  static constexpr uint32_t kStagingBytes = kIo ? 4 * kRing * 2 * kTileBytes : kEpi * (kDual ? 3 : 1) * kTileBytes;
  static constexpr uint32_t kBars = kStaging + kStagingBytes;
  static constexpr uint32_t kTable = kBars + (kIo ? 432 : 384);   // one word per expert of the launch
  static_assert((2 * kMaxStages + 4 + (kIo ? 8 * kRing : 0)) * 8 + 16 <= (kIo ? 432 : 384), "barrier block");
  static_assert(kTable + 4 * kWmMaxExperts + 1024 <= kSmemMax, "shared-memory budget");
};

struct WmParams {
  const int32_t* offsets;        // [n_experts + 1] group starts
  const int32_t* rows;           // [n_experts] true group sizes, or NULL: the padded ones
  int n_experts, expert_base;
  int Mdim, Kdim, f;             // weight rows per expert (fwd1: f), contraction, expert width
  int n_wt;                      // weight tiles per expert: ceil(Mdim / 256)
  __nv_bfloat16 *out0, *out1;    // row-major outputs, for the pad rows (NULL: not needed)
  int32_t* status;
};

struct TokenMaps { CUtensorMap m[kBoxes]; };    // boxes of 64 x (16 (i + 1)) tokens
struct BlockMaps { CUtensorMap m[4]; };         // 32 features x 8, 16, 24, 32 tokens

// One unit of work: n tokens from row t0 on (n a multiple of 16, of 32 above 256) in one or two accumulators of
// N columns; each CTA loads h = n / 2 of them, from row t0 + rank * h on.
struct Unit { int pos, cum, e, wt, t0, n, N, h, pad_lo, pad_hi; bool two; };

// The experts of a launch in order of decreasing unit size, one word each: expert | tokens / 16 << 9 (experts
// without tokens are left out).  Units are numbered along this list (weight tile, then chunk inside an
// expert) and dealt to the CTA pairs forwards and backwards in turn, so that every deal holds units of similar
// length, the long ones first: groups of 237 .. 450 rows dealt in expert order had left the slowest pair
// 25 % behind the average on some 300 units for 74 pairs.
template <int MODE>
__device__ __forceinline__ int group_chunks(int n16) {
  const int n = n16 * 16;
  if constexpr (Wm<MODE>::kMaxTok > 256) {
    // A k-block of n tokens moves 32 KB + 128 n bytes through shared memory with one MMA, 48 KB + 128 n with two
    // (the weights are read again): 256 or 384 times the number of chunks is what the split decides.  Chunks of
    // up to 256 against 384 everywhere: 819 rows 118 against 124 us (down projection, 40 experts of 768 x 2048),
    // 500 rows 178 against 169 us.
    const int one = (n + 255) / 256, two = (n + 383) / 384;
    return 384 * two <= 256 * one ? two : one;
  }
  return (n + Wm<MODE>::kMaxTok - 1) / Wm<MODE>::kMaxTok;
}
template <int MODE>
__device__ __forceinline__ int chunk_size(int n16, int chunks) {          // <= kMaxTok
  return chunks == 1 ? n16 * 16 : ((n16 * 16 + chunks - 1) / chunks + 31) / 32 * 32;
}

// tokens of group e in steps of kRowStep
static_assert(kRowStep == 16, "steps of the unit list");
__device__ __forceinline__ int group_n16(const WmParams& p, int e) {
  const int padded = p.offsets[e + 1] - p.offsets[e];
  return ((p.rows ? min(max(p.rows[e], 0), padded) : padded) + 15) / 16;
}

// Fills in unit u.  q.pos, q.cum: list position and units before it, moved on from an earlier unit's; `single`: every
// group is one chunk, the list position follows from u (the walk over the experts of a deal, 25 of them at three
// weight tiles each, held up all roles: dgrad gate/up 85 -> 68 us at 768 x 256 and 20
// rows, 146 -> 136 us at 768 x 2048 and 170 rows).
template <int MODE, bool ROWS = true>
__device__ __forceinline__ void seek(const WmParams& p, const uint32_t* list, bool single, int u, Unit& q) {
  uint32_t word;
  int n16, chunks;
  if (single) {
    q.pos = u / p.n_wt;
    q.cum = q.pos * p.n_wt;
  }
  for (;;) {
    word = list[q.pos];
    n16 = (int)(word >> 9);
    chunks = group_chunks<MODE>(n16);
    if (u < q.cum + chunks * p.n_wt) break;
    q.cum += chunks * p.n_wt;
    ++q.pos;
  }
  q.e = (int)(word & 511u);
  const int local = u - q.cum;
  q.wt = local / chunks;
  const int c = local - q.wt * chunks;
  const int size = chunk_size<MODE>(n16, chunks);
  const bool last = c + 1 == chunks;
  const int n = last ? n16 * 16 - c * size : size;
  q.two = Wm<MODE>::kMaxTok > 256 && n > 256;
  q.n = q.two ? (n + 31) / 32 * 32 : n;                           // within the group's 128-row padding
  q.N = q.two ? q.n / 2 : q.n;
  q.h = q.n / 2;
  if constexpr (ROWS) {
    q.t0 = p.offsets[q.e] + c * size;
    q.pad_lo = last ? q.t0 + q.n : 0;                             // rows of the group that no unit covers
    q.pad_hi = last ? p.offsets[q.e + 1] : 0;
  }
}
__device__ __forceinline__ int snake(int round, int pair, int n_pairs) {
  return round * n_pairs + ((round & 1) ? n_pairs - 1 - pair : pair);
}

// Epilogue block b of a unit: nt tokens from row `row` on at accumulator column `col`.
struct Block { int col, row, nt; };
__device__ __forceinline__ int unit_blocks(const Unit& q) {
  return q.two ? 4 * ((q.N / 2 + kTok - 1) / kTok) : (q.N + kTok - 1) / kTok;
}
__device__ __forceinline__ Block unit_block(const Unit& q, int b) {
  Block k;
  if (!q.two) {
    k.col = b * kTok;
    k.row = q.t0 + k.col;
    k.nt = min(kTok, q.N - k.col);
  } else {                       // MMA i >> 1, the half of its columns whose tokens CTA (i & 1) loaded
    const int len = q.N / 2, per = (len + kTok - 1) / kTok;
    const int i = b / per, o = (b % per) * kTok;
    k.col = (i >> 1) * kSecond + (i & 1) * len + o;
    k.row = q.t0 + (i & 1) * q.h + (i >> 1) * len + o;
    k.nt = min(kTok, len - o);
  }
  return k;
}

__device__ __forceinline__ void wm_timeout(const WmParams& p, volatile int* abort, int site) {
  *abort = 1;
  if (atomicCAS(p.status, 0, kStatusTimeout) == 0) {
    p.status[1] = site;
    p.status[2] = (int)blockIdx.x;
  }
}

// 32 lanes x 32 columns as fragments: v[4 j + {0, 1}] = lane t/4, columns 8 j + 2 (t % 4) + {0, 1} for thread t;
// v[4 j + {2, 3}] = lane t/4 + 8; v[16 + ..] the lanes 16 further on.
__device__ __forceinline__ void load_fragments(uint32_t taddr, uint32_t (&v)[32]) {
  tc::tmem_ld_16x256b_x4(taddr, *reinterpret_cast<uint32_t(*)[16]>(&v[0]));
  tc::tmem_ld_16x256b_x4(taddr + (16u << 16), *reinterpret_cast<uint32_t(*)[16]>(&v[16]));
}
// Byte offset of this lane's row in a stmatrix / ldmatrix (.x4, .trans) of token group j: matrix lane / 8 =
// features [8 (lane / 8), + 8), its row lane % 8 = token 8 j + lane % 8; piece q of row r sits at q ^ ((r >> 1) & 3).
__device__ __forceinline__ uint32_t fragment_row(int lane, int j) {
  const int i = lane >> 3, r = lane & 7;
  return (uint32_t)(j * 512 + r * 64 + ((i ^ ((r >> 1) & 3)) << 4));
}
// pk: the fragments of load_fragments rounded to bf16, two columns of a lane in a word.
__device__ __forceinline__ void store_packed(uint8_t* tile, int lane, const uint32_t (&pk)[16]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    tc::stmatrix_x4_trans(tile + fragment_row(lane, j), pk[2 * j], pk[2 * j + 1], pk[8 + 2 * j], pk[9 + 2 * j]);
}
__device__ __forceinline__ void store_fragments(uint8_t* tile, int lane, const float (&v)[32]) {
  uint32_t pk[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) pk[j] = tc::pack_bf16(v[2 * j], v[2 * j + 1]);
  store_packed(tile, lane, pk);
}
__device__ __forceinline__ void read_fragments(const uint8_t* tile, int lane, float (&v)[32]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t w[4];
    tc::ldmatrix_x4_trans(tile + fragment_row(lane, j), w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = (i >> 1) * 16 + 4 * j + (i & 1) * 2;
      v[o] = __uint_as_float(w[i] << 16);
      v[o + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
}

// Zeros rows [lo, hi) x 32 features of a row-major matrix (the warp that owns these features).
__device__ __forceinline__ void zero_rows(__nv_bfloat16* out, int64_t ld, int col, int lo, int hi, int lane) {
  for (int r = lo + lane / 4; r < hi; r += 8)
    *reinterpret_cast<uint4*>(out + (int64_t)r * ld + col + (lane & 3) * 8) = make_uint4(0, 0, 0, 0);
}

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Wm<MODE>::kThreads, 1)
wm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ TokenMaps tmB,
          const __grid_constant__ BlockMaps tmC0, const __grid_constant__ BlockMaps tmC1, const WmParams p) {
  using W = Wm<MODE>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + W::kBars);
  uint64_t* empty_bar = full_bar + W::kMaxStages;
  uint64_t* tmem_full = empty_bar + W::kMaxStages;           // [2] by unit parity
  uint64_t* tmem_empty = tmem_full + 2;                      // [2]
  uint64_t* ring_full = tmem_empty + 2;                      // dgrad1: [4][kRing] a block's G and U have landed
  uint64_t* ring_staged = ring_full + (W::kIo ? 4 * W::kRing : 0);   // dgrad1: dG and dU are in their place
  uint32_t* tmem_ptr = reinterpret_cast<uint32_t*>(ring_staged + (W::kIo ? 4 * W::kRing : 0));
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_ptr + 1);
  int* n_units = reinterpret_cast<int*>(tmem_ptr + 2);       // [0] units, [1] groups with tokens
  uint32_t* list = reinterpret_cast<uint32_t*>(smem + W::kTable);              // [n_experts]

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = (int)tc::cluster_ctarank();               // 0 = leader
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < W::kMaxStages; ++s) { tc::mbar_init(&full_bar[s], 1); tc::mbar_init(&empty_bar[s], 1); }
    for (int a = 0; a < 2; ++a) { tc::mbar_init(&tmem_full[a], 1); tc::mbar_init(&tmem_empty[a], 2 * kEpi); }
    if constexpr (W::kIo)
      for (int i = 0; i < 4 * W::kRing; ++i) { tc::mbar_init(&ring_full[i], 1); tc::mbar_init(&ring_staged[i], 1); }
    *abort = 0;
    tc::fence_barrier_init();
    tc::tma_prefetch_desc(&tmA);
  }
  if (warp == 1) {
    tc::tmem_alloc_pair(tmem_ptr, 512);
    tc::tmem_relinquish_pair();
  }
  grid_wait();
  // the list of experts: a thread ranks its expert by counting the larger keys (unit size, then lower index first);
  // every CTA computes the same list
  uint32_t* key = reinterpret_cast<uint32_t*>(smem);                           // the stages are idle still
  if (threadIdx.x == 0) n_units[0] = n_units[1] = 0;
  const int n4 = (p.n_experts + 3) & ~3;
  for (int e = threadIdx.x; e < n4; e += blockDim.x) {
    uint32_t v = 0;                                                            // no tokens: behind all others
    if (e < p.n_experts) {
      const int n16 = group_n16(p, e);
      if (n16 > 0) v = (uint32_t)chunk_size<MODE>(n16, group_chunks<MODE>(n16)) << 9 | (511u - (uint32_t)e);
    }
    key[e] = v;
  }
  __syncthreads();
  for (int e0 = warp * 32; e0 < p.n_experts; e0 += (int)blockDim.x) {
    const int e = e0 + lane;
    const uint32_t mine = e < p.n_experts ? key[e] : 0;
    int before = 0;
    for (int o = 0; o < n4; o += 4) {
      const uint4 k = *reinterpret_cast<const uint4*>(key + o);
      before += (k.x > mine) + (k.y > mine) + (k.z > mine) + (k.w > mine);
    }
    int units = 0;
    if (mine != 0) {
      const int n16 = group_n16(p, e);
      list[before] = (uint32_t)e | (uint32_t)n16 << 9;
      units = group_chunks<MODE>(n16) * p.n_wt;
    }
    const int groups = __popc(__ballot_sync(0xffffffffu, units > 0));
    units = __reduce_add_sync(0xffffffffu, units);
    if (lane == 0 && units > 0) { atomicAdd(n_units, units); atomicAdd(n_units + 1, groups); }
  }
  tc::tc_fence_before_sync();
  __syncthreads();
  tc::cluster_sync();                                        // both CTAs' barriers exist before any remote use
  tc::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_ptr;
  const int total = n_units[0];
  const bool single = total == n_units[1] * p.n_wt;
  tc::fence_proxy_async();                                   // the scratch above is about to be written by TMA
  const int kblocks = p.Kdim / kBK;
  // the list begins with the largest units
  uint32_t stage_bytes = W::kStageRoom;
  if (total > 0) {
    const int n16 = (int)(list[0] >> 9), size = chunk_size<MODE>(n16, group_chunks<MODE>(n16));
    stage_bytes = W::kABytes + (uint32_t)(size / 2 + 15) / 16 * (16 * 128);
  }
  const int slots = min(W::kMaxStages, (int)(W::kStageRoom / stage_bytes));
  const int kpb = !W::kDual && !W::kIo && slots >= 6 ? 2 : 1, n_stages = slots / kpb;   // k-blocks a stage, stages
  const uint32_t stage_step = (uint32_t)kpb * stage_bytes;

  if (warp < W::kEpiBase) {
  // gate/up: 384 threads are launched with 168 registers: 48 x 128 + 224 x 256 <= 168 x 384
  if constexpr (W::kDual) tc::regs_dec<48>();
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (one in each CTA)
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      Unit q{}, next{};
      if (pair < total) seek<MODE>(p, list, single, pair, next);
      for (int round = 0; ok; ++round) {
        if (snake(round, pair, n_pairs) >= total) break;
        q = next;                                            // the next unit is looked up while this one streams
        if (snake(round + 1, pair, n_pairs) < total) seek<MODE>(p, list, single, snake(round + 1, pair, n_pairs), next);
        const int pe = p.expert_base + q.e;
        const int box = (q.h + 15) / 16;
        const CUtensorMap* mapB = &tmB.m[box - 1];
        const uint32_t tx1 = 2 * (W::kABytes + (uint32_t)box * (16 * 128));
        const int trow = q.t0 + rank * q.h;
        for (int kb0 = 0; kb0 < kblocks; kb0 += kpb) {
          if (!tc::mbar_wait(&empty_bar[stage], phase ^ 1u, abort)) { wm_timeout(p, abort, 41); ok = false; break; }
          const int kb1 = min(kb0 + kpb, kblocks);
          uint8_t* sA = smem + (uint32_t)stage * stage_step;
          if (rank == 0) tc::mbar_expect_tx(&full_bar[stage], (uint32_t)(kb1 - kb0) * tx1);     // both CTAs' bytes
          for (int kb = kb0; kb < kb1; ++kb, sA += stage_bytes) {
            if constexpr (MODE == kFwd1)         // 128 gate and the same 128 up features: W_gu as [2M][f][d]
              tc::tma_load_3d_pair(sA, &tmA, &full_bar[stage], kb * kBK, q.wt * 256 + rank * 128, 2 * pe);
            else if constexpr (MODE == kFwd2)    // 128 rows of W_down
              tc::tma_load_2d_pair(sA, &tmA, &full_bar[stage], kb * kBK, pe * p.Mdim + q.wt * 256 + rank * 128);
            else                                 // 128 columns of W_down / W_gu: two 64-column blocks
              tc::tma_load_3d_pair(sA, &tmA, &full_bar[stage], 0, pe * p.Kdim + kb * kBK, q.wt * 4 + rank * 2);
            tc::tma_load_2d_pair(sA + W::kABytes, mapB, &full_bar[stage], kb * kBK, trow);
          }
          if (++stage == n_stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader CTA only)
    // The plain GEMMs run the loop as a whole warp and one lane issues: eight MMAs of N = 176 take 704 clocks, a lane
    // alone needs as long to issue them (against that: down 131 -> 126 us, dgrad gate/up 226 -> 213 at 96 experts of
    // 768 x 2048, 341 rows; 879 -> 832 and 1715 -> 1629 at 1536 x 4096).  Gate/up and dgrad down are bound by their
    // epilogues' share of shared memory, and did not gain (their registers: 272 -> 274, 194 -> 197 us).
    constexpr bool kWarp = !W::kDual && !W::kIo;
    if (rank == 0 && (kWarp || lane == 0)) {
      constexpr uint32_t a_lbo = W::kAMn ? kMnBlock : 16;
      constexpr uint32_t a_step = (W::kAMn ? 16 * 128 : 32) >> 4;          // descriptor units per K = 16
      const uint32_t issue = lane == 0 ? 1u : 0u;
      auto uni = [](uint32_t v) { return kWarp ? tc::uniform(v) : v; };
      auto all = [](bool v) { return kWarp ? __all_sync(0xffffffffu, v) != 0 : v; };
      auto mma = [&](uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accumulate) {
        if constexpr (kWarp) tc::umma_bf16_pair_if(issue, d, ad, bd, idesc, accumulate);
        else tc::umma_bf16_pair(d, ad, bd, idesc, accumulate);
      };
      auto commit = [&](uint64_t* bar) {                                   // arrives in both CTAs
        if constexpr (kWarp) tc::umma_commit_pair_if(issue, bar, 3);
        else tc::umma_commit_pair(bar, 3);
      };
      const int n_total = (int)uni((uint32_t)total), per = (int)uni((uint32_t)kpb), n_st = (int)uni((uint32_t)n_stages);
      const uint32_t tmem = uni(tmem_base), smem0 = uni(tc::smem_u32(smem)), bytes = uni(stage_bytes);
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true, wide_before = false;
      Unit next{};
      if (pair < n_total) seek<MODE, false>(p, list, single, pair, next);
      for (; ok && snake(local, pair, n_pairs) < n_total; ++local) {
        const int N = (int)uni((uint32_t)next.N);
        const bool two = W::kDual || uni(next.two ? 1u : 0u) != 0;
        if (snake(local + 1, pair, n_pairs) < n_total) seek<MODE, false>(p, list, single, snake(local + 1, pair, n_pairs), next);
        const int cols = two ? 2 * N : N;
        const bool wide = cols > 256;
        // the accumulator of two units ago, and the previous one if either reaches into the other's half
        ok = local < 2 || tc::mbar_wait(&tmem_empty[local & 1], ((local >> 1) & 1) ^ 1u, abort);
        if (ok && local >= 1 && (wide || wide_before))
          ok = tc::mbar_wait(&tmem_empty[(local - 1) & 1], ((local - 1) >> 1) & 1, abort);
        if (!all(ok)) {
          if (issue) wm_timeout(p, abort, 42);
          break;
        }
        wide_before = wide;
        tc::tc_fence_after_sync();
        const uint32_t d0 = tmem + (wide ? 0 : (local & 1) * 256), d1 = d0 + (wide ? kSecond : 128);
        const uint32_t idesc = tc::instr_desc_bf16(N, W::kAMn, false, 256);
        const uint32_t b2 = !W::kDual && two ? (uint32_t)(N / 2 * 128) >> 4 : 0;   // second MMA: the next N / 2 tokens
        auto block = [&](uint32_t aaddr, uint32_t more) {                  // the MMAs of one k-block
          const uint64_t adesc = tc::smem_desc_sw128(aaddr, a_lbo, 1024);
          const uint64_t bdesc = tc::smem_desc_sw128(aaddr + W::kABytes, 16, 1024);
#pragma unroll
          for (int j = 0; j < kBK / 16; ++j) mma(d0, adesc + j * a_step, bdesc + j * 2, idesc, j > 0 ? 1u : more);
          if (two) {
            const uint64_t adesc2 = W::kDual ? adesc + (16384 >> 4) : adesc;
#pragma unroll
            for (int j = 0; j < kBK / 16; ++j)
              mma(d1, adesc2 + j * a_step, bdesc + b2 + j * 2, idesc, j > 0 ? 1u : more);
          }
        };
        for (int kb = 0; kb < kblocks; kb += per) {
          ok = all(tc::mbar_wait(&full_bar[stage], phase, abort));
          if (!ok) {
            if (issue) wm_timeout(p, abort, 43);
            break;
          }
          tc::tc_fence_after_sync();
          const uint32_t aaddr = smem0 + (uint32_t)stage * ((uint32_t)per * bytes);
          block(aaddr, kb != 0 ? 1u : 0u);
          if (per > 1 && kb + 1 < kblocks) block(aaddr + bytes, 1u);
          commit(&empty_bar[stage]);                                       // frees the stage
          if (++stage == n_st) { stage = 0; phase ^= 1u; }
        }
        if (ok) commit(&tmem_full[local & 1]);                             // accumulator complete
      }
    }
  }
  } else if (W::kIo && warp >= W::kEpiBase + kEpi) {
    // ------------------------------------------------------------ dgrad1: operand mover of one lane quarter
    // One lane.  Keeps the G and U blocks of the quarter's features up to kRing - 1 ahead of the epilogue (TMA
    // loads into the ring) and writes each block back once the epilogue has turned it into dG, dU in place.
    if constexpr (W::kIo) {
      if (lane == 0) {
        const int ew = warp - (W::kEpiBase + kEpi), quarter = (ew + 2) & 3;
        uint8_t* ring = smem + W::kStaging + ew * (W::kRing * 2 * kTileBytes);
        uint64_t* full = ring_full + W::kRing * ew;
        uint64_t* staged = ring_staged + W::kRing * ew;
        Unit lq{}, sq{};
        int lr = 0, sr = 0, lb = 0, sb = 0, fetched = 0, stored = 0;       // deals, blocks in a unit, blocks in all
        bool ok = true;
        auto feature = [&](const Unit& q) { return q.wt * 256 + rank * 128 + quarter * 32; };
        bool more = pair < total, live = more;                            // blocks left to fetch, to store
        if (more) { seek<MODE>(p, list, single, pair, lq); sq = lq; }
        while (live && ok) {
          while (fetched < stored + W::kRing - 1 && more) {
            if (feature(lq) < p.f) {
              const int slot = fetched % W::kRing;
              uint8_t* buf = ring + slot * 2 * kTileBytes;
              const Block k = unit_block(lq, lb);
              // fetched - kRing <= stored - 2: the store that last read this slot is not the newest one
              tc::bulk_wait_read<1>();
              tc::mbar_expect_tx(&full[slot], 2 * kTileBytes);
              tc::tma_load_2d(buf, &tmC1.m[3], &full[slot], feature(lq), k.row);
              tc::tma_load_2d(buf + kTileBytes, &tmC1.m[3], &full[slot], p.f + feature(lq), k.row);
              ++fetched;
            } else {
              lb = unit_blocks(lq);
            }
            if (++lb >= unit_blocks(lq)) {
              lb = 0;
              const int u = snake(++lr, pair, n_pairs);
              more = u < total;
              if (more) seek<MODE>(p, list, single, u, lq);
            }
          }
          if (feature(sq) < p.f) {
            const int slot = stored % W::kRing;
            uint8_t* buf = ring + slot * 2 * kTileBytes;
            const Block k = unit_block(sq, sb);
            if (!tc::mbar_wait(&staged[slot], (stored / W::kRing) & 1, abort)) { wm_timeout(p, abort, 46); ok = false; break; }
            const CUtensorMap* map = &tmC0.m[k.nt / 8 - 1];
            tc::tma_store_2d(map, buf, feature(sq), k.row);
            tc::tma_store_2d(map, buf + kTileBytes, p.f + feature(sq), k.row);
            tc::bulk_commit();
            ++stored;
          } else {
            sb = unit_blocks(sq);
          }
          if (++sb >= unit_blocks(sq)) {
            sb = 0;
            const int u = snake(++sr, pair, n_pairs);
            live = u < total;
            if (live) seek<MODE>(p, list, single, u, sq);
          }
        }
        if (!ok)
          for (int i = 0; i < 200; ++i) __nanosleep(1000);        // let loads already in flight land
        tc::bulk_wait<0>();
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue: this CTA's 128 weight rows
    if constexpr (W::kDual) tc::regs_inc<224>();
    const int quarter = warp & 3, half = (warp - W::kEpiBase) >> 2;
    const int ew = (warp - W::kEpiBase) & 3;
    uint8_t* stg = smem + W::kStaging + (W::kIo ? ew * (W::kRing * 2 * kTileBytes)
                                                : (uint32_t)(warp - W::kEpiBase) * (W::kDual ? 3 : 1) * kTileBytes);
    int local = 0, gblock = 0;
    (void)gblock;
    bool ok = true;
    Unit q{};
    for (; ok && snake(local, pair, n_pairs) < total; ++local) {
      seek<MODE>(p, list, single, snake(local, pair, n_pairs), q);
      const int feat = q.wt * 256 + rank * 128 + quarter * 32;     // first of this warp's 32 weight rows
      const bool live = feat < p.Mdim;
      const bool wide = (W::kDual || q.two ? 2 * q.N : q.N) > 256;
      const int nb = unit_blocks(q);
      if (!tc::mbar_wait(&tmem_full[local & 1], (local >> 1) & 1, abort)) {
        if (lane == 0) wm_timeout(p, abort, 44);
        break;
      }
      tc::tc_fence_after_sync();
      const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + (wide ? 0 : (local & 1) * 256);
      // TMEM is given back as soon as this warp holds its part of it in registers: the next unit's MMAs wait for
      // that when either unit is wide.
      auto release = [&] {
        tc::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {                                           // the leader's MMA thread waits for both CTAs
          if (rank == 0) tc::mbar_arrive(&tmem_empty[local & 1]);
          else tc::mbar_arrive_leader(&tmem_empty[local & 1]);
        }
      };
      if (!live) {
        release();
      } else if constexpr (MODE == kFwd1) {
        // this warp's blocks: half, half + 2, half + 4; the first is packed, the other two wait in fp32
        uint32_t rg[3][32], ru[3][32], pk[3][16];
        auto load = [&](int i) {
          load_fragments(t_row + (half + 2 * i) * kTok, rg[i]);
          load_fragments(t_row + (wide ? kSecond : 128) + (half + 2 * i) * kTok, ru[i]);
        };
        auto pack = [&](int i) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float g[2], x[2], a[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              g[c] = __uint_as_float(rg[i][2 * j + c]);
              x[c] = __uint_as_float(ru[i][2 * j + c]);
              a[c] = g[c] * tc::sigmoid_fast(g[c]) * x[c];
            }
            pk[0][j] = tc::pack_bf16(g[0], g[1]);
            pk[1][j] = tc::pack_bf16(x[0], x[1]);
            pk[2][j] = tc::pack_bf16(a[0], a[1]);
          }
        };
        auto store = [&](int i) {
          const Block k = unit_block(q, half + 2 * i);
          if (lane < 3) tc::bulk_wait_read<0>();                   // the previous block's stores have drained the tiles
          __syncwarp();
#pragma unroll
          for (int t = 0; t < 3; ++t) store_packed(stg + t * kTileBytes, lane, pk[t]);
          tc::fence_proxy_async();
          __syncwarp();
          if (lane == 0) tc::tma_store_2d(&tmC0.m[k.nt / 8 - 1], stg, feat, k.row);
          else if (lane == 1) tc::tma_store_2d(&tmC0.m[k.nt / 8 - 1], stg + kTileBytes, p.f + feat, k.row);
          else if (lane == 2) tc::tma_store_2d(&tmC1.m[k.nt / 8 - 1], stg + 2 * kTileBytes, feat, k.row);
          if (lane < 3) tc::bulk_commit();
        };
        if (half < nb) { load(0); tc::tmem_ld_wait(); pack(0); }
        if (half + 2 < nb) load(1);
        if (half + 4 < nb) load(2);
        tc::tmem_ld_wait();
        release();
        if (half < nb) store(0);
        if (half + 2 < nb) { pack(1); store(1); }
        if (half + 4 < nb) { pack(2); store(2); }
      } else if constexpr (W::kIo) {
#pragma unroll 1
        for (int b = (gblock ^ half) & 1; b < nb; b += 2) {
          const Block k = unit_block(q, b);
          uint32_t rr[32];
          load_fragments(t_row + k.col, rr);
          const int slot = (gblock + b) % W::kRing;
          uint8_t* buf = stg + slot * 2 * kTileBytes;
          tc::tmem_ld_wait();
          if (!tc::mbar_wait(&ring_full[W::kRing * ew + slot], ((gblock + b) / W::kRing) & 1, abort)) {
            if (lane == 0) wm_timeout(p, abort, 45);
            ok = false;
            break;
          }
          float g[32], x[32];
          read_fragments(buf, lane, g);
          read_fragments(buf + kTileBytes, lane, x);
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float dA = __uint_as_float(rr[i]);
            const float sig = tc::sigmoid_fast(g[i]);
            const float sl = g[i] * sig;
            g[i] = dA * x[i] * (sig + sl * (1.0f - sig));          // silu'(g) = sig (1 + g (1 - sig))
            x[i] = dA * sl;
          }
          __syncwarp();
          store_fragments(buf, lane, g);                           // in place
          store_fragments(buf + kTileBytes, lane, x);
          tc::fence_proxy_async();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&ring_staged[W::kRing * ew + slot]);   // the mover stores the block
        }
        gblock += nb;
        if (!ok) break;
        release();
      } else {
        constexpr int kMine = 6;                                   // blocks of a warp: 2 x 192 columns / 32 over two warps
        uint32_t pk[kMine][16];
#pragma unroll
        for (int i = 0; i < kMine; ++i) {
          if (half + 2 * i < nb) {
            uint32_t rr[32];
            load_fragments(t_row + unit_block(q, half + 2 * i).col, rr);
            tc::tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j)
              pk[i][j] = tc::pack_bf16(__uint_as_float(rr[2 * j]), __uint_as_float(rr[2 * j + 1]));
          }
        }
        release();
#pragma unroll
        for (int i = 0; i < kMine; ++i) {
          if (half + 2 * i < nb) {
            const Block k = unit_block(q, half + 2 * i);
            if (lane == 0) tc::bulk_wait_read<0>();
            __syncwarp();
            store_packed(stg, lane, pk[i]);
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tc::tma_store_2d(&tmC0.m[k.nt / 8 - 1], stg, feat, k.row);
              tc::bulk_commit();
            }
          }
        }
      }
      const bool pads = MODE != kDgrad1 || p.rows == nullptr;
      if (pads && live && half == 0 && q.pad_lo < q.pad_hi) {              // pad rows behind the group's last unit
        if constexpr (MODE == kFwd1) {
          zero_rows(p.out0, 2 * p.f, feat, q.pad_lo, q.pad_hi, lane);
          zero_rows(p.out0, 2 * p.f, p.f + feat, q.pad_lo, q.pad_hi, lane);
          zero_rows(p.out1, p.f, feat, q.pad_lo, q.pad_hi, lane);
        } else if constexpr (MODE == kDgrad1) {
          zero_rows(p.out0, 2 * p.f, feat, q.pad_lo, q.pad_hi, lane);
          zero_rows(p.out0, 2 * p.f, p.f + feat, q.pad_lo, q.pad_hi, lane);
        } else if constexpr (MODE == kFwd2) {
          zero_rows(p.out0, p.Mdim, feat, q.pad_lo, q.pad_hi, lane);
        }
      }
    }
    if (!ok && lane == 0)
      for (int i = 0; i < 200; ++i) __nanosleep(1000);             // let loads already in flight land before the CTA retires
    if (lane < 3) tc::bulk_wait<0>();
    __syncwarp();
  }

  tc::tc_fence_before_sync();
  __syncthreads();
  tc::cluster_sync();                                        // neither CTA leaves while the other may still signal it
  if (warp == 1) {
    tc::tc_fence_after_sync();
    tc::tmem_dealloc_pair(tmem_base, 512);
  }
}

// Token operand: row-major [rows, cols], boxes of 64 columns x 16 .. 192 rows.
int token_maps(unipool_ctx* ctx, TokenMaps* out, const void* base, uint64_t cols, uint64_t rows, int max_tok) {
  for (int i = 0; i < kBoxes; ++i) {
    const int box = 16 * (i + 1);
    if (box > max_tok / 2) { out->m[i] = out->m[i - 1]; continue; }
    const int rc = map_2d(ctx, &out->m[i], base, cols, rows, kBK, (uint32_t)box);
    if (rc != UNIPOOL_OK) return rc;
  }
  return UNIPOOL_OK;
}
int block_maps(unipool_ctx* ctx, BlockMaps* out, const void* base, uint64_t cols, uint64_t rows) {
  for (int i = 0; i < 4; ++i) {
    const int rc = map_2d(ctx, &out->m[i], base, cols, rows, kTok, (uint32_t)(8 * (i + 1)), kMapBf16Chunk);
    if (rc != UNIPOOL_OK) return rc;
  }
  return UNIPOOL_OK;
}

template <int MODE>
int wm_launch(unipool_ctx* ctx, int phase, const CUtensorMap& tmA, const TokenMaps& tmB, const BlockMaps& tmC0,
              const BlockMaps& tmC1, const WmParams& p, cudaStream_t s) {
  PhaseTimer pt(ctx, phase, 1, s);
  auto kern = wm_kernel<MODE>;
  // (the limit belongs to the function, not to the launch: the same for every caller, or a thread with fewer experts
  // lowers it between another's call and launch)
  constexpr int most = (int)Wm<MODE>::kTable + 4 * kWmMaxExperts + 1024;
  const int smem = (int)Wm<MODE>::kTable + 4 * p.n_experts + 1024;
  UP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  UP_KERNEL(kern, ctx->sm_count / 2 * 2, Wm<MODE>::kThreads, smem, s, tmA, tmB, tmC0, tmC1, p);
  return UNIPOOL_OK;
}

template <typename Args>
WmParams wm_params(const unipool_ctx* ctx, const Args& a) {
  WmParams p{};
  p.offsets = a.offsets;
  p.rows = a.rows;
  p.n_experts = a.n_experts;
  p.expert_base = a.expert_base;
  p.f = ctx->cfg.d_ff;
  p.status = ctx->ws.status;
  return p;
}

}  // namespace

int wm_fwd_gu(unipool_ctx* ctx, const ExpertFwdArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff, M = ctx->cfg.pool_size;
  const uint64_t cap = (uint64_t)ctx->row_capacity;
  WmParams p = wm_params(ctx, a);
  CUtensorMap tmA;
  TokenMaps tmB;
  BlockMaps tmC0, tmC1;
  int rc;
  {                                                      // GU = Xp [W_gate; W_up]^T, A = silu(G) * U
    const uint64_t dims[3] = {(uint64_t)d, (uint64_t)f, (uint64_t)2 * M};
    const uint64_t strides[2] = {(uint64_t)d, (uint64_t)f * d};
    const uint32_t box[3] = {kBK, 128, 2};
    if ((rc = make_tmap(ctx, &tmA, kMapOperand, a.W_gu, 3, dims, strides, box)) != UNIPOOL_OK) return rc;
  }
  if ((rc = token_maps(ctx, &tmB, a.Xp, d, cap, Wm<kFwd1>::kMaxTok)) != UNIPOOL_OK) return rc;
  if ((rc = block_maps(ctx, &tmC0, a.GU, 2 * f, cap)) != UNIPOOL_OK) return rc;
  if ((rc = block_maps(ctx, &tmC1, a.A, f, cap)) != UNIPOOL_OK) return rc;
  p.Mdim = f; p.Kdim = d; p.n_wt = (f + 255) / 256;
  p.out0 = static_cast<__nv_bfloat16*>(a.GU); p.out1 = static_cast<__nv_bfloat16*>(a.A);
  return wm_launch<kFwd1>(ctx, UNIPOOL_PH_EXPERT_FWD_GU, tmA, tmB, tmC0, tmC1, p, s);
}

int wm_fwd_down(unipool_ctx* ctx, const ExpertFwdArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff, M = ctx->cfg.pool_size;
  const uint64_t cap = (uint64_t)ctx->row_capacity;
  WmParams p = wm_params(ctx, a);
  CUtensorMap tmA;
  TokenMaps tmB;
  BlockMaps tmC0;
  int rc;
  // Yp = A W_down^T
  if ((rc = map_2d(ctx, &tmA, a.W_down, f, (uint64_t)M * d, kBK, 128)) != UNIPOOL_OK) return rc;
  if ((rc = token_maps(ctx, &tmB, a.A, f, cap, Wm<kFwd2>::kMaxTok)) != UNIPOOL_OK) return rc;
  if ((rc = block_maps(ctx, &tmC0, a.Yp, d, cap)) != UNIPOOL_OK) return rc;
  p.Mdim = d; p.Kdim = f; p.n_wt = (d + 255) / 256;
  p.out0 = static_cast<__nv_bfloat16*>(a.Yp); p.out1 = nullptr;
  return wm_launch<kFwd2>(ctx, UNIPOOL_PH_EXPERT_FWD_DOWN, tmA, tmB, tmC0, tmC0, p, s);
}

int wm_dgrad_down(unipool_ctx* ctx, const ExpertBwdArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff, M = ctx->cfg.pool_size;
  const uint64_t cap = (uint64_t)ctx->row_capacity;
  WmParams p = wm_params(ctx, a);
  CUtensorMap tmA;
  TokenMaps tmB;
  BlockMaps tmC0, tmC1;
  int rc;
  // dA = dYp W_down, fused with the SwiGLU derivative -> dGU
  if ((rc = map_mn(ctx, &tmA, a.W_down, f, (uint64_t)M * d, 2)) != UNIPOOL_OK) return rc;
  if ((rc = token_maps(ctx, &tmB, a.dYp, d, cap, Wm<kDgrad1>::kMaxTok)) != UNIPOOL_OK) return rc;
  if ((rc = block_maps(ctx, &tmC0, a.dGU, 2 * f, cap)) != UNIPOOL_OK) return rc;
  if ((rc = block_maps(ctx, &tmC1, a.GU, 2 * f, cap)) != UNIPOOL_OK) return rc;
  p.Mdim = f; p.Kdim = d; p.n_wt = (f + 255) / 256;
  p.out0 = static_cast<__nv_bfloat16*>(a.dGU);
  return wm_launch<kDgrad1>(ctx, UNIPOOL_PH_DGRAD_DOWN, tmA, tmB, tmC0, tmC1, p, s);
}

int wm_dgrad_gu(unipool_ctx* ctx, const ExpertBwdArgs& a, cudaStream_t s) {
  const int d = ctx->cfg.d_model, f = ctx->cfg.d_ff, M = ctx->cfg.pool_size;
  const uint64_t cap = (uint64_t)ctx->row_capacity;
  WmParams p = wm_params(ctx, a);
  CUtensorMap tmA;
  TokenMaps tmB;
  BlockMaps tmC0;
  int rc;
  // dXp = dGU [W_gate; W_up]; its pad rows are never read
  if ((rc = map_mn(ctx, &tmA, a.W_gu, d, (uint64_t)M * 2 * f, 2)) != UNIPOOL_OK) return rc;
  if ((rc = token_maps(ctx, &tmB, a.dGU, 2 * f, cap, Wm<kDgrad2>::kMaxTok)) != UNIPOOL_OK) return rc;
  if ((rc = block_maps(ctx, &tmC0, a.dXp, d, cap)) != UNIPOOL_OK) return rc;
  p.Mdim = d; p.Kdim = 2 * f; p.n_wt = (d + 255) / 256;
  p.out0 = nullptr;
  return wm_launch<kDgrad2>(ctx, UNIPOOL_PH_DGRAD_GU, tmA, tmB, tmC0, tmC0, p, s);
}

}  // namespace unipool
