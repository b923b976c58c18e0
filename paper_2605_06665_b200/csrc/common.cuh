// Shared host/device declarations of the UniPool library (internal header).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "unipool.h"

namespace unipool {

// ---------------------------------------------------------------- errors
void set_error(const char* fmt, ...);

#define UP_REQUIRE(cond, code, ...)      \
  do {                                   \
    if (!(cond)) {                       \
      unipool::set_error(__VA_ARGS__);   \
      return (code);                     \
    }                                    \
  } while (0)

// (The runtime keeps an error for cudaGetLastError too: taken there, or whoever asks next takes it for its own.)
#define UP_CUDA(call)                                                                  \
  do {                                                                                 \
    cudaError_t e__ = (call);                                                          \
    if (e__ != cudaSuccess) {                                                          \
      cudaGetLastError();                                                              \
      unipool::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e__), __FILE__, \
                         __LINE__);                                                    \
      return UNIPOOL_ERR_CUDA;                                                         \
    }                                                                                  \
  } while (0)

#define UP_LAUNCH_CHECK()                                                              \
  do {                                                                                 \
    cudaError_t e__ = cudaGetLastError();                                              \
    if (e__ != cudaSuccess) {                                                          \
      unipool::set_error("kernel launch failed: %s (%s:%d)", cudaGetErrorString(e__),  \
                         __FILE__, __LINE__);                                          \
      return UNIPOOL_ERR_CUDA;                                                         \
    }                                                                                  \
  } while (0)

// ---------------------------------------------------------------- launches
// Every kernel of a pass is launched with programmatic serialization and waits for the one before it in grid_wait(), behind
// what of its set-up needs no memory of others (the router on the tensor cores reads two flags first and waits in front of its
// own).  No kernel triggers its successor early, so that a kernel's blocks start when the last block of the kernel before
// has left: hidden are the launch and the flush of that kernel's writes, not its last blocks.  (An early trigger would put
// two kernels' blocks on an SM, which their tensor memory, allocated whole, and shared memory do not allow.)
// Between two kernels of an eager pass lie 0.2 us instead of 2.0 .. 2.8; a pass of 16 experts of
// 256 x 512 over 512 tokens in fp32 (55 launches) takes 856 us instead of 959, a forward pass of 33 tokens through
// twelve layers 1509 instead of 1632, a step of 16384 tokens over private experts 12455 instead of 12772.
// Not while a stream is captured: the kernels of a graph follow one another within 0.3 us as they are, and with programmatic
// edges a recorded step takes 0.7 % longer (four layers of 876 tokens 1499 us against 1489).
template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(s, &capture);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = capture == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}
#define UP_KERNEL(kern, grid, block, smem, s, ...) \
  UP_CUDA(unipool::launch_kernel(kern, dim3(grid), dim3(block), smem, s, __VA_ARGS__))

#ifdef __CUDACC__
// Waits until the kernels before this one in the stream are complete and their writes visible.  All threads call it,
// before they touch global memory.  The pointers that it is given, members of a parameter struct too, come out of it, so
// that no load through them (a read-only one has no order of its own) can be moved in front of it.  (They are no longer
// restrict-qualified to the compiler: loads through them that may pass stores and atomics are written as __ldg.  Without,
// placing 2253 tokens took 8.0 us instead of 6.7.)
template <typename P>
__device__ __forceinline__ void after_asm(P& p) {
  asm volatile("" : "+l"(p));
  __builtin_assume(__isGlobal(p));             // what the compiler knew of a kernel's argument
}
template <typename... P>
__device__ __forceinline__ void grid_wait(P&... p) {
  asm volatile("griddepcontrol.wait;" : : : "memory");
  (after_asm(p), ...);
}
#endif

// ---------------------------------------------------------------- workspace
// Fixed layout of the caller's workspace; every region is 256-byte aligned.
struct Workspace {
  int32_t* status;        // [4]   device status word (+ spare)
  int32_t* route_counts;  // [MAX_EXPERTS] self-cleaning accumulators of route
  double*  route_sums;    // [MAX_EXPERTS]
  uint32_t* tickets;      // [8]   "last block done" counters, self-cleaning
  double*  dsigma_acc;    // [2]   self-cleaning accumulator of route_bwd / calibrate_c
  int32_t* block_hist;    // permute scratch: per-chunk counts (16 bits) and their sums over 16 chunks, per expert
  float*   dz;            // route_bwd scratch: fp32 [max_tokens, pool_size], or bf16 [max_tokens, ceil64(pool_size)]
  int32_t* split_any;     // [n_layers + 1][4] which bf16 terms of a router's split weights are non-zero
  void*    w_split;       // [n_layers + 1][3, pool_size, d] bf16 terms of the router weights (bf16 mode): one slot
                          // per prepared layer, the last one scratch for routers that were not prepared
  float*   w_copy;        // [n_layers][pool_size, d] the prepared layers' weights as they are (bf16 mode; same region)
  int32_t* part_counts;   // [2 ceil(max_tokens/256), pool_size] per-CTA routing counts (bf16 mode)
  float*   part_sums;     // [2 ceil(max_tokens/256), pool_size] per-CTA score sums
  float*   part_dsigma;   // [ceil(max_tokens/64)] per-block dsigma terms
  void*    dXp;           // [row_capacity, d] expert_bwd scratch (ctx dtype)
  size_t   bytes;         // total
  char*    guards[16];    // debug mode: the 256-byte guard band behind each region
  int      n_guards;      // 0 unless UNIPOOL_DEBUG=1
};
constexpr int kGuardBytes = 256;
constexpr unsigned kGuardWord = 0xA5A5A5A5u;
constexpr int kGuardSite = 200;               // status site of guard band i: kGuardSite + i

constexpr int kDispatchChunkTokens = 256;     // most tokens per block of the placing kernel (eight warps of 32)
constexpr int kDispatchMinChunkTokens = 16;   // fewest
constexpr int kDispatchSuperChunks = 16;      // chunks whose counts are summed up together
constexpr int kDispatchMaxSms = 1024;         // chunks smaller than 256 tokens are used up to two per SM of so many

Workspace carve_workspace(const unipool_config& cfg, void* base);

}  // namespace unipool

namespace unipool {
struct ProfRecord { int phase; int launches; cudaEvent_t start, stop; };
struct Profiler {
  bool enabled = false;
  std::vector<ProfRecord> records;       // events recorded since the last read
  std::vector<cudaEvent_t> free_events;  // recycled events
  cudaEvent_t get() {
    if (!free_events.empty()) { cudaEvent_t e = free_events.back(); free_events.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
  }
};
}  // namespace unipool

struct unipool_ctx {
  unipool::Profiler prof;
  unipool_config cfg;
  unipool::Workspace ws;
  int device;
  int sm_count;
  int64_t row_capacity;
  size_t elem_bytes;
  void* tmap_cache;   // opaque, owned by the tensor-core GEMM module
  const float* prepared_base;   // router weights last given to unipool_router_prepare (NULL: none)
  int prepared_layers, prepared_experts;
  bool prepared_copied;         // their fp32 weights were kept too (ws.w_copy)
  bool prepared_now;            // they were prepared by the running call, from the weights as they are
  bool copy_read;               // some launch reads ws.w_copy, recorded in a graph maybe: every preparation keeps it up to date
};

namespace unipool {

// Brackets the kernels launched during its lifetime with a pair of events (when profiling is on).
struct PhaseTimer {
  unipool_ctx* ctx; cudaStream_t s; cudaEvent_t stop = nullptr;
  PhaseTimer(unipool_ctx* c, int phase, int launches, cudaStream_t stream) : ctx(c), s(stream) {
    if (ctx == nullptr || !ctx->prof.enabled) return;
    cudaEvent_t start = ctx->prof.get();
    stop = ctx->prof.get();
    if (!start || !stop) { stop = nullptr; return; }
    cudaEventRecord(start, s);
    ctx->prof.records.push_back({phase, launches, start, stop});
  }
  ~PhaseTimer() { if (stop) cudaEventRecord(stop, s); }
};

// ---------------------------------------------------------------- element helpers
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

__device__ __forceinline__ float silu_f(float a) { return a / (1.0f + __expf(-a)); }
__device__ __forceinline__ float silu_grad_f(float a) {
  float sig = 1.0f / (1.0f + __expf(-a));
  return sig * (1.0f + a * (1.0f - sig));
}

// status codes written by kernels into ws.status[0]
constexpr int kStatusTimeout = 1;
constexpr int kStatusCheck = 2;

// ---------------------------------------------------------------- module entry points
int route_launch(unipool_ctx*, const void* x, int T, const float* W_r, float sigma,
                 const float* bias, int n_experts, int32_t* idx, float* gate, int32_t* counts,
                 float* score_sum, float* znorm, float* z_saved, cudaStream_t);
int route_bwd_launch(unipool_ctx*, const void* x, int T, const float* W_r, float sigma,
                     int n_experts, const float* znorm, const float* z_saved, const int32_t* idx,
                     const float* dgate, const float* coef, void* dx, float* dW_r, float* dsigma,
                     cudaStream_t);
int dispatch_launch(unipool_ctx*, const void* x, int T, const int32_t* idx, int n_experts,
                    int32_t* offsets, int32_t* row_of, int32_t* token_of, int32_t* tile_expert,
                    int32_t* rows, void* Xp, cudaStream_t);
int combine_launch(unipool_ctx*, const void* Yp, const int32_t* row_of, const float* gate, int T,
                   const void* residual, void* y, cudaStream_t);
// With the group sizes at hand the bf16 kernels contract over a group's rows up to the next multiple of kRowStep (the K
// of one MMA): that far the pad rows of dYp and dGU hold zeros; what follows up to the next group start is not written
// (1501 tokens over 96 experts of 768 x 2048, 31 rows in 128: scaling dY 14.6 -> 8.8 us, dgrad down 80 -> 71 us).
constexpr int kRowStep = 16;
int combine_bwd_launch(unipool_ctx*, const void* dy, int T, const int32_t* row_of,
                       const float* gate, const int32_t* token_of, const int32_t* offsets, int32_t* rows,
                       int n_experts, const void* Yp, void* dYp, float* dgate, cudaStream_t);
int unpermute_sum_launch(unipool_ctx*, const void* dXp, const int32_t* row_of, int T,
                         const void* residual, void* dx, cudaStream_t);
int aux_launch(unipool_ctx*, const int32_t* counts, const float* S, int L, int n_experts, int T,
               float alpha, const float* fbar_prev, float* loss, float* coef, float* fbar_out,
               cudaStream_t);
int unique_experts_launch(unipool_ctx*, const int32_t* idx, const int32_t* expert_base, int L, int T,
                          int32_t* unique, unsigned long long* total, cudaStream_t);
int wait_selftest_launch(unipool_ctx*, long long limit_cycles, cudaStream_t);
int guard_check_launch(unipool_ctx*, cudaStream_t);
int calibrate_launch(unipool_ctx*, int n_experts, int top_k, int n_samples, uint64_t seed,
                     float* c_out, cudaStream_t);

// grouped GEMMs: CUDA-core path (fp32 mode) and tcgen05 path (bf16 mode)
struct ExpertFwdArgs {
  const void* Xp; const int32_t* offsets; const int32_t* tile_expert;
  const void* W_gu; const void* W_down; int expert_base; int n_experts;
  void* GU; void* A; void* Yp;
  const int32_t* rows;                   // true group sizes, NULL: the padded ones
};
struct ExpertBwdArgs {
  const int32_t* offsets; const int32_t* tile_expert;
  const void* Xp; const void* GU; const void* A; const void* W_gu; const void* W_down;
  int expert_base; int n_experts;
  const void* dYp; void* dGU; void* dXp; float* dW_gu; float* dW_down; bool wgrad; bool overwrite;
  const int32_t* rows;
};
struct PoolWgradArgs {
  int n_layers; int64_t layer_stride_rows; const int32_t* offsets;
  const void* Xp; const void* A; const void* dYp; const void* dGU;
  int expert_base; int n_experts; float* dW_gu; float* dW_down; bool overwrite;
  const int32_t* rows;                   // [n_layers, n_experts]
};
int route_tc_launch(unipool_ctx*, const void* x, int T, const float* W_r, float sigma, const float* bias,
                    int n_experts, int32_t* idx, float* gate, int32_t* counts, float* score_sum,
                    float* znorm, float* z_saved, cudaStream_t);
bool route_on_few(const unipool_ctx*, const float* W_r, int T, int n_experts);
int route_few_launch(unipool_ctx*, const void* x, int T, const float* W_r, float sigma, const float* bias,
                     int n_experts, int32_t* idx, float* gate, int32_t* counts, float* score_sum,
                     float* znorm, float* z_saved, cudaStream_t);
int router_prepare_launch(unipool_ctx*, const float* W_r, int n_layers, int n_experts, bool copy, cudaStream_t);
int prepared_layer(const unipool_ctx*, const float* W_r, int n_experts);
int route_bwd_tc_launch(unipool_ctx*, const void* x, int T, const float* W_r, float sigma, int n_experts,
                        const float* znorm, const float* z_saved, const int32_t* idx, const float* dgate,
                        const float* coef, void* dx, float* dW_r, float* dsigma, cudaStream_t);
int tc_operand_map(unipool_ctx*, void* out_tensor_map, const void* base, uint64_t cols, uint64_t rows,
                   uint32_t box_rows);
int tc_f32_chunk_map(unipool_ctx*, void* out_tensor_map, const void* base, uint64_t cols, uint64_t rows);
int router_bwd_gemms_tc(unipool_ctx*, const void* dz16, int Mp, const void* W16, const void* x, int T, int M,
                        void* dx, float* dW_r, cudaStream_t);
int expert_fwd_simt(unipool_ctx*, const ExpertFwdArgs&, cudaStream_t);
int expert_bwd_simt(unipool_ctx*, const ExpertBwdArgs&, cudaStream_t);
int pool_wgrad_simt(unipool_ctx*, const PoolWgradArgs&, cudaStream_t);
int expert_fwd_tc(unipool_ctx*, const ExpertFwdArgs&, cudaStream_t);
const char* row_gemm_kernel(const unipool_ctx*, int phase, int n_experts, bool sizes_known);
int expert_bwd_tc(unipool_ctx*, const ExpertBwdArgs&, cudaStream_t);
int pool_wgrad_tc(unipool_ctx*, const PoolWgradArgs&, cudaStream_t);
int wm_fwd_gu(unipool_ctx*, const ExpertFwdArgs&, cudaStream_t);
int wm_fwd_down(unipool_ctx*, const ExpertFwdArgs&, cudaStream_t);
int wm_dgrad_down(unipool_ctx*, const ExpertBwdArgs&, cudaStream_t);
int wm_dgrad_gu(unipool_ctx*, const ExpertBwdArgs&, cudaStream_t);
int tc_module_init(unipool_ctx*);
void tc_module_destroy(unipool_ctx*);

}  // namespace unipool
