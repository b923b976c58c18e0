// A whole residual stack per call: the per-layer calls of the library in their order, issued from native code.
// A pass of twelve layers is some sixty calls forward and a hundred backward; issued one by one through a
// Python binding they cost the host 13 us each (argument conversion, tensor slicing), more than the kernels of
// a small batch take.
#include <type_traits>

#include "common.cuh"

using namespace unipool;

namespace {

// Layer l's slice of a stacked array of `elems` elements per layer.
template <typename T> T* at(T* base, int64_t l, int64_t elems) { return base ? base + l * elems : nullptr; }
template <typename V> V* at_bytes(V* base, int64_t l, int64_t bytes) {
  using Byte = typename std::conditional<std::is_const<V>::value, const char, char>::type;
  return base ? static_cast<V*>(static_cast<Byte*>(base) + l * bytes) : nullptr;
}

struct Layer {
  const unipool_ctx* c;
  const unipool_stack* s;
  int l;
  int64_t T, k, m, cap, d, f, eb;
  Layer(const unipool_ctx* ctx, const unipool_stack* st, int layer)
      : c(ctx), s(st), l(layer), T(ctx->cfg.max_tokens), k(ctx->cfg.top_k), m(st->n_experts), cap(ctx->row_capacity),
        d(ctx->cfg.d_model), f(ctx->cfg.d_ff), eb((int64_t)ctx->elem_bytes) {}
  int base() const { return l / s->layers_per_group * s->n_experts; }
  int slot() const { return s->recompute ? 0 : l; }                       // GU, Yp
  void* x(int i) const { return at_bytes(s->x, i, T * d * eb); }
  const float* W_r() const { return at(s->W_r, l, m * d); }
  float* dW_r() const { return at(s->dW_r, l, m * d); }
  const float* bias() const { return at(s->bias, l, m); }
  int32_t* idx() const { return at(s->idx, l, T * k); }
  float* gate() const { return at(s->gate, l, T * k); }
  int32_t* row_of() const { return at(s->row_of, l, T * k); }
  int32_t* offsets() const { return at(s->offsets, l, m + 1); }
  int32_t* rows() const { return at(s->rows, l, m); }
  int32_t* token_of() const { return at(s->token_of, l, cap); }
  int32_t* tile_expert() const { return at(s->tile_expert, l, cap / UNIPOOL_ROW_ALIGN); }
  float* znorm() const { return at(s->znorm, l, T); }
  float* z() const { return at(s->z, l, T * m); }
  void* per_row(void* p, int sl, int64_t width) const { return at_bytes(p, sl, cap * width * eb); }
};

#define UP_TRY(call)                     \
  do {                                   \
    const int rc__ = (call);             \
    if (rc__ != UNIPOOL_OK) return rc__; \
  } while (0)

int check_stack(const unipool_ctx* ctx, const unipool_stack* s) {
  UP_REQUIRE(ctx != nullptr && s != nullptr, UNIPOOL_ERR_INVALID_ARG, "ctx or stack is NULL");
  UP_REQUIRE(s->n_layers >= 1 && s->n_layers <= ctx->cfg.n_layers && s->layers_per_group >= 1 &&
                 s->n_layers % s->layers_per_group == 0,
             UNIPOOL_ERR_INVALID_ARG, "stack of %d layers in groups of %d", s->n_layers, s->layers_per_group);
  UP_REQUIRE(s->sigma != nullptr && s->x != nullptr, UNIPOOL_ERR_INVALID_ARG, "sigma or x is NULL");
  return UNIPOOL_OK;
}

// dispatch + expert forward of a layer; w: slot of Xp and A
int permute_and_experts(unipool_ctx* ctx, const Layer& a, int32_t T, int w, unipool_stream stream) {
  const unipool_stack* s = a.s;
  UP_TRY(unipool_dispatch_rows(ctx, a.x(a.l), T, a.idx(), s->n_experts, a.offsets(), a.row_of(), a.token_of(),
                               a.tile_expert(), a.rows(), a.per_row(s->Xp, w, a.d), stream));
  return unipool_expert_fwd_rows(ctx, a.per_row(s->Xp, w, a.d), a.offsets(), a.rows(), a.tile_expert(), s->W_gu,
                                 s->W_down, a.base(), s->n_experts, a.per_row(s->GU, a.slot(), 2 * a.f),
                                 a.per_row(s->A, w, a.f), a.per_row(s->Yp, a.slot(), a.d), stream);
}

}  // namespace

extern "C" {

int unipool_stack_forward(unipool_ctx* ctx, const unipool_stack* s, int32_t T, unipool_stream stream) {
  UP_TRY(check_stack(ctx, s));
  // The terms of all routers, for this pass and the backward pass that follows it; few tokens read the weights themselves, so
  // no copy is kept beside the terms (8.2 us instead of 10.2 for twelve routers of 96 x 768).
  struct Now {
    unipool_ctx* c;
    explicit Now(unipool_ctx* ctx) : c(ctx) { c->prepared_now = true; }
    ~Now() { c->prepared_now = false; }
  } now(ctx);
  UP_TRY(unipool_router_prepare(ctx, s->W_r, s->n_layers, s->n_experts, stream));
  for (int l = 0; l < s->n_layers; ++l) {
    const Layer a(ctx, s, l);
    UP_TRY(unipool_route(ctx, a.x(l), T, a.W_r(), s->sigma[l], a.bias(), s->n_experts, a.idx(), a.gate(),
                         at(s->counts, l, a.m), at(s->score_sum, l, a.m), a.znorm(), a.z(), stream));
    UP_TRY(permute_and_experts(ctx, a, T, a.slot(), stream));
    UP_TRY(unipool_combine(ctx, a.per_row(s->Yp, a.slot(), a.d), a.row_of(), a.gate(), T, a.x(l), a.x(l + 1), stream));
  }
  return UNIPOOL_OK;
}

int unipool_stack_aux_loss(unipool_ctx* ctx, const unipool_stack* s, int32_t T, float alpha, const float* fbar_prev,
                           unipool_stream stream) {
  UP_TRY(check_stack(ctx, s));
  const int64_t m = s->n_experts, lg = s->layers_per_group;
  for (int g = 0; g < s->n_layers / lg; ++g)
    UP_TRY(unipool_pool_aux_loss(ctx, at(s->counts, g * lg, m), at(s->score_sum, g * lg, m), (int32_t)lg, s->n_experts, T,
                                 alpha, at(fbar_prev, g, m), at(s->loss, g, 1), at(s->coef, g, m), at(s->fbar, g, m), stream));
  return UNIPOOL_OK;
}

int unipool_stack_backward(unipool_ctx* ctx, const unipool_stack* s, int32_t T, int32_t flags, unipool_stream stream) {
  UP_TRY(check_stack(ctx, s));
  UP_REQUIRE((flags & ~(UNIPOOL_WGRAD_OVERWRITE | UNIPOOL_STACK_NO_AUX | UNIPOOL_STACK_LEAVE_WGRAD)) == 0,
             UNIPOOL_ERR_INVALID_ARG, "unknown flags 0x%x", flags);
  UP_REQUIRE(s->wgrad_layers >= 1 && s->dx != nullptr, UNIPOOL_ERR_INVALID_ARG, "wgrad_layers = %d, or dx is NULL",
             s->wgrad_layers);
  const int lg = s->layers_per_group, overwrite = flags & UNIPOOL_WGRAD_OVERWRITE;
  const int run = s->wgrad_layers < lg ? s->wgrad_layers : lg;            // layers contracted together
  // operands of the layer's weight gradient: stacked over all layers, or slots of one run
  const bool stacked = !s->recompute && run > 1;
  int cur = 0;
  for (int l = s->n_layers - 1; l >= 0; --l, cur ^= 1) {
    const Layer a(ctx, s, l);
    const int i = l % lg, hold = i % run;
    const int w = s->recompute ? hold : l;                                // Xp, A
    const int b = stacked ? l : hold;                                     // dYp, dGU
    // the first contribution to a group's experts: its top layer, or the run that layer belongs to
    const int over = overwrite && i >= (lg - 1) / run * run ? UNIPOOL_WGRAD_OVERWRITE : 0;
    if (s->recompute) UP_TRY(permute_and_experts(ctx, a, T, w, stream));
    void *dx_next = at_bytes(s->dx, cur, a.T * a.d * a.eb), *dx_out = at_bytes(s->dx, cur ^ 1, a.T * a.d * a.eb);
    UP_TRY(unipool_expert_bwd_rows(ctx, dx_next, T, a.row_of(), a.gate(), a.token_of(), a.offsets(), a.rows(),
                                   a.tile_expert(), a.per_row(s->Xp, w, a.d), a.per_row(s->GU, a.slot(), 2 * a.f),
                                   a.per_row(s->A, w, a.f), a.per_row(s->Yp, a.slot(), a.d), s->W_gu, s->W_down, a.base(),
                                   s->n_experts, dx_next, a.per_row(s->dYp, b, a.d), a.per_row(s->dGU, b, 2 * a.f), dx_out,
                                   s->dgate, s->dW_gu, s->dW_down, run > 1 ? UNIPOOL_BWD_SKIP_WGRAD : over, stream));
    UP_TRY(unipool_route_bwd(ctx, a.x(l), T, a.W_r(), s->sigma[l], s->n_experts, a.znorm(), a.z(), a.idx(), s->dgate,
                             (flags & UNIPOOL_STACK_NO_AUX) ? nullptr : at(s->coef, l / lg, a.m), dx_out, a.dW_r(),
                             at(s->dsigma, l, 1), stream));
    if (run > 1 && !stacked && hold == 0)                                 // the lowest layer of a run
      UP_TRY(unipool_pool_wgrad_rows(ctx, run < lg - i ? run : lg - i, a.cap, a.offsets(), a.rows(), s->Xp, s->A, s->dYp,
                                     s->dGU, a.base(), s->n_experts, s->dW_gu, s->dW_down, over, stream));
  }
  if (!stacked || (flags & UNIPOOL_STACK_LEAVE_WGRAD)) return UNIPOOL_OK;
  for (int l0 = 0; l0 < s->n_layers; l0 += lg) {                          // one pass per sharing group over its layers
    const Layer a(ctx, s, l0);
    UP_TRY(unipool_pool_wgrad_rows(ctx, lg, a.cap, a.offsets(), a.rows(), a.per_row(s->Xp, l0, a.d), a.per_row(s->A, l0, a.f),
                                   a.per_row(s->dYp, l0, a.d), a.per_row(s->dGU, l0, 2 * a.f), a.base(), s->n_experts,
                                   s->dW_gu, s->dW_down, overwrite, stream));
  }
  return UNIPOOL_OK;
}

}  // extern "C"
