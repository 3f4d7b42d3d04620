// The epoch body of Algorithm 1 as one call: for every layer pull (predict) -> forward -> push, then loss, backward, commit and parameter
// step, on buffers the caller describes once.  It only strings the entry points together; what it saves is the host time between them
// (marshalling of ~10 calls per partition took longer than the kernels of a graph of a few thousand nodes).
#include "sat_internal.h"

static sat_status epoch_pass(sat_ctx *ctx, const sat_epoch_buffers *e, int32_t part, bool first, int grad_history)
{
    const int accumulate = first ? 0 : SAT_BWD_ACCUMULATE, reuse_state = first ? 0 : 1;
    PartView v;
    SAT_TRY(sat_part_view(ctx, part, &v));
    const int32_t L = e->n_layers;
    const float *h_in = e->x;
    int32_t ld_in = e->ld_x;
    for (int32_t l = 1; l <= L; ++l) {
        int act = l < L ? SAT_ACT_RELU | SAT_FWD_PUSH : SAT_ACT_NONE;
        const float *halo = nullptr;
        const sat_pred_params *p = l > 1 && e->pred ? e->pred[l - 2] : nullptr;
        if (l == 1) {
            // in- and out-of-subgraph rows are raw features, exact: the layer reads both from the feature matrix itself
            act |= SAT_FWD_INPUT_GLOBAL;
        } else if (!p) {
            act |= SAT_FWD_HALO_CACHED;   // plain historical embeddings: read from the ring
        } else {
            float *hv = e->halo + v.halo0 * e->ld_halo;
            SAT_TRY(sat_predict(ctx, l - 1, part, p, reuse_state, hv, e->ld_halo));
            halo = hv;
        }
        float *h_out = e->h[l - 1] + (int64_t)v.row0 * e->ld_h[l - 1];
        SAT_TRY(sat_layer_fwd(ctx, part, l, e->dims[l - 1], e->dims[l], h_in, ld_in, halo, halo ? e->ld_halo : 0, e->w[l - 1], e->b[l - 1], act, h_out,
                              e->ld_h[l - 1]));
        h_in = h_out;
        ld_in = e->ld_h[l - 1];
    }
    const int32_t C = e->dims[L];
    const char *labels = (const char *)e->labels + (int64_t)v.row0 * (e->loss_kind == SAT_LOSS_SOFTMAX_CE ? (int64_t)sizeof(int32_t) : C);
    const float *g = e->g[L - 1] + (int64_t)v.row0 * e->ld_g[L - 1];
    SAT_TRY(sat_loss_into(ctx, part, e->loss_kind, C, h_in, ld_in, labels, e->loss_sum, (float *)g, e->ld_g[L - 1], first));
    for (int32_t l = L; l >= 1; --l) {
        float *g_in = l > 1 ? e->g[l - 2] + (int64_t)v.row0 * e->ld_g[l - 2] : nullptr;
        // the gradient handed down is written already multiplied by the ReLU mask of the layer below (no separate pass)
        const int flags = accumulate | (l > 1 ? SAT_BWD_MASK_G_IN : 0) | (l < L ? SAT_BWD_G_OUT_MASKED : 0) | (grad_history && l > 1 ? SAT_BWD_GRAD_HISTORY : 0);
        SAT_TRY(sat_layer_bwd(ctx, part, l, g, e->ld_g[l - 1], e->w[l - 1], e->gw[l - 1], e->gb[l - 1], flags, g_in, l > 1 ? e->ld_g[l - 2] : 0, nullptr, 0));
        g = g_in;
    }
    return SAT_OK;
}

// What the calls of a pass would refuse, before the first of them has written anything.
static sat_status epoch_check(sat_ctx *ctx, const sat_epoch_buffers *e, const int32_t *order, int32_t n_order, int flags)
{
    if (!e || e->n_layers < 1 || e->n_layers > SAT_MAX_LAYERS || !e->dims || !e->x || !e->labels || !e->h || !e->ld_h || !e->g || !e->ld_g || !e->w || !e->b ||
        !e->gw || !e->gb || (n_order != 0 && !order) || n_order < 0 || (flags & ~(SAT_EPOCH_GRAD_HISTORY | SAT_EPOCH_COMMIT | SAT_EPOCH_STEP | SAT_EPOCH_CONTINUE)))
        return sat_fail(ctx, SAT_EINVAL, "sat_epoch: incomplete description or unknown flags");
    PartView v;
    for (int32_t i = 0; i < (n_order > 0 ? n_order : 1); ++i) SAT_TRY(sat_part_view(ctx, n_order > 0 ? order[i] : (int32_t)SAT_ALL_PARTS, &v));
    const int32_t L = e->n_layers;
    if (e->loss_kind != SAT_LOSS_SOFTMAX_CE && e->loss_kind != SAT_LOSS_SIGMOID_BCE) return sat_fail(ctx, SAT_EINVAL, "sat_epoch: unknown loss");
    if ((L > 1 || (flags & SAT_EPOCH_COMMIT)) && !ctx->cache_ok) return sat_fail(ctx, SAT_ESTATE, "sat_epoch: call sat_cache_init first");
    if (e->dims[0] <= 0 || !ok_ld(e->ld_x, e->dims[0]) || !aligned16(e->x)) return sat_fail(ctx, SAT_EINVAL, "sat_epoch: misaligned x or bad leading dimension");
    for (int32_t l = 0; l < L; ++l) {
        const int32_t d = e->dims[l + 1];
        if (!e->w[l] || !e->gw[l] || !e->h[l] || !e->g[l]) return sat_fail(ctx, SAT_EINVAL, "sat_epoch: null array of layer %d", l + 1);
        if (d <= 0 || !ok_ld(e->ld_h[l], d) || !ok_ld(e->ld_g[l], d) || !aligned16(e->h[l]) || !aligned16(e->g[l]))
            return sat_fail(ctx, SAT_EINVAL, "sat_epoch: misaligned rows or bad leading dimension of layer %d", l + 1);
        if (l + 1 == L) break;
        if (l >= ctx->n_cached || ctx->cache[l].width != d) return sat_fail(ctx, SAT_EINVAL, "sat_epoch: layer %d is not cached at width %d", l + 1, d);
        const sat_pred_params *p = e->pred ? e->pred[l] : nullptr;
        if (!p) continue;
        if (p->h <= 0 || (p->h & 3) || !p->Wx || !p->Uh || !p->b || !p->Wg || !p->bg || (p->cell != SAT_CELL_LSTM && p->cell != SAT_CELL_GRU))
            return sat_fail(ctx, SAT_EINVAL, "sat_epoch: bad predictor of layer %d", l + 1);
        if ((flags & SAT_EPOCH_CONTINUE) && !(order && n_order == 0) && (!ctx->cache[l].S_valid || ctx->cache[l].S_h != p->h))
            return sat_fail(ctx, SAT_ESTATE, "sat_epoch: no state table of layer %d to go on with", l + 1);
        if (ctx->nb > 0 && (!e->halo || !ok_ld(e->ld_halo, d) || !aligned16(e->halo)))
            return sat_fail(ctx, SAT_EINVAL, "sat_epoch: no room for the predicted rows of layer %d", l + 1);
    }
    return SAT_OK;
}

extern "C" sat_status sat_epoch(sat_ctx *ctx, const sat_epoch_buffers *e, const int32_t *order, int32_t n_order, int flags, float lr)
{
    CHECK_CTX(ctx);
    SAT_TRY(epoch_check(ctx, e, order, n_order, flags));
    const bool begin = !(flags & SAT_EPOCH_CONTINUE);
    for (int32_t l = 0; l <= SAT_MAX_LAYERS; ++l) ctx->layers[l].packed_as[0] = ctx->layers[l].packed_as[1] = 0;
    ctx->keep_packed = order && n_order > 1;   // the parameter step comes after the passes
    sat_status st = SAT_OK;
    for (int32_t i = 0; i < (order ? n_order : 1) && st == SAT_OK; ++i)
        st = epoch_pass(ctx, e, order ? order[i] : (int32_t)SAT_ALL_PARTS, i == 0 && begin, flags & SAT_EPOCH_GRAD_HISTORY);
    ctx->keep_packed = false;
    SAT_TRY(st);
    if (order && n_order == 0 && begin && e->loss_sum) SAT_CUDA(ctx, cudaMemsetAsync(e->loss_sum, 0, sizeof(double), ctx->stream));   // the loss of no partition
    if (flags & SAT_EPOCH_COMMIT) SAT_TRY(sat_cache_commit(ctx));
    if (flags & SAT_EPOCH_STEP) {
        int64_t counts[2 * SAT_MAX_LAYERS];
        float *w[2 * SAT_MAX_LAYERS];
        const float *g[2 * SAT_MAX_LAYERS];
        int32_t k = 0;
        for (int32_t l = 0; l < e->n_layers; ++l, ++k) {
            counts[k] = (int64_t)e->dims[l] * e->dims[l + 1];
            w[k] = e->w[l];
            g[k] = e->gw[l];
        }
        for (int32_t l = 0; l < e->n_layers; ++l) {
            if (!e->b[l] || !e->gb[l]) continue;
            counts[k] = e->dims[l + 1];
            w[k] = e->b[l];
            g[k++] = e->gb[l];
        }
        SAT_TRY(sat_sgd_steps(ctx, k, counts, w, g, lr));
    }
    return SAT_OK;
}
