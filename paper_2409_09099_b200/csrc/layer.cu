// One call per phase of a layer's iteration (prune, forward, backward): the calls of the path in order, on the buffers of an
// sste_layer.  A caller in an interpreted language pays for one call instead of two to four, each with a dozen arguments
// to convert: on a 256 x 256 layer that conversion, not the GPU, set the pace.
#include <initializer_list>

#include "common.cuh"

namespace {

bool fp8_of(const sste_layer *l) { return l->op_dtype == SSTE_E4M3; }

// bf16 with none of the FP8 buffers, or E4M3 with all of them
bool layer_ok(const sste_layer *l)
{
    if (!l || (l->op_dtype != SSTE_BF16 && l->op_dtype != SSTE_E4M3)) return false;
    return !fp8_of(l) || (l->amax && l->Xq && l->dYq && l->scratch);
}

// What the kernels of a phase ask of the layer, looked at before the first of them is launched: sizes, and the buffers that
// they need.  (A prune does not look at T.)
sste_status phase_ok(const sste_layer *l, int T, std::initializer_list<const void *> needed)
{
    for (const void *b : needed)
        if (!b) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(l->O) || !sste_mult128(l->I) || !sste_mult128(T)) return SSTE_ERR_SHAPE;
    for (const void *b : needed)
        if (!sste_aligned(b, 128)) return SSTE_ERR_ALIGN;
    return fp8_of(l) && (!sste_aligned(l->amax, 4) || !sste_aligned(l->scratch, 8)) ? SSTE_ERR_ALIGN : SSTE_OK;
}
// Where the blocks of a one-launch maximum leave theirs, behind the scratch's first 8 bytes; null if there is no room.
unsigned int *slots_of(const sste_layer *l)
{
    return l->scratch_bytes == SSTE_LAYER_SCRATCH_BYTES ? static_cast<unsigned int *>(l->scratch) + 2 : nullptr;
}

bool out_dtype_ok(const sste_layer *l) { return l->out_dtype == SSTE_BF16 || l->out_dtype == SSTE_F32; }

sste_status forward_ok(const sste_layer *l, const void *X)
{
    if (!out_dtype_ok(l)) return SSTE_ERR_DTYPE;
    if (fp8_of(l) && !sste_aligned(X, 16)) return SSTE_ERR_ALIGN;      // read by the amax and quantising passes only
    return phase_ok(l, l->T, {l->vals, l->meta, l->Y, fp8_of(l) ? l->Xq : X});
}
sste_status grads_ok(const sste_layer *l, const void *X, const void *dY)
{
    if (!out_dtype_ok(l)) return SSTE_ERR_DTYPE;
    const bool fp8 = fp8_of(l);
    const void *v = l->w_dense ? l->w_dense : l->vals, *m = l->w_dense ? l->w_dense : l->meta;
    return phase_ok(l, l->T, {l->gvals, l->gmeta, fp8 ? l->Xq : X, fp8 ? l->dYq : dY, v, m, l->dW, l->dX});
}
sste_status backward_ok(const sste_layer *l, const void *X, const void *dY, uint64_t token_offset)
{
    const sste_status st = grads_ok(l, X, dY);
    if (st != SSTE_OK) return st;
    if (l->counter_cols < 0 || l->counter_cols > l->O) return SSTE_ERR_INVALID_ARG;
    if (token_offset % 4 != 0) return SSTE_ERR_SHAPE;
    return sste_aligned(dY, 128) ? SSTE_OK : SSTE_ERR_ALIGN;
}

// The status of the product that should have emptied the layer's scratch; if a call was refused, a memset does.
sste_status emptied(const sste_layer *l, sste_status st, void *stream)
{
    if (st != SSTE_OK) cudaMemsetAsync(l->scratch, 0, 8, static_cast<cudaStream_t>(stream));
    return st;
}

}  // namespace

extern "C" sste_status sste_layer_prune(sste_ctx *ctx, const sste_layer *l, void *stream)
{
    if (!ctx || !layer_ok(l) || !l->beta) return SSTE_ERR_INVALID_ARG;
    const sste_status ok = phase_ok(l, 128, {l->W, l->vals, l->meta, l->w_dense ? l->w_dense : l->vals});
    if (ok != SSTE_OK) return ok;
    if (!fp8_of(l))
        return sste_project_compress(ctx, l->W, l->O, l->I, SSTE_BF16, l->beta, nullptr, SSTE_BF16, l->vals, l->meta, l->w_dense,
                                     stream);
    if (slots_of(l) && sste_project_fp8_fits(ctx, l->O, l->I))
        return sste_project_fp8(ctx, l->W, l->O, l->I, l->beta, l->amax + 1, slots_of(l), l->vals, l->meta, l->w_dense, stream);
    sste_status st = sste_project_amax_scratch(ctx, l->W, l->O, l->I, l->beta, l->amax + 1, l->scratch, stream);
    if (st != SSTE_OK) return st;
    return sste_project_compress(ctx, l->W, l->O, l->I, SSTE_BF16, l->beta, l->amax + 1, SSTE_E4M3, l->vals, l->meta, l->w_dense,
                                 stream);
}

extern "C" sste_status sste_layer_forward(sste_ctx *ctx, const sste_layer *l, const void *X, float *y_amax_out_dev, void *stream)
{
    if (!ctx || !layer_ok(l) || !X) return SSTE_ERR_INVALID_ARG;
    const sste_status ok = forward_ok(l, X);
    if (ok != SSTE_OK) return ok;
    float *x_amax = nullptr, *w_amax = nullptr;
    if (fp8_of(l)) {
        x_amax = l->amax;
        w_amax = l->amax + 1;
        const size_t n = static_cast<size_t>(l->T) * l->I;
        if (slots_of(l) && sste_amax_quantize_fits(ctx, n)) {
            const sste_status st = sste_amax_quantize(ctx, X, n, x_amax, slots_of(l), l->Xq, stream);
            if (st != SSTE_OK) return st;
            return sste_linear_fwd(ctx, l->Xq, l->T, l->vals, l->meta, l->O, l->I, SSTE_E4M3, x_amax, w_amax, l->Y,
                                   static_cast<sste_dtype>(l->out_dtype), y_amax_out_dev, stream);
        }
        sste_status st = sste_amax_scratch(ctx, X, n, x_amax, l->scratch, stream);
        if (st != SSTE_OK) return st;
        st = sste_quantize_scratch(ctx, X, n, x_amax, l->scratch, l->Xq, stream);
        if (st == SSTE_OK) {
            sste_ctx emptying = *ctx;
            emptying.zero_after = static_cast<unsigned int *>(l->scratch);
            st = sste_linear_fwd(&emptying, l->Xq, l->T, l->vals, l->meta, l->O, l->I, SSTE_E4M3, x_amax, w_amax, l->Y,
                                 static_cast<sste_dtype>(l->out_dtype), y_amax_out_dev, stream);
        }
        return emptied(l, st, stream);
    }
    return sste_linear_fwd(ctx, X, l->T, l->vals, l->meta, l->O, l->I, SSTE_BF16, nullptr, nullptr, l->Y,
                           static_cast<sste_dtype>(l->out_dtype), y_amax_out_dev, stream);
}

extern "C" sste_status sste_layer_backward(sste_ctx *ctx, const sste_layer *l, const void *X, const void *dY, uint32_t step,
                                           uint64_t token_offset, void *stream)
{
    if (!ctx || !layer_ok(l) || !dY) return SSTE_ERR_INVALID_ARG;
    sste_status st = backward_ok(l, X, dY, token_offset);
    if (st != SSTE_OK) return st;
    if (fp8_of(l)) {
        float *g_amax = l->amax + 2;
        st = sste_amax_scratch(ctx, dY, static_cast<size_t>(l->T) * l->O, g_amax, l->scratch, stream);
        if (st != SSTE_OK) return st;
        st = sste_mvue_scratch(ctx, dY, l->T, l->O, l->seed, l->tensor_id, step, token_offset, l->counter_cols, g_amax,
                               l->scratch, l->gvals, l->gmeta, l->dYq, stream);
        if (st == SSTE_OK) {
            sste_ctx emptying = *ctx;
            emptying.zero_after = static_cast<unsigned int *>(l->scratch);
            st = sste_layer_grads(&emptying, l, X, dY, stream);
        }
        return emptied(l, st, stream);
    } else {
        st = sste_mvue_sparsify(ctx, dY, l->T, l->O, SSTE_BF16, l->seed, l->tensor_id, step, token_offset, l->counter_cols, nullptr,
                                SSTE_BF16, l->gvals, l->gmeta, nullptr, stream);
    }
    if (st != SSTE_OK) return st;
    return sste_layer_grads(ctx, l, X, dY, stream);
}

extern "C" sste_status sste_layer_grads(sste_ctx *ctx, const sste_layer *l, const void *X, const void *dY, void *stream)
{
    if (!ctx || !layer_ok(l) || !dY) return SSTE_ERR_INVALID_ARG;
    const sste_status ok = grads_ok(l, X, dY);
    if (ok != SSTE_OK) return ok;
    const bool fp8 = fp8_of(l);
    return sste_bwd_products(ctx, l->gvals, l->gmeta, fp8 ? l->Xq : X, fp8 ? l->dYq : dY, l->O, l->I, l->T,
                             fp8 ? SSTE_E5M2 : SSTE_BF16, static_cast<sste_dtype>(l->op_dtype), l->w_dense, l->vals, l->meta,
                             fp8 ? l->amax + 2 : nullptr, fp8 ? l->amax : nullptr, fp8 ? l->amax + 1 : nullptr, l->dW, l->dX,
                             static_cast<sste_dtype>(l->out_dtype), stream);
}

namespace {
bool one_launch(const sste_ctx *ctx, const sste_layer *l, bool beside)
{
    if (!ctx || !layer_ok(l) || !sste_mult128(l->O) || !sste_mult128(l->I) || !sste_mult128(l->T)) return false;
    return sste_bwd_in_one_launch(ctx, fp8_of(l) ? 1 : 2, l->O, l->I, l->T, l->w_dense != nullptr,
                                  static_cast<sste_dtype>(l->out_dtype), beside);
}
}  // namespace

extern "C" int sste_layer_grads_joint(const sste_ctx *ctx, const sste_layer *l) { return one_launch(ctx, l, false); }
extern "C" int sste_layer_grads_beside(const sste_ctx *ctx, const sste_layer *l) { return !one_launch(ctx, l, true); }

namespace {

bool padded_ok(const sste_padded_layer *l)
{
    return l && layer_ok(&l->inner) && l->inner.out_dtype == SSTE_BF16 && l->Xp && l->dYp && l->O > 0 && l->I > 0 && l->T > 0 &&
           l->O <= l->inner.O && l->I <= l->inner.I && l->T <= l->inner.T;
}

}  // namespace

extern "C" sste_status sste_padded_forward(sste_ctx *ctx, const sste_padded_layer *l, const void *X, void *stream)
{
    if (!ctx || !padded_ok(l) || !X) return SSTE_ERR_INVALID_ARG;
    const sste_layer &in = l->inner;
    sste_status st = forward_ok(&in, l->Xp);
    if (st == SSTE_OK && (!sste_aligned(X, 2) || !sste_aligned(l->Y, 2))) st = SSTE_ERR_ALIGN;
    if (st == SSTE_OK) st = sste_pad_2d(ctx, X, l->T, l->I, l->Xp, in.T, in.I, stream);
    if (st == SSTE_OK) st = sste_layer_forward(ctx, &in, l->Xp, nullptr, stream);
    if (st == SSTE_OK && l->Y) st = sste_crop_2d(ctx, in.Y, in.T, in.O, l->Y, l->T, l->O, stream);
    return st;
}

extern "C" sste_status sste_padded_backward(sste_ctx *ctx, const sste_padded_layer *l, const void *dY, uint32_t step,
                                            uint64_t token_offset, void *stream)
{
    if (!ctx || !padded_ok(l) || !dY) return SSTE_ERR_INVALID_ARG;
    const sste_layer &in = l->inner;
    sste_status st = backward_ok(&in, l->Xp, l->dYp, token_offset);
    if (st == SSTE_OK && (!sste_aligned(dY, 2) || !sste_aligned(l->dX, 2) || !sste_aligned(l->dW, 2))) st = SSTE_ERR_ALIGN;
    if (st != SSTE_OK) return st;
    if (fp8_of(&in)) {       // the quantisation needs max|dY| before the sparsification reads it
        st = sste_pad_2d(ctx, dY, l->T, l->O, l->dYp, in.T, in.O, stream);
        if (st == SSTE_OK) st = sste_layer_backward(ctx, &in, l->Xp, l->dYp, step, token_offset, stream);
    } else {
        st = sste_mvue_padded(ctx, dY, l->T, l->O, l->dYp, in.T, in.O, in.seed, in.tensor_id, step, token_offset, in.counter_cols,
                              in.gvals, in.gmeta, stream);
        if (st == SSTE_OK) st = sste_layer_grads(ctx, &in, l->Xp, l->dYp, stream);
    }
    if (st != SSTE_OK) return st;
    if (l->dX && l->dW)
        return sste_crop_two(ctx, in.dX, in.T, in.I, l->dX, l->T, l->I, in.dW, in.O, in.I, l->dW, l->O, l->I, stream);
    if (l->dX) return sste_crop_2d(ctx, in.dX, in.T, in.I, l->dX, l->T, l->I, stream);
    if (l->dW) return sste_crop_2d(ctx, in.dW, in.O, in.I, l->dW, l->O, l->I, stream);
    return SSTE_OK;
}
