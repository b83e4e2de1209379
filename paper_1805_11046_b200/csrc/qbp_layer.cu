// Whole quantised layer (Sections 4 and 6): the composition of the library's
// own entry points in the order the method prescribes.
//   forward : quantise x, w to 8 bits (nearest) -> 8-bit product -> Range BN (+ReLU)
//   backward: Range BN backward -> gradient bifurcation (8-bit and 16-bit copies,
//             stochastic rounding) -> layer gradient from the 8-bit copy and the
//             forward's weight codes; weight gradient from the 16-bit copy and
//             the forward's input codes.
// The straight-through estimator through the quantiser is the identity here:
// the clamping values are the tensor's own min and max, so nothing is clipped.
// Everything is enqueued on the caller's stream; temporaries live in the
// caller's workspace.
#include "qbp_mma.cuh"

#include <algorithm>

namespace qbp {

struct LayerShape {
    bool conv;
    int64_t rows;        // batch, or N*H*W
    int64_t cin, cout;   // reduced / produced channels of the forward product
    int64_t x_elems, w_elems;
};

static int layer_shape(const qbp_layer_desc *L, LayerShape &s)
{
    if (!L) return fail(QBP_ERR_INVALID_ARG, "layer: descriptor is NULL");
    s.conv = L->conv.R != 0;
    if (s.conv) {
        const qbp_conv_desc &d = L->conv;
        if (d.N <= 0 || d.H <= 0 || d.W <= 0 || d.C <= 0 || d.K <= 0 || d.R <= 0 || d.S <= 0)
            return fail(QBP_ERR_INVALID_ARG, "layer: bad convolution geometry");
        // what every product of the step implements, checked before anything is launched
        if (!conv_supported(&d) || !wgrad_conv_supported(&d))
            return fail(QBP_ERR_UNSUPPORTED_SHAPE,
                        "layer: needs stride 1, R = S in {1,3}, pad = (R-1)/2, C and K multiples of 32");
        if ((int64_t)d.R * d.S * std::max(d.C, d.K) > 33025)
            return fail(QBP_ERR_OVERFLOW_K, "layer: reduction length exceeds 33025");
        s.rows = (int64_t)d.N * d.H * d.W; s.cin = d.C; s.cout = d.K;
        s.x_elems = s.rows * d.C; s.w_elems = (int64_t)d.K * d.R * d.S * d.C;
    } else {
        if (L->batch <= 0 || L->in_features <= 0 || L->out_features <= 0)
            return fail(QBP_ERR_INVALID_ARG, "layer: batch, in_features, out_features must be positive");
        if (L->batch % 16 || L->in_features % 16 || L->out_features % 16)
            return fail(QBP_ERR_UNSUPPORTED_SHAPE, "layer: batch, in_features, out_features must be multiples of 16");
        if (L->in_features > 33025 || L->out_features > 33025)
            return fail(QBP_ERR_OVERFLOW_K, "layer: in_features and out_features are reduction lengths of 8-bit products (at most 33025)");
        s.rows = L->batch; s.cin = L->in_features; s.cout = L->out_features;
        s.x_elems = s.rows * s.cin; s.w_elems = s.cin * s.cout;
    }
    if (s.rows < 2) return fail(QBP_ERR_INVALID_ARG, "layer: Range BN needs at least 2 rows");
    return QBP_OK;
}

// The layer's workspace: [0, kLayerHead) the sticky status word of the whole step (cleared once by the forward
// call, raised by any product whose bounded wait runs out, never overwritten by a later step), then the scratch
// the steps share (they run one after another on the stream), then the buffers that live across steps.
constexpr size_t kLayerHead = 256;

static size_t step_scratch_bytes(const qbp_layer_desc *L, const LayerShape &s)
{
    size_t b = std::max(quantize_operands_ws_bytes(), qbp_quantize_workspace_bytes(s.rows, std::max(s.cin, s.cout), QBP_PER_TENSOR));
    b = std::max(b, qbp_rangebn_workspace_bytes(s.rows, s.cout));
    if (s.conv) {
        b = std::max(b, qbp_conv_s8_workspace_bytes(QBP_CONV_FPROP, &L->conv));
        b = std::max(b, qbp_wgrad_s16_workspace_bytes(&L->conv, 0, 0, 0));
    } else {
        b = std::max({b, qbp_gemm_s8_workspace_bytes(s.rows, s.cout, s.cin), qbp_gemm_s8_workspace_bytes(s.rows, s.cin, s.cout)});
        b = std::max(b, qbp_wgrad_s16_workspace_bytes(nullptr, s.rows, s.cout, s.cin));
    }
    return align_up(b, 256);
}

// (a convolution's epilogue takes the output's per-channel statistics for any number of channels that leaves a CTA one
// column tile: 256 channels per tile, one CTA per SM)
static bool epilogue_stats(const LayerShape &s) { return s.conv && (s.cout + 255) / 256 <= sm_count(); }
static size_t colstat_cells(const LayerShape &s) { return epilogue_stats(s) ? (size_t)colstat_rows_max() * (size_t)s.cout : 0; }
// The layer's own pieces of the workspace, in order.
struct LayerWs {
    int *status;                 // byte 0 of the workspace
    void *scratch; size_t scratch_bytes;
    int32_t *row_sums;           // [rows] code sums of the operand of the next product
    float2 *range_parts;         // range partials of the gradient
    ColStatParts parts;          // per-channel (sum, min, max) partials of the output, from the convolution's epilogue
    float4 *fold;                // per-channel constants of the normalisation, for the recompute fusion
    int64_t *tot_g;              // [cout] per-channel totals of the 16-bit gradient codes, and behind them ...
    int64_t *wg_table;           // ... the table of the weight gradient's sums (NULL: in pieces): cleared together
    int64_t clear_words;
    int32_t *w_sums;             // the weights' code sums: forward, then layer gradient
    SumJob wg_sums[6];           // the weight gradient's code sums (count: wg_count)
    int wg_count;
    size_t bytes;
};
static SumJob weight_sum_job(const qbp_layer_desc *L, const LayerShape &s, bool bwd, const int8_t *w, int32_t *out)
{
    if (s.conv) return filter_sum_job(&L->conv, bwd, w, out);
    return bwd ? SumJob{w, s.cin, s.cout, kSumRows, 1, out} : SumJob{w, s.cin, s.cout, kSumCols, 1, out};
}
static LayerWs layer_ws(const qbp_layer_desc *L, const LayerShape &s, void *ws, const int8_t *x = nullptr, const int8_t *hi = nullptr,
                        const uint8_t *lo = nullptr)
{
    LayerWs l{};
    WsCarver c(ws, SIZE_MAX);
    l.status = c.take<int>(kLayerHead / sizeof(int));
    l.scratch_bytes = step_scratch_bytes(L, s);
    l.scratch = c.take<char>(l.scratch_bytes);
    l.row_sums = c.take<int32_t>((size_t)s.rows);
    l.range_parts = c.take<float2>(rangebn_range_parts_capacity(s.cout));
    const size_t cells = colstat_cells(s);
    if (cells) { l.parts.lo = c.take<float>(cells); l.parts.hi = c.take<float>(cells); l.parts.sum = c.take<double>(cells); }
    l.fold = c.take<float4>((size_t)s.cout);
    const qbp_conv_desc *d = s.conv ? &L->conv : nullptr;
    const size_t table = wgrad_sum_table(d, s.rows, s.cout, s.cin);
    l.tot_g = c.take<int64_t>((size_t)s.cout + table);
    l.wg_table = table ? l.tot_g + s.cout : nullptr;
    l.clear_words = table ? 2 * ((int64_t)s.cout + (int64_t)table) : 0;
    l.w_sums = c.take<int32_t>(std::max(sum_elems(weight_sum_job(L, s, false, nullptr, nullptr)), sum_elems(weight_sum_job(L, s, true, nullptr, nullptr))));
    l.wg_count = wgrad_sum_jobs(d, s.rows, s.cout, s.cin, x, hi, lo, true, l.wg_table, l.wg_sums);
    for (int i = 0; i < l.wg_count && !table; ++i) l.wg_sums[i].out = c.take<int32_t>(sum_elems(l.wg_sums[i]));
    l.bytes = c.off;
    return l;
}

// Recompute instead of store (motivated by Section 7's memory and bandwidth argument): convolution -> Range BN
// (+ReLU) -> 8-bit codes for the next layer without ever writing the fp32 output of the product.  The
// convolution runs twice: the first run leaves only the per-channel statistics (its epilogue stores nothing), the
// second run normalises, rectifies and requantises in its epilogue and writes one byte per output.
static int conv_rangebn_recompute(const qbp_conv_desc *d, const int8_t *x_codes, const qbp_qparams *qx, const int32_t *in_sums,
                                  const int8_t *w_codes, const qbp_qparams *qw, const float *gamma, const float *beta, int relu,
                                  float *save_mean, float *save_min, float *save_max, const qbp_requant *out,
                                  ColStatParts parts, float4 *fold, const CodeSums &w_sums, int *status, void *ws, size_t scratch,
                                  bool beside, const SumJob *extra, int extra_count, bool totals_cleared, cudaStream_t st)
{
    const int64_t rows = (int64_t)d->N * d->H * d->W;
    const EpilogueTail first{nullptr, 0, nullptr, nullptr, nullptr, 0, &w_sums, extra, extra_count, beside};
    int rc = conv_s8_impl(QBP_CONV_FPROP, d, x_codes, qx, w_codes, qw, nullptr, nullptr, in_sums, &parts, status, ws, scratch, st,
                          &first);
    if (rc) return rc;
    if ((rc = rangebn_fold_from_parts(rows, d->K, gamma, beta, relu, save_mean, save_min, save_max, parts, out->qp, fold, st))) return rc;
    const EpilogueTail tail{fold, relu, out->qp, out->q, out->row_sums, 1, &w_sums};
    rc = conv_s8_impl(QBP_CONV_FPROP, d, x_codes, qx, w_codes, qw, nullptr, nullptr, in_sums, nullptr, status, ws, scratch, st, &tail);
    if (rc || !out->chan_sums) return rc;
    return launch_colsum(out->q, true, rows, d->K, out->chan_sums, st, totals_cleared);
}

}  // namespace qbp

using namespace qbp;

extern "C" __attribute__((visibility("default"))) size_t qbp_layer_workspace_bytes(const qbp_layer_desc *L)
{
    LayerShape s;
    if (layer_shape(L, s)) return 0;
    return layer_ws(L, s, nullptr).bytes;
}

extern "C" __attribute__((visibility("default"))) int qbp_layer_fwd(const qbp_layer_desc *L, const float *x,
                                                                   const float *w, const float *gamma,
                                                                   const float *beta, float *y,
                                                                   const qbp_layer_ctx *saved, void *ws,
                                                                   size_t ws_bytes, void *stream)
{
    if (!x || !y) return fail(QBP_ERR_INVALID_ARG, "layer_fwd: NULL argument");
    return qbp_layer_fwd_chained(L, x, nullptr, w, gamma, beta, y, nullptr, saved, ws, ws_bytes, stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_layer_fwd_chained(const qbp_layer_desc *L, const float *x,
                                                                           const qbp_requant *in, const float *w,
                                                                           const float *gamma, const float *beta,
                                                                           float *y, const qbp_requant *out,
                                                                           const qbp_layer_ctx *saved, void *ws,
                                                                           size_t ws_bytes, void *stream)
{
    LayerShape s;
    int rc = layer_shape(L, s);
    if (rc) return rc;
    if (!w || !saved) return fail(QBP_ERR_INVALID_ARG, "layer_fwd: NULL argument");
    if ((x != nullptr) == (in != nullptr))
        return fail(QBP_ERR_INVALID_ARG, "layer_fwd: exactly one of x (fp32 input) and in (input already quantised) is needed");
    if (!y && !out) return fail(QBP_ERR_INVALID_ARG, "layer_fwd: neither y nor 8-bit output codes wanted");
    if (out && (!out->q || !out->qp)) return fail(QBP_ERR_INVALID_ARG, "layer_fwd: the output record needs q and qp");
    if (!saved->x_codes || !saved->qx || !saved->w_codes || !saved->qw || !saved->save_mean ||
        !saved->save_min || !saved->save_max)
        return fail(QBP_ERR_INVALID_ARG, "layer_fwd: the saved-state record has a NULL buffer");
    // saved->z == NULL: the fp32 output of the product is not kept (forward only): the convolution is run twice instead
    const bool recompute = saved->z == nullptr;
    if (recompute && !(s.conv && s.cout <= QBP_EPILOGUE_MAX_COLUMNS && out && !y))
        return fail(QBP_ERR_INVALID_ARG, "layer_fwd: without saved->z the layer must be a convolution of at most %d output "
                    "channels that writes 8-bit codes only (out given, y NULL)", QBP_EPILOGUE_MAX_COLUMNS);
    if (in && (in->q != saved->x_codes || in->qp != saved->qx))
        return fail(QBP_ERR_INVALID_ARG, "layer_fwd: in->q / in->qp must be the layer's saved x_codes / qx");
    const bool want_totals = s.conv && saved->x_chan_sums != nullptr;
    if (want_totals && s.rows >= (1ll << 22)) return fail(QBP_ERR_UNSUPPORTED_SHAPE, "layer_fwd: x_chan_sums for fewer than 2^22 positions");
    if (want_totals && in && in->chan_sums && in->chan_sums != saved->x_chan_sums)
        return fail(QBP_ERR_INVALID_ARG, "layer_fwd: in->chan_sums must be the layer's saved x_chan_sums");
    const LayerWs l = layer_ws(L, s, ws);
    if (!ws || ws_bytes < l.bytes)
        return fail(QBP_ERR_WORKSPACE, "layer_fwd: workspace of %zu bytes needed, %zu given", l.bytes, ws_bytes);
    cudaStream_t st = (cudaStream_t)stream;
    int *status = l.status;

    // activations: nearest rounding, clamping values = min and max (Appendix B) -- or already quantised by the
    // Range BN of the layer before (Section 4); weights the same.  (the first launch also clears the status word)
    const int64_t w_rows = s.conv ? (int64_t)L->conv.K * L->conv.R * L->conv.S : s.cin;
    QuantOperand xo{x, s.rows, s.cin, saved->x_codes, saved->qx, in && in->row_sums ? nullptr : l.row_sums, want_totals ? saved->x_chan_sums : nullptr, nullptr};
    QuantOperand wo{w, w_rows, s.w_elems / w_rows, saved->w_codes, saved->qw, s.conv ? l.w_sums : nullptr, nullptr, s.conv ? nullptr : l.w_sums};
    // (an input that came without its channel totals: cleared with the rest, summed up below; a filter has cin columns)
    const bool chained_totals = !x && want_totals && !in->chan_sums;
    if (chained_totals) wo.tot = saved->x_chan_sums;
    // ... and the totals that the last kernel of this call adds to, so that no launch for it stands between two kernels -- unless a
    // later step of this call refuses it (they then stay as they are), or their memory holds what the steps before that kernel still
    // read or add to
    const bool goes_through = aligned16(saved->x_codes) && aligned16(saved->w_codes) &&
                              (recompute ? aligned16(out->q) : aligned16(saved->z) && s.rows < (1ll << 22));
    const auto apart = [&](const void *p, int64_t bytes) {
        const uintptr_t a = (uintptr_t)p, o = (uintptr_t)out->chan_sums;
        return !p || o + sizeof(int64_t) * (size_t)s.cout <= a || a + (size_t)bytes <= o;
    };
    const bool clear_out = out && out->chan_sums && goes_through && apart(x, 4 * s.x_elems) && apart(w, 4 * s.w_elems) &&
                           apart(saved->x_codes, s.x_elems) && apart(saved->w_codes, s.w_elems) &&
                           apart(want_totals ? saved->x_chan_sums : nullptr, 8 * s.cin) && apart(in ? in->row_sums : nullptr, 4 * s.rows);
    const bool no_launch = !s.conv || L->conv.R == 3 || !want_totals || (x ? quantizer_totals_supported(s.cin) : !chained_totals);
    if ((rc = quantize_operands(x ? &xo : nullptr, &wo, status, l.scratch, l.scratch_bytes, st, no_launch, clear_out ? out->chan_sums : nullptr,
                                clear_out ? 2 * s.cout : 0))) return rc;
    // what the products need beside the codes: each input row's code sum (convolution: each pixel's), the weights' sums,
    // each input channel's total -- whatever the quantising kernel did not leave, in one launch
    SumJob jobs[3];
    int njobs = 0;
    const int32_t *in_sums = l.row_sums;
    if (in && in->row_sums) in_sums = in->row_sums;
    else if (!xo.row_sums_left) jobs[njobs++] = SumJob{saved->x_codes, s.rows, s.cin, kSumRows, 1, l.row_sums};
    const SumJob w_job = weight_sum_job(L, s, false, saved->w_codes, l.w_sums);
    if (!wo.row_sums_left && !wo.col_sums_left) jobs[njobs++] = w_job;
    // (the totals alone, of a 3 x 3 convolution: in the launch of its correction terms)
    const SumJob tot_job{saved->x_codes, s.rows, s.cin, kSumCols, 1, nullptr, 0, 0, saved->x_chan_sums};
    const bool tot_wanted = (want_totals && x && !xo.tot_left) || chained_totals, tot_with_terms = tot_wanted && !njobs && L->conv.R == 3;
    if (tot_wanted && !tot_with_terms) jobs[njobs++] = tot_job;
    bool beside = false;
    if (njobs && (rc = launch_code_sums(jobs, njobs, st, ZeroJobs{}, &beside))) return rc;
    const CodeSums w_sums = sums_of(w_job), x_sums = sums_of(in_sums);
    ColStatParts parts = l.parts;
    if (recompute)
        return conv_rangebn_recompute(&L->conv, saved->x_codes, saved->qx, in_sums, saved->w_codes, saved->qw, gamma, beta, L->relu,
                                      saved->save_mean, saved->save_min, saved->save_max, out, parts, l.fold, w_sums, status,
                                      l.scratch, l.scratch_bytes, beside, &tot_job, tot_with_terms ? 1 : 0, clear_out, st);
    const EpilogueTail with_sums{nullptr, 0, nullptr, nullptr, nullptr, 0, &w_sums, &tot_job, tot_with_terms ? 1 : 0, beside};
    if (s.conv)
        rc = conv_s8_impl(QBP_CONV_FPROP, &L->conv, saved->x_codes, saved->qx, saved->w_codes, saved->qw, nullptr, saved->z,
                          in_sums, parts.sum ? &parts : nullptr, status, l.scratch, l.scratch_bytes, st, &with_sums);
    else
        rc = gemm_s8_impl(0, 0, s.rows, s.cout, s.cin, saved->x_codes, saved->qx, saved->w_codes, saved->qw, nullptr,
                          saved->z, nullptr, status, l.scratch, l.scratch_bytes, st, &x_sums, &w_sums, beside);
    if (rc) return rc;
    // the convolution's epilogue has left the statistics of z: no pass over z for them
    if (parts.sum)
        return rangebn_fwd_from_parts(saved->z, s.rows, s.cout, gamma, beta, L->relu, y, saved->save_mean, saved->save_min,
                                      saved->save_max, parts, nullptr, out, st, clear_out);
    return qbp_rangebn_fwd_q8(saved->z, s.rows, s.cout, gamma, beta, L->relu, y, saved->save_mean, saved->save_min,
                              saved->save_max, nullptr, out, l.scratch, l.scratch_bytes, stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_layer_bwd(const qbp_layer_desc *L, const qbp_layer_ctx *saved,
                                                                   const float *dy, const float *gamma,
                                                                   const float *beta, float *dx, float *dw,
                                                                   float *dgamma, float *dbeta, void *ws,
                                                                   size_t ws_bytes, void *stream)
{
    LayerShape s;
    int rc = layer_shape(L, s);
    if (rc) return rc;
    if (!saved || !dy || !dx || !dw) return fail(QBP_ERR_INVALID_ARG, "layer_bwd: NULL argument");
    if (!saved->g8 || !saved->qg8 || !saved->g_hi || !saved->g_lo || !saved->qg16 || !saved->z)
        return fail(QBP_ERR_INVALID_ARG, "layer_bwd: the saved-state record has a NULL buffer (the backward pass needs z and the gradient buffers)");
    // (the forward's codes are summed up beside the first pass, and its statistics are read there)
    if (!saved->x_codes || !saved->qx || !saved->w_codes || !saved->qw || !saved->save_mean || !saved->save_min || !saved->save_max)
        return fail(QBP_ERR_INVALID_ARG, "layer_bwd: the saved-state record has a NULL buffer (codes, parameters or statistics of the forward)");
    float *g = saved->g;
    int8_t *g8 = saved->g8, *ghi = saved->g_hi;
    uint8_t *glo = saved->g_lo;
    qbp_qparams *qp8 = saved->qg8, *qp16 = saved->qg16;
    const LayerWs l = layer_ws(L, s, ws, saved->x_codes, ghi, glo);
    if (!ws || ws_bytes < l.bytes)
        return fail(QBP_ERR_WORKSPACE, "layer_bwd: workspace of %zu bytes needed, %zu given", l.bytes, ws_bytes);

    cudaStream_t st = (cudaStream_t)stream;
    int *status = l.status;                        // the forward call cleared it; the backward only ever raises it
    // two copies of the gradient: 8 bits for the layer gradient, 16 bits for the weight gradient
    // (convolution with the input's per-channel code totals at hand: the bifurcation leaves the gradient's, and the
    // weight gradient reads only the edges of the images again for its zero-point terms)
    // ... and when the weight-gradient product has a spare chunk of MMA rows, it takes the gradient's totals itself
    const bool self_totals = s.conv && saved->x_chan_sums && wgrad_self_totals(&L->conv) && s.rows < (1ll << 22);
    const bool totals = s.conv && saved->x_chan_sums && (self_totals || quantizer_totals_supported(s.cout)) && s.rows < (1ll << 22);
    // Range BN backward and the two copies of its result.  Where the shape allows, in two passes over (dy, z): the
    // statistics pass also takes the extremes of dy, from which the exact range of the gradient follows (Section 4:
    // the range without a scan), and the second pass quantises the gradient as it computes it -- the fp32 gradient is
    // written only when the caller keeps saved->g.  Else: the pass that writes the gradient leaves its range, and the
    // bifurcation reads the gradient back.
    const bool two_pass = rangebn_bwd_bifurcate_supported(dy, saved->z, g, s.rows, s.cout);
    // A linear layer's second pass leaves the gradient's row sums and column totals: no launch for them before the products
    // (64 x 256 -> 128: 37.6 -> 35.7 us a step, 1024 x 2048 -> 1008 77.6 -> 75.5, 4096 x 1024 -> 48 70.2 -> 63.8).
    const bool lin_totals = !s.conv && two_pass && !l.wg_table;
    int64_t *tot_g = totals || lin_totals ? l.tot_g : nullptr;
    const int64_t clear_words = lin_totals ? 2 * s.cout : l.clear_words;
    // the code sums that the two products need: of the weights and the input beside the statistics of the Range BN backward ...
    SumJob early[kMaxSumJobs], late[kMaxSumJobs];
    int nearly = 0, nlate = 0;
    const SumJob w_job = weight_sum_job(L, s, true, saved->w_codes, l.w_sums);
    early[nearly++] = w_job;
    const bool x_early = !s.conv || !rangebn_bwd_one_launch(s.rows, s.cout);      // (a convolution's are added to what is cleared there)
    for (int i = totals ? 3 : 0; i < l.wg_count; ++i) {
        if (lin_totals && i) continue;
        if (i % 3 == 0 && x_early) early[nearly++] = l.wg_sums[i];
        else            late[nlate++] = l.wg_sums[i];          // ... of the gradient's copies once they are there
    }
    if (!s.conv && !lin_totals) late[nlate++] = SumJob{g8, s.rows, s.cout, kSumRows, 1, l.row_sums};
    if (two_pass) {
        rc = rangebn_bwd_bifurcate_impl(dy, saved->z, s.rows, s.cout, gamma, beta, L->relu, saved->save_mean, saved->save_min,
                                        saved->save_max, g, dgamma, dbeta, L->seed, L->tensor_id8, L->tensor_id16, g8, qp8,
                                        s.conv || lin_totals ? l.row_sums : nullptr, ghi, glo, qp16, true, l.scratch, l.scratch_bytes, st,
                                        self_totals ? nullptr : tot_g, l.tot_g, clear_words, early, nearly);
    } else {
        if (!g) return fail(QBP_ERR_INVALID_ARG, "layer_bwd: this shape needs saved->g (the fp32 gradient is written and read back)");
        if ((rc = launch_clear(l.tot_g, l.clear_words, st))) return rc;
        int nparts = 0;
        rc = rangebn_bwd_impl(dy, saved->z, s.rows, s.cout, gamma, beta, L->relu, saved->save_mean, saved->save_min,
                              saved->save_max, g, dgamma, dbeta, l.scratch, l.scratch_bytes, l.range_parts, &nparts, st);
        if (rc) return rc;
        rc = bifurcate_with_range_partials(g, s.rows, s.cout, L->seed, L->tensor_id8, L->tensor_id16, g8, qp8,
                                           s.conv ? l.row_sums : nullptr, ghi, glo, qp16, l.range_parts, nparts, st,
                                           self_totals ? nullptr : tot_g, true);
        if (!rc) rc = launch_code_sums(early, nearly, st);
    }
    if (rc) return rc;
    // (a 3 x 3 convolution: in the launch of the layer gradient's correction terms)
    const bool with_terms = s.conv && L->conv.R == 3;
    bool beside = false;
    if (!with_terms && nlate && (rc = launch_code_sums(late, nlate, st, ZeroJobs{}, &beside))) return rc;
    const CodeSums w_sums = sums_of(w_job), g_sums = sums_of(l.row_sums);
    if (s.conv) {
        const EpilogueTail with_sums{nullptr, 0, nullptr, nullptr, nullptr, 0, &w_sums, late, with_terms ? nlate : 0, beside};
        rc = conv_s8_impl(QBP_CONV_DGRAD, &L->conv, g8, qp8, saved->w_codes, saved->qw, nullptr, dx, l.row_sums, nullptr, status,
                          l.scratch, l.scratch_bytes, st, &with_sums);
        if (rc) return rc;
        return wgrad_s16_impl(&L->conv, 0, 0, 0, saved->x_codes, saved->qx, ghi, glo, qp16, nullptr, dw, status, l.scratch, l.scratch_bytes,
                              st, totals ? saved->x_chan_sums : nullptr, tot_g, !self_totals, true, l.wg_sums);
    }
    // dx [batch x in] = g8 [batch x out] . w^T, w stored [in x out]
    rc = gemm_s8_impl(0, 1, s.rows, s.cin, s.cout, g8, qp8, saved->w_codes, saved->qw, nullptr, dx, nullptr, status, l.scratch,
                      l.scratch_bytes, st, &g_sums, &w_sums, beside);
    if (rc) return rc;
    return wgrad_s16_impl(nullptr, s.rows, s.cout, s.cin, saved->x_codes, saved->qx, ghi, glo, qp16, nullptr, dw, status, l.scratch,
                          l.scratch_bytes, st, nullptr, tot_g, true, true, l.wg_sums);
}
