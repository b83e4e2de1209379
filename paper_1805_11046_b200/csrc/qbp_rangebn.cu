// Range Batch-Normalization (Section 3, Eq. (range)) forward and backward
// (Section 7: derivative of max/min is one where attained).
//
// Both directions are two streaming passes over [n x C] fp32 with the channel
// innermost: a statistics pass (per-channel min, max, sum -- or sum dy,
// sum dy*xhat) and an apply pass, with a one-warp-per-channel combine between
// them.  Sums are carried in fp64 per thread (the fp64 pipe is far from being
// the limit at HBM rate); everything an element's value depends on follows a
// fixed fp32 operation order so that forward and backward agree on which
// outputs the ReLU kept.
#include "qbp_colscan.cuh"
#include "qbp_mma.cuh"
#include "qbp_sums.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace qbp {

// The second pass of either direction walks the rows from the last to the first and finds in the L2 what the statistics pass read
// last: its rows from keep_from on (kKeepBytes of what the second pass reads), with loads that leave the lines there; the rest passes
// through, evict-first, and so does all that the second passes read for the last time and write.  A forward's second pass leaves
// the head of x for the backward of the same call site in the same way (keep_head).  Forward + backward, with the forward's pass
// from the front and all of its loads evict-first, the backward's from the front with ordinary loads and stores, and so, on the same
// buffers again and again: 50176 x 256 86.5 -> 72.4 us, 802816 x 64 272.5 -> 261.5, 12544 x 2048 151.6 -> 139.0; alone on inputs that
// another kernel has just written 84.0 -> 73.8, 272.4 -> 264.2, 151.6 -> 141.3, on ones out of HBM 94.2 -> 77.8, 280.6 -> 268.3, 157.7 ->
// 145.4.  48, 88 or 104 MB: within 0.5 us.
constexpr int64_t kKeepBytes = 64ll << 20;
static int64_t keep_from_row(int64_t rows, int64_t row_bytes) { return std::max<int64_t>(0, rows - kKeepBytes / row_bytes); }

// ---------------------------------------------------------------- forward
template <int VEC>
__global__ void __launch_bounds__(kScanThreads) bn_stats_kernel(const float *__restrict__ x, int64_t rows, int C, int tw,
                                                                float *__restrict__ part_lo, float *__restrict__ part_hi,
                                                                double *__restrict__ part_sum, int64_t keep_from)
{
    pdl_wait();
    const ScanPos p = scan_pos<VEC>(C, tw);
    const int rpb = kScanThreads / tw;
    float lo[VEC], hi[VEC];
    double sum[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) { lo[e] = INFINITY; hi[e] = -INFINITY; sum[e] = 0.0; }
    if (p.active) {
        const int64_t step = (int64_t)gridDim.x * rpb;
        for (int64_t r0 = (int64_t)blockIdx.x * rpb + p.ty; r0 < rows; r0 += step * kScanUnroll) {
            VecF<VEC> v[kScanUnroll];
            bool ok[kScanUnroll];
#pragma unroll
            for (int u = 0; u < kScanUnroll; ++u) {
                int64_t r = r0 + u * step;
                ok[u] = r < rows;
                if (ok[u]) { if (r0 < keep_from) v[u].load_stream(x + r * C + p.col); else v[u].load(x + r * C + p.col); }
            }
#pragma unroll
            for (int u = 0; u < kScanUnroll; ++u)
                if (ok[u]) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        lo[e] = fminf(lo[e], v[u].v[e]);
                        hi[e] = fmaxf(hi[e], v[u].v[e]);
                        sum[e] += (double)v[u].v[e];
                    }
                }
        }
    }
    __shared__ float s_lo[kScanThreads * VEC], s_hi[kScanThreads * VEC];
    __shared__ double s_sum[kScanThreads * VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        s_lo[threadIdx.x * VEC + e] = lo[e]; s_hi[threadIdx.x * VEC + e] = hi[e]; s_sum[threadIdx.x * VEC + e] = sum[e];
    }
    __syncthreads();
    if (p.ty == 0 && p.active) {
        for (int y = 1; y < rpb; ++y)
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const int i = (y * tw + p.tx) * VEC + e;
                lo[e] = fminf(lo[e], s_lo[i]); hi[e] = fmaxf(hi[e], s_hi[i]); sum[e] += s_sum[i];
            }
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            const int64_t i = (int64_t)blockIdx.x * C + p.col + e;
            part_lo[i] = lo[e]; part_hi[i] = hi[e]; part_sum[i] = sum[e];
        }
    }
}

// One block of 128 threads per channel: mean (or, with sum_out, the raw fp64 sum for a later combination over
// several GPUs), min, max.
__global__ void __launch_bounds__(128) bn_stats_finalize_kernel(const float *__restrict__ part_lo,
                                                                const float *__restrict__ part_hi,
                                                                const double *__restrict__ part_sum, int nparts, int C,
                                                                int64_t n, float *__restrict__ mean,
                                                                float *__restrict__ vmin, float *__restrict__ vmax,
                                                                double *__restrict__ sum_out)
{
    pdl_wait();
    const int c = blockIdx.x;
    float lo = INFINITY, hi = -INFINITY;
    double sum = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 128) {
        lo = fminf(lo, part_lo[(int64_t)i * C + c]);
        hi = fmaxf(hi, part_hi[(int64_t)i * C + c]);
        sum += part_sum[(int64_t)i * C + c];
    }
    lo = warp_min(lo); hi = warp_max(hi);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    __shared__ float s_lo[4], s_hi[4];
    __shared__ double s_sum[4];
    if ((threadIdx.x & 31) == 0) { s_lo[threadIdx.x >> 5] = lo; s_hi[threadIdx.x >> 5] = hi; s_sum[threadIdx.x >> 5] = sum; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 4; ++w) { lo = fminf(lo, s_lo[w]); hi = fmaxf(hi, s_hi[w]); sum += s_sum[w]; }
        if (mean) mean[c] = (float)(sum / (double)n);
        if (sum_out) sum_out[c] = sum;
        vmin[c] = lo; vmax[c] = hi;
    }
}

// Mean from a (possibly all-reduced) per-channel sum over n rows; min and max are copied alongside.
__global__ void bn_mean_from_sum_kernel(const double *__restrict__ col_sum, const float *__restrict__ col_min,
                                        const float *__restrict__ col_max, int C, int64_t n, float *__restrict__ mean,
                                        float *__restrict__ vmin, float *__restrict__ vmax)
{
    pdl_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    mean[c] = (float)(col_sum[c] / (double)n);
    vmin[c] = col_min[c]; vmax[c] = col_max[c];
}

// Requantisation of the output for the next layer (Section 4: the range of an activation that a Range BN produced
// is known from its statistics, so quantising it costs no scan): with rq, the 8-bit codes of y (nearest rounding,
// parameters *rq) are written beside y, or instead of it (y == NULL); rowsum (nullable; rs_group = lanes per row,
// a power of two <= 32 that covers the row) receives each row's sum of stored codes, which the next product's
// zero-point correction needs.
// chansum (nullable, [C], added to with 64-bit atomics): per-channel totals of the stored codes over all rows.
// own_range: every block works the range of y out itself (C channels: a microsecond or so; a launch for it takes more), and the
// first one writes *rq.
struct BnRequant { qbp_qparams *rq; int8_t *q; int32_t *rowsum; int rs_group; unsigned long long *chansum; int own_range; };
constexpr int kBnOwnRangeMax = 1024;       // channels up to which it is worth it

// The exact range of y over the channels a thread is given, from the per-channel statistics: y is a monotone function of x in
// each channel, computed with the same rounded operations, so its extremes sit at x = min and x = max.
__device__ __forceinline__ float2 bn_out_extremes(const float *mean, const float *vmin, const float *vmax, const float *gamma,
                                                  const float *beta, int C, float Cn, bool relu, int first, int step, float4 *fold)
{
    float lo = INFINITY, hi = -INFINITY;
    for (int c = first; c < C; c += step) {
        const float s = bn_scale(vmin[c], vmax[c], Cn);
        const float g = gamma ? gamma[c] : 1.0f, b = beta ? beta[c] : 0.0f;
        if (fold) fold[c] = make_float4(mean[c], s, g, b);      // what a product's epilogue needs to normalise a column
        float a = bn_y(bn_xhat(vmin[c], mean[c], s), g, b);
        float z = bn_y(bn_xhat(vmax[c], mean[c], s), g, b);
        if (relu) { a = fmaxf(a, 0.0f); z = fmaxf(z, 0.0f); }
        lo = fminf(lo, fminf(a, z)); hi = fmaxf(hi, fmaxf(a, z));
    }
    return make_float2(lo, hi);
}

template <int VEC, bool RELU, bool REQUANT>
__global__ void __launch_bounds__(kScanThreads) bn_apply_kernel(const float *__restrict__ x, int64_t rows, int C, int tw,
                                                                const float *__restrict__ mean,
                                                                const float *__restrict__ vmin,
                                                                const float *__restrict__ vmax,
                                                                const float *__restrict__ gamma,
                                                                const float *__restrict__ beta, float Cn,
                                                                float *__restrict__ y, BnRequant R, int reverse, int64_t keep_head)
{
    pdl_wait();
    const ScanPos p = scan_pos<VEC>(C, tw);
    float inv = 0.0f, zp_u = 0.0f;
    if (REQUANT) {
        qbp_qparams qp;
        if (R.own_range) {
            const float2 t = bn_out_extremes(mean, vmin, vmax, gamma, beta, C, Cn, RELU, (int)threadIdx.x, kScanThreads, nullptr);
            const float2 r = block_min_max(t.x, t.y);
            qp = make_qparams(r.x, r.y, 8);
            if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *R.rq = qp;
        } else qp = *R.rq;
        const QParamsReg t = qparams_reg(qp, 8);
        inv = t.inv; zp_u = t.zp_u;
    }
    // (with row sums the idle threads of a ragged last slab take part in the shuffles: tw <= 32 then, one slab)
    if (!p.active && !(REQUANT && (R.rowsum || R.chansum))) return;
    const int rpb = kScanThreads / tw;
    float mu[VEC], s[VEC], g[VEC], b[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        const int c = p.active ? p.col + e : 0;
        mu[e] = mean[c];
        s[e] = bn_scale(vmin[c], vmax[c], Cn);
        g[e] = gamma ? gamma[c] : 1.0f;
        b[e] = beta ? beta[c] : 0.0f;
    }
    int cs[VEC];                                            // totals of the stored codes of this thread's channels
#pragma unroll
    for (int e = 0; e < VEC; ++e) cs[e] = 0;
    const int64_t step = (int64_t)gridDim.x * rpb;
    // (the loop bound is the same for every thread of the block, so that the shuffles below see whole warps)
    for (int64_t rb = (int64_t)blockIdx.x * rpb; rb < rows; rb += step * kScanUnroll) {
        const int64_t r0 = rb + p.ty;
        VecF<VEC> v[kScanUnroll];
        bool ok[kScanUnroll];
#pragma unroll
        for (int u = 0; u < kScanUnroll; ++u) {
            int64_t r = r0 + u * step;
            ok[u] = p.active && r < rows;
            // (reverse: rows from the last to the first, when the kernel that wrote or read x just before has left the tail of x
            // in the L2; of those, the first keep_head rows stay)
            const float *const at = x + (reverse ? rows - 1 - r : r) * C + p.col;
            if (ok[u]) { if (rows - rb <= keep_head) v[u].load(at); else v[u].load_stream(at); }
        }
#pragma unroll
        for (int u = 0; u < kScanUnroll; ++u) {
            int rs = 0;
            if (ok[u]) {
                uint32_t code[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    float yv = bn_y(bn_xhat(v[u].v[e], mu[e], s[e]), g[e], b[e]);
                    v[u].v[e] = RELU ? fmaxf(yv, 0.0f) : yv;
                    if (REQUANT) code[e] = (uint32_t)quantize_code<false>(v[u].v[e], inv, zp_u, 255.0f, 0u);
                }
                const int64_t at = (reverse ? rows - 1 - (r0 + u * step) : r0 + u * step) * C + p.col;
                if (y) v[u].store_stream(y + at);
                if (REQUANT) {
                    if (VEC == 4) {
                        const uint32_t packed = (code[0] | (code[1] << 8) | (code[2] << 16) | (code[3] << 24)) ^ 0x80808080u;
                        *reinterpret_cast<uint32_t *>(R.q + at) = packed;
                        rs = __dp4a((int)packed, 0x01010101, 0);
                        if (R.chansum) {
#pragma unroll
                            for (int e = 0; e < VEC; ++e) cs[e] = __dp4a((int)packed, 1 << (8 * (e & 3)), cs[e]);
                        }
                    } else {
                        R.q[at] = (int8_t)((int)code[0] - 128);
                        rs = (int)code[0] - 128;
                        cs[0] += rs;
                    }
                }
            }
            if (REQUANT && R.rowsum) {
                // a row is rs_group consecutive lanes of one warp (idle lanes add nothing)
                for (int off = 16; off > 0; off >>= 1)
                    if (off < R.rs_group) rs += __shfl_xor_sync(0xffffffffu, rs, off);
                const int64_t r = r0 + u * step;
                if (p.tx == 0 && r < rows) R.rowsum[reverse ? rows - 1 - r : r] = rs;
            }
        }
    }
    if (REQUANT && R.chansum) {
        // the block's threads meet in shared memory (fewer than 2^22 rows: int32 is enough), then one atomic per channel
        __shared__ int s_tot[kScanMaxTw * 4];
        for (int i = threadIdx.x; i < tw * VEC; i += kScanThreads) s_tot[i] = 0;
        __syncthreads();
        if (p.active) {
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                if (cs[e]) atomicAdd(&s_tot[p.tx * VEC + e], cs[e]);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < tw * VEC; i += kScanThreads) {
            const int c = (int)blockIdx.y * tw * VEC + i;
            if (c < C && s_tot[i]) atomicAdd(R.chansum + c, (unsigned long long)(long long)s_tot[i]);
        }
    }
}

// The same in a launch of its own.
__global__ void __launch_bounds__(256) bn_out_range_kernel(const float *__restrict__ mean, const float *__restrict__ vmin,
                                                           const float *__restrict__ vmax,
                                                           const float *__restrict__ gamma,
                                                           const float *__restrict__ beta, int C, float Cn, int relu,
                                                           qbp_qparams *__restrict__ out, qbp_qparams *__restrict__ qp8_out,
                                                           float4 *__restrict__ fold)
{
    pdl_wait();
    const float2 t = bn_out_extremes(mean, vmin, vmax, gamma, beta, C, Cn, relu != 0, (int)threadIdx.x, 256, fold);
    const float2 r = block_min_max(t.x, t.y);
    if (threadIdx.x == 0) {
        if (out) { out->scale = 0.0f; out->zero_point = 0; out->vmin = r.x; out->vmax = r.y; }
        if (qp8_out) *qp8_out = make_qparams(r.x, r.y, 8);
    }
}

// --------------------------------------------------------------- backward
// EXT: also the extremes of the (rectifier-masked) dy of each channel over three sets of positions -- where x is the
// channel's maximum, where it is its minimum, and everywhere else -- as ext [6][blocks][C] (min, max of the ordinary
// positions, then of the maxima, then of the minima).  dx is a monotone function of dy on each set (bn_dx), so the
// finalize kernel knows the exact range of dx from these, before dx is computed.
// The last kKeepBytes of both tensors stay in the L2 for the second pass (see above) where that is bound by HBM: the plain one, and
// the bifurcating one that also writes the gradient (25.7 M elements 74 -> 68 us).  The bifurcating pass alone is bound by arithmetic
// and gains nothing (the layers of 56 x 56 x 64 and 14 x 14 x 256 lose a microsecond).
template <int VEC, bool RELU, bool EXT>
__global__ void __launch_bounds__(kScanThreads) bn_bwd_stats_kernel(const float *__restrict__ dy,
                                                                    const float *__restrict__ x, int64_t rows, int C,
                                                                    int tw, const float *__restrict__ mean,
                                                                    const float *__restrict__ vmin,
                                                                    const float *__restrict__ vmax,
                                                                    const float *__restrict__ gamma,
                                                                    const float *__restrict__ beta, float Cn,
                                                                    double *__restrict__ part_dy,
                                                                    double *__restrict__ part_dyx,
                                                                    float *__restrict__ ext, const ZeroJobs zero, int64_t keep_from)
{
    pdl_wait();
    if (EXT)
        run_zero_jobs(zero, ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kScanThreads + threadIdx.x,
                      (int64_t)gridDim.x * gridDim.y * kScanThreads);
    const ScanPos p = scan_pos<VEC>(C, tw);
    const int rpb = kScanThreads / tw;
    double sdy[VEC], sdyx[VEC];
    // (the extremes of the ordinary positions in registers; those of the few positions at a channel's maximum or
    // minimum in shared memory, as integers that order like the floats)
    float elo[VEC], ehi[VEC];
    __shared__ int s_tie[EXT ? 4 * kScanThreads * VEC / 4 : 1];      // [min at max, max at max, min at min, max at min][tw * VEC]
#pragma unroll
    for (int e = 0; e < VEC; ++e) { sdy[e] = 0.0; sdyx[e] = 0.0; elo[e] = INFINITY; ehi[e] = -INFINITY; }
    if (EXT) {
        for (int i = threadIdx.x; i < 4 * tw * VEC; i += kScanThreads) s_tie[i] = ((i / (tw * VEC)) & 1) ? float_order(-INFINITY) : float_order(INFINITY);
        __syncthreads();
    }
    if (p.active) {
        float mu[VEC], s[VEC], g[VEC], b[VEC], lo[VEC], hi[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            mu[e] = mean[p.col + e];
            lo[e] = vmin[p.col + e]; hi[e] = vmax[p.col + e];
            s[e] = bn_scale(lo[e], hi[e], Cn);
            g[e] = gamma ? gamma[p.col + e] : 1.0f;
            b[e] = beta ? beta[p.col + e] : 0.0f;
        }
        const int64_t step = (int64_t)gridDim.x * rpb;
        auto pass = [&](auto stream, int64_t &r0, int64_t end) {       // (stream: evict-first loads)
        for (; r0 < end; r0 += step * kScanUnroll) {
            VecF<VEC> vx[kScanUnroll], vd[kScanUnroll];
            bool ok[kScanUnroll];
#pragma unroll
            for (int u = 0; u < kScanUnroll; ++u) {
                int64_t r = r0 + u * step;
                ok[u] = r < rows;
                if (ok[u]) {
                    if (decltype(stream)::value) { vx[u].load_stream(x + r * C + p.col); vd[u].load_stream(dy + r * C + p.col); }
                    else                         { vx[u].load(x + r * C + p.col); vd[u].load(dy + r * C + p.col); }
                }
            }
            // (the few rows of one step are added in fp32, the steps in fp64: a quarter of the conversions and fp64
            // additions, and an error of a few ulp of four terms)
            float fs[VEC], fp[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) { fs[e] = 0.0f; fp[e] = 0.0f; }
#pragma unroll
            for (int u = 0; u < kScanUnroll; ++u)
                if (ok[u]) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        float xh = bn_xhat(vx[u].v[e], mu[e], s[e]);
                        float d = vd[u].v[e];
                        if (RELU && !(bn_y(xh, g[e], b[e]) > 0.0f)) d = 0.0f;
                        fs[e] += d;
                        fp[e] = fmaf(d, xh, fp[e]);
                        if (EXT) {
                            const bool ih = vx[u].v[e] == hi[e], il = vx[u].v[e] == lo[e];
                            if (ih == il) { elo[e] = fminf(elo[e], d); ehi[e] = fmaxf(ehi[e], d); }
                            else {
                                int *t = s_tie + (ih ? 0 : 2) * tw * VEC + p.tx * VEC + e;
                                atomicMin(t, float_order(d)); atomicMax(t + tw * VEC, float_order(d));
                            }
                        }
                    }
                }
#pragma unroll
            for (int e = 0; e < VEC; ++e) { sdy[e] += (double)fs[e]; sdyx[e] += (double)fp[e]; }
        }
        };
        int64_t r0 = (int64_t)blockIdx.x * rpb + p.ty;
        pass(std::true_type{}, r0, keep_from);
        pass(std::false_type{}, r0, rows);
    }
    __shared__ double s_ab[2 * kScanThreads * VEC];
    double *s_a = s_ab, *s_b = s_ab + kScanThreads * VEC;
#pragma unroll
    for (int e = 0; e < VEC; ++e) { s_a[threadIdx.x * VEC + e] = sdy[e]; s_b[threadIdx.x * VEC + e] = sdyx[e]; }
    __syncthreads();
    if (p.ty == 0 && p.active) {
        for (int y = 1; y < rpb; ++y)
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                sdy[e] += s_a[(y * tw + p.tx) * VEC + e];
                sdyx[e] += s_b[(y * tw + p.tx) * VEC + e];
            }
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            part_dy[(int64_t)blockIdx.x * C + p.col + e] = sdy[e];
            part_dyx[(int64_t)blockIdx.x * C + p.col + e] = sdyx[e];
        }
    }
    if (EXT) {
        // the block's rows meet in shared memory (the arrays of the sums, read by now, hold two tables each)
        float *s_f = reinterpret_cast<float *>(s_ab);          // room for four tables of kScanThreads * VEC floats
        static_assert(sizeof(double) == 2 * sizeof(float), "two float tables per double table");
        __syncthreads();
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            s_f[threadIdx.x * VEC + e] = elo[e];
            s_f[(kScanThreads + threadIdx.x) * VEC + e] = ehi[e];
        }
        __syncthreads();
        if (p.ty == 0 && p.active) {
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                float lo0 = elo[e], hi0 = ehi[e];
                for (int y = 1; y < rpb; ++y) {
                    lo0 = fminf(lo0, s_f[(y * tw + p.tx) * VEC + e]);
                    hi0 = fmaxf(hi0, s_f[(kScanThreads + y * tw + p.tx) * VEC + e]);
                }
                const int64_t at = (int64_t)blockIdx.x * C + p.col + e, tbl = (int64_t)gridDim.x * C;
                ext[at] = lo0; ext[tbl + at] = hi0;
#pragma unroll
                for (int k = 0; k < 4; ++k) ext[(2 + k) * tbl + at] = order_float(s_tie[k * tw * VEC + p.tx * VEC + e]);
            }
        }
    }
}

// What the backward's second pass needs of a channel, from its complete sums: dbeta = sum dy, dgamma = sum dy*xhat,
// m1 = gamma*dbeta/n, k2 = C(n)*gamma*dgamma; with the extremes ev of dy over the three sets of positions (see
// bn_bwd_stats_kernel) also the exact range of the channel's dx and the rectifier's mask as a threshold on x.
struct BnBwdOut { float *dgamma, *dbeta; float2 *coef, *chan_range, *relu_thr; };
__device__ __forceinline__ void bn_bwd_channel(int c, double sdy, double sdyx, int64_t n, double Cn, float g, float b, float mu, float lo,
                                               float hi, float Cn_f, const float *ev, const BnBwdOut &o)
{
    if (o.dbeta) o.dbeta[c] = (float)sdy;
    if (o.dgamma) o.dgamma[c] = (float)sdyx;
    const float m1 = (float)((double)g * sdy / (double)n), k2 = (float)(Cn * (double)g * sdyx);
    o.coef[c] = make_float2(m1, k2);
    if (!ev) return;
    const float s = bn_scale(lo, hi, Cn_f);
    float rlo = INFINITY, rhi = -INFINITY;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (!(ev[2 * k] <= ev[2 * k + 1])) continue;           // (a set with no position keeps +inf, -inf)
        const float t = k == 0 ? 0.0f : k == 1 ? k2 : -k2;
        const float v0 = bn_dx(ev[2 * k], t, s, g, m1), v1 = bn_dx(ev[2 * k + 1], t, s, g, m1);
        rlo = fminf(rlo, fminf(v0, v1)); rhi = fmaxf(rhi, fmaxf(v0, v1));
    }
    o.chan_range[c] = make_float2(rlo, rhi);
    if (o.relu_thr) o.relu_thr[c] = relu_threshold(mu, s, g, b);
}

// One block of T threads per channel: kSumThreads, or, when there are no code sums to take, as few as have every partial in flight
// at once, two per thread (statistics and this of 25.7 M elements in 2048 channels of 37 partials 44.3 -> 38.6 us with 64, of 6.4 M
// in 512 channels of 148 17.0 -> 15.3 with 128; 128 channels of 296 37.3 with 128, 36.6 with 256): dbeta, dgamma, and the two per-channel
// constants of dx: m1 = gamma*dbeta/n, k2 = C(n)*gamma*dgamma.
template <int T>
__global__ void __launch_bounds__(T) bn_bwd_finalize_kernel(const double *__restrict__ part_dy,
                                                              const double *__restrict__ part_dyx, int nparts, int C,
                                                              int64_t n, const float *__restrict__ gamma, double Cn,
                                                              float *__restrict__ dgamma, float *__restrict__ dbeta,
                                                              float2 *__restrict__ coef, double *__restrict__ sum_dy,
                                                              double *__restrict__ sum_dyx,
                                                              const float *__restrict__ ext = nullptr,
                                                              const float *__restrict__ vmin = nullptr,
                                                              const float *__restrict__ vmax = nullptr, float Cn_f = 0.0f,
                                                              float2 *__restrict__ chan_range = nullptr,
                                                              const float *__restrict__ mean = nullptr,
                                                              const float *__restrict__ beta = nullptr,
                                                              float2 *__restrict__ relu_thr = nullptr,
                                                              const __grid_constant__ SumJobs J = SumJobs{})
{
    pdl_wait();
    const int c = blockIdx.x;
    // (the blocks behind the channels take code sums that a later product needs: C short blocks leave most SMs idle)
    if (T == kSumThreads && c >= C) { code_sums_block(J, c - C); return; }
    double a = 0.0, b = 0.0;
    // ext (see bn_bwd_stats_kernel): the extremes of dy over the three sets of positions, then (below) the exact range
    // of this channel's dx, left in chan_range[c] for the quantiser of the gradient
    float ev[6];
    __shared__ float s_e[6][T / 32];
#pragma unroll
    for (int k = 0; k < 6; ++k) ev[k] = (k & 1) ? -INFINITY : INFINITY;
    // (all loads of two partials at once: the whole table in one round trip for up to two blocks per SM)
    for (int i0 = threadIdx.x; i0 < nparts; i0 += 2 * T) {
        double pa_[2], pb_[2];
        float o[2][6];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = i0 + u * T;
            const bool ok = i < nparts;
            pa_[u] = ok ? part_dy[(int64_t)i * C + c] : 0.0; pb_[u] = ok ? part_dyx[(int64_t)i * C + c] : 0.0;
#pragma unroll
            for (int k = 0; k < 6; ++k) o[u][k] = ok && ext ? ext[((int64_t)k * nparts + i) * C + c] : (k & 1) ? -INFINITY : INFINITY;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            a += pa_[u]; b += pb_[u];
#pragma unroll
            for (int k = 0; k < 6; ++k) ev[k] = (k & 1) ? fmaxf(ev[k], o[u][k]) : fminf(ev[k], o[u][k]);
        }
    }
    if (ext) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            ev[k] = (k & 1) ? warp_max(ev[k]) : warp_min(ev[k]);
            if ((threadIdx.x & 31) == 0) s_e[k][threadIdx.x >> 5] = ev[k];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    __shared__ double s_a[T / 32], s_b[T / 32];
    if ((threadIdx.x & 31) == 0) { s_a[threadIdx.x >> 5] = a; s_b[threadIdx.x >> 5] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < T / 32; ++w) { a += s_a[w]; b += s_b[w]; }
        if (sum_dy) {                       // raw sums only: combined over several GPUs before the coefficients
            sum_dy[c] = a; sum_dyx[c] = b;
            return;
        }
        BnBwdOut o{dgamma, dbeta, coef, chan_range, relu_thr};
        if (ext) {
#pragma unroll
            for (int k = 0; k < 6; ++k)
                for (int w = 1; w < T / 32; ++w) ev[k] = (k & 1) ? fmaxf(ev[k], s_e[k][w]) : fminf(ev[k], s_e[k][w]);
        }
        bn_bwd_channel(c, a, b, n, Cn, gamma ? gamma[c] : 1.0f, beta ? beta[c] : 0.0f, ext ? mean[c] : 0.0f, ext ? vmin[c] : 0.0f,
                       ext ? vmax[c] : 0.0f, Cn_f, ext ? ev : nullptr, o);
    }
}

// The Range BN backward apply pass and the bifurcation of the gradient it computes (Sections 3 and 6) in one pass:
// dx goes from registers into its 8-bit copy (stochastic rounding), the two limbs of its 16-bit copy and each row's
// 8-bit code sum; the fp32 dx itself is written only when the caller keeps it (g_out).  The parameters of both copies
// are known beforehand (from the ranges bn_bwd_finalize_kernel leaves per channel).  Element i of the [rows x C] tensor draws from
// Philox block i / 4 as in quantize_kernel: a thread's four channels are one block.  rowsum8: a row's lanes
// of one warp add up by shuffles; when a row spans several warps or blocks (tw > 32 or several slabs) the pieces are added
// to rowsum8 [rows], zeroed beforehand.
// TOTALS: also each channel's total of the stored 16-bit codes (256 * hi + lo with lo unsigned, whatever lo_flip) over
// all rows, added to chansum16 [C] (zeroed beforehand): a thread keeps its four channels for its whole life, a block
// adds its threads' totals in shared memory and ends with one 64-bit atomic per channel.
// The operands come through a ring in shared memory, filled by each thread's own asynchronous copies one tile ahead of the one
// it computes (a thread reads back only what it copied itself: no barrier), so the memory system always has work.
// What bounds it: the integer pipes (about 25 instructions per element in Philox and the two roundings alone).  So the rest is
// kept small: 32-bit indices, no check per row in the whole tiles, the rare terms of the extremes on a path outside the
// straight line (one branch per tile of four rows, after which all of them are quantised together), the channels' constants
// read from shared memory once per tile.  With tiles of two rows and checks per row (69 instructions per element, now 47) 51.4 M
// elements of 64 channels take 131 us, so 109; 102.8 M of 512 channels 277 and 209 (5.5 TB/s), 12.8 M of 256 channels 43 and 35.  Not better: four blocks of 64 registers (113, spills with four rows), two of 105 (109), a third slot.
constexpr int kBabRows = 4;       // rows per thread and tile (an even number)
constexpr int kBabSlots = 2;      // ring depth in tiles
constexpr int kBabBlocks = 3;     // blocks per SM (at most 80 registers a thread)
constexpr size_t kBabRingBytes = (size_t)kBabSlots * 2 * kBabRows * kScanThreads * sizeof(float4);
static_assert(kBabBlocks * (kBabRingBytes + 8192 + 1024) <= 228 * 1024, "the rings of an SM's blocks, their 7.3 KB of static shared memory beside them");
// ONE: both copies have one tensor id and share their Philox blocks.
template <bool RELU, bool STORE_G, bool TOTALS, bool ONE>
__global__ void __launch_bounds__(kScanThreads, kBabBlocks) bn_bwd_apply_bifurcate_kernel(
    const float4 *__restrict__ dy, const float4 *__restrict__ x, uint32_t rows, int C, int tw, const float *__restrict__ vmin,
    const float *__restrict__ vmax, const float *__restrict__ gamma, float Cn, const float2 *__restrict__ coef,
    float4 *__restrict__ g_out, const RangeSrc range, uint32_t id8, uint32_t id16, const __grid_constant__ PhiloxKeys keys,
    uint32_t *__restrict__ q8, uint32_t *__restrict__ q_hi, uint32_t *__restrict__ q_lo, uint32_t lo_flip,
    int32_t *__restrict__ rowsum8, unsigned long long *__restrict__ chansum16, const float2 *__restrict__ relu_thr)
{
    pdl_wait();
    const ScanPos p = scan_pos<4>(C, tw);
    int cs16[4] = {0, 0, 0, 0};                   // stored codes of this thread's rows (fewer than 65536 rows)
    // the channels' constants in shared memory, read again for every tile: 28 registers that the 80 of a thread have no room for
    __shared__ float4 s_const[7][kScanMaxTw];     // scale, gamma, centre, half of the range, m1, the mask's threshold and sign
    if ((int)threadIdx.x < tw) {
        float k[7][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = p.active ? p.col + e : 0;
            const float2 th = RELU ? relu_thr[c] : make_float2(0.0f, 1.0f);   // (the mask y > 0 as sgn * x >= threshold)
            const float lo = vmin[c], hi = vmax[c];
            k[0][e] = bn_scale(lo, hi, Cn);
            // |x - centre| >= half holds for the extremes (both sides rounded alike) and for hardly anything else
            k[2][e] = 0.5f * lo + 0.5f * hi;
            k[3][e] = fminf(__fsub_rn(hi, k[2][e]), __fsub_rn(k[2][e], lo));
            k[1][e] = gamma ? gamma[c] : 1.0f;
            k[4][e] = coef[c].x; k[5][e] = th.x; k[6][e] = th.y;
        }
#pragma unroll
        for (int i = 0; i < 7; ++i) s_const[i][p.tx] = make_float4(k[i][0], k[i][1], k[i][2], k[i][3]);
    }
    __syncthreads();
    // both codes in fixed point with 16 fraction bits (quantize_sr8_byte2 / quantize_sr16_top_half)
    QParamsReg q8r, q16r;
    resolve_range(range, true, true, blockIdx.x == 0 && blockIdx.y == 0, q8r, q16r);
    const float inv8 = q8r.inv * 65536.0f, zp8 = q8r.zp_u * 65536.0f, inv16 = q16r.inv * 65536.0f, zp16 = q16r.zp_u * 65536.0f;

    // The gradients of a tile's rows without the terms of the maxima and minima; whether one of those may be among them.
    auto dx = [&](const float4 *src, float (&v)[kBabRows][4]) {
        float s[4], g[4], mid[4], half[4], m1[4], thr[4], tsg[4];
        auto get = [&](int i, float (&k)[4]) { const float4 c = s_const[i][p.tx]; k[0] = c.x; k[1] = c.y; k[2] = c.z; k[3] = c.w; };
        get(0, s); get(1, g); get(2, mid); get(3, half); get(4, m1);
        if (RELU) { get(5, thr); get(6, tsg); }
        bool edge = false;
#pragma unroll
        for (int u = 0; u < kBabRows; ++u) {
            const float4 fx = src[2 * u * kScanThreads], fd = src[(2 * u + 1) * kScanThreads];
            const float ax[4] = {fx.x, fx.y, fx.z, fx.w}, ad[4] = {fd.x, fd.y, fd.z, fd.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float d = RELU && !(__fmul_rn(tsg[e], ax[e]) >= thr[e]) ? 0.0f : ad[e];
                v[u][e] = bn_dx(d, 0.0f, s[e], g[e], m1[e]);
                edge |= fabsf(__fsub_rn(ax[e], mid[e])) >= half[e];
            }
        }
        return edge;
    };
    // ... of one float4, with them.
    auto dx_edge = [&](const float4 &fx, const float4 &fd, float (&v)[4]) {
        const float ax[4] = {fx.x, fx.y, fx.z, fx.w}, ad[4] = {fd.x, fd.y, fd.z, fd.w};
        const float *const k = reinterpret_cast<const float *>(&s_const[0][p.tx]);
        constexpr int kRow = 4 * kScanMaxTw;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = p.active ? p.col + e : 0;
            const float d = RELU && !(__fmul_rn(k[6 * kRow + e], ax[e]) >= k[5 * kRow + e]) ? 0.0f : ad[e];
            v[e] = bn_dx(d, bn_k2_ind(ax[e], vmin[c], vmax[c], coef[c].y), k[e], k[kRow + e], k[4 * kRow + e]);
        }
    };
    // The codes and stores of one float4; returns the sum of its 8-bit codes.  store: false for a thread beyond the columns.
    auto codes = [&](const float (&v)[4], uint32_t j, bool store) {
        // the thread's Philox block = its float4's index
        const uint4 r8 = philox4x32_10(make_uint4(j, 0u, id8, 0u), keys);
        const uint4 r16 = ONE ? r8 : philox4x32_10(make_uint4(j, 0u, id16, 0u), keys);
        uint32_t c16[4];
        const BifWords w = bifurcate4(v, inv8, zp8, inv16, zp16, r8, r16, lo_flip, c16);
        if (store) {
            if (STORE_G) __stcs(g_out + j, make_float4(v[0], v[1], v[2], v[3]));
            q8[j] = w.q8; q_hi[j] = w.hi; q_lo[j] = w.lo;
        }
        if (TOTALS) {
#pragma unroll
            for (int e = 0; e < 4; ++e) cs16[e] += (int)c16[e] >> 16;
        }
        return store ? __dp4a((int)w.q8, 0x01010101, 0) : 0;
    };
    // A row's code sum of a step's rows.  Two of them ride in one word: at most 32 lanes of a warp share a row, four codes each,
    // offset by 512 per lane.  Lane 0 of the row stores the first row's sum, lane 1 the second's (a single lane, both); of a row
    // wider than the warp, or than the block, each piece is added to the zeroed sum.
    const int lanes = tw < 32 ? tw : 32, lane = p.tx & (lanes - 1);
    const bool rowsum_pieces = tw > 32 || gridDim.y > 1;
    auto row_sums = [&](int rs0, int rs1, uint32_t r0, uint32_t r1, bool ok0, bool ok1) {
        uint32_t two = (uint32_t)(rs0 + 512) + ((uint32_t)(rs1 + 512) << 16);
        if (lanes == 32) two = __reduce_add_sync(0xffffffffu, two);
        else
#pragma unroll
            for (int off = 8; off > 0; off >>= 1)
                if (off < lanes) two += __shfl_xor_sync(0xffffffffu, two, off);
        if (lane < 2 && (lane ? ok1 : ok0)) {
            const int sum = (int)((lane ? two >> 16 : two & 0xFFFFu)) - 512 * lanes;
            int32_t *const dst = rowsum8 + (lane ? r1 : r0);
            if (rowsum_pieces) atomicAdd(dst, sum); else *dst = sum;
            if (lanes == 1 && ok1) rowsum8[r1] = (int)(two >> 16) - 512;
        }
    };
    // A block takes tiles of kBabRows * rpb rows; rows and float4 indices in 32 bits (fewer than 2^32 of either).
    const uint32_t rpb = kScanThreads / tw, cv = (uint32_t)C >> 2, tile = kBabRows * rpb, jrow = rpb * cv;
    const uint32_t tiles = rows / tile;                        // whole ones; the rows that are left over come last
    const uint32_t mine = blockIdx.x < tiles ? (tiles - blockIdx.x - 1) / gridDim.x + 1 : 0;
    const uint32_t jt = gridDim.x * tile * cv;
    // (from the last tile to the first: the statistics' pass, just before, left the end of both tensors in the L2)
    uint32_t r = (tiles - 1 - blockIdx.x) * tile + p.ty, j = r * cv + (uint32_t)((p.active ? p.col : 0) >> 2);
    extern __shared__ __align__(16) float4 bab_ring[];         // [slot][row][x | dy][thread]
    float4 *const mine_ring = bab_ring + threadIdx.x;
    auto fetch = [&](uint32_t jf, int slot) {
        float4 *const dst = mine_ring + slot * (2 * kBabRows * kScanThreads);
#pragma unroll
        for (int u = 0; u < kBabRows; ++u) {
            cp_async16(dst + (2 * u) * kScanThreads, x + (jf + u * jrow));
            cp_async16(dst + (2 * u + 1) * kScanThreads, dy + (jf + u * jrow));
        }
    };
#pragma unroll
    for (uint32_t k = 0; k < kBabSlots - 1; ++k) {
        if (k < mine) fetch(j - k * jt, (int)k);
        cp_async_commit();                                     // (a group per tile, empty past the end: the count below is uniform)
    }
    int slot = 0;
    for (uint32_t t = 0; t < mine; ++t) {
        // the slot this thread emptied in the step before takes the tile kBabSlots - 1 ahead; then this step's data is in
        if (t + (kBabSlots - 1) < mine) fetch(j - (kBabSlots - 1) * jt, slot == 0 ? kBabSlots - 1 : slot - 1);
        cp_async_commit();
        cp_async_wait<kBabSlots - 1>();
        const float4 *const src = mine_ring + slot * (2 * kBabRows * kScanThreads);
        float v[kBabRows][4];
        if (dx(src, v)) {                                      // (few: two positions per channel, or ties)
#pragma unroll
            for (int u = 0; u < kBabRows; ++u) dx_edge(src[2 * u * kScanThreads], src[(2 * u + 1) * kScanThreads], v[u]);
        }
#pragma unroll
        for (int u = 0; u < kBabRows; u += 2) {
            const int rs0 = codes(v[u], j + u * jrow, p.active), rs1 = codes(v[u + 1], j + (u + 1) * jrow, p.active);
            if (rowsum8) row_sums(rs0, rs1, r + u * rpb, r + (u + 1) * rpb, true, true);
        }
        slot = slot + 1 == kBabSlots ? 0 : slot + 1;
        j -= jt; r -= gridDim.x * tile;
    }
    // the rows left over (fewer than a tile): the last block's
    if (blockIdx.x == gridDim.x - 1 && tiles * tile < rows) {
        const uint32_t rl = tiles * tile + p.ty;
#pragma unroll 1
        for (int u = 0; u < kBabRows; u += 2) {
            int rs[2] = {0, 0};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t ru = rl + (u + h) * rpb;
                if (!(p.active && ru < rows)) continue;
                const uint32_t ju = ru * cv + (uint32_t)(p.col >> 2);
                float v[4];
                dx_edge(x[ju], dy[ju], v);
                rs[h] = codes(v, ju, true);
            }
            if (rowsum8) row_sums(rs[0], rs[1], rl + u * rpb, rl + (u + 1) * rpb, rl + u * rpb < rows, rl + (u + 1) * rpb < rows);
        }
    }
    if (TOTALS) {
        int *const s_tot = reinterpret_cast<int *>(s_const);     // (the constants' room)
        __syncthreads();
        for (int i = threadIdx.x; i < tw * 4; i += kScanThreads) s_tot[i] = 0;
        __syncthreads();
        if (p.active) {
#pragma unroll
            for (int e = 0; e < 4; ++e) atomicAdd(&s_tot[p.tx * 4 + e], cs16[e]);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < tw * 4; i += kScanThreads) {
            const int c = blockIdx.y * tw * 4 + i;
            if (c < C && s_tot[i]) atomicAdd(chansum16 + c, (unsigned long long)(long long)s_tot[i]);
        }
    }
}

// The same coefficients from per-channel sums that are already complete (n: the rows they were taken over).
__global__ void bn_bwd_coef_kernel(const double *__restrict__ sum_dy, const double *__restrict__ sum_dyx, int C, int64_t n,
                                   const float *__restrict__ gamma, double Cn, float *__restrict__ dgamma,
                                   float *__restrict__ dbeta, float2 *__restrict__ coef)
{
    pdl_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const double a = sum_dy[c], b = sum_dyx[c];
    const double g = gamma ? (double)gamma[c] : 1.0;
    if (dbeta) dbeta[c] = (float)a;
    if (dgamma) dgamma[c] = (float)b;
    coef[c] = make_float2((float)(g * a / (double)n), (float)(Cn * g * b));
}

// RANGE: also leave the block's (min, max) of the dx values it wrote in range_parts[block], so that the
// quantiser that follows needs no scan of its own (Section 4: the range comes for free).
// Walks from the last row to the first (see above), but not where channels are read one by one: four stores to a sector that
// leaves the L2 at the first cost more than what is found there (271138 x 179 184 us from the front, 218 from the end).
template <int VEC, bool RELU, bool RANGE>
__global__ void __launch_bounds__(kScanThreads) bn_bwd_apply_kernel(const float *__restrict__ dy,
                                                                    const float *__restrict__ x, int64_t rows, int C,
                                                                    int tw, const float *__restrict__ mean,
                                                                    const float *__restrict__ vmin,
                                                                    const float *__restrict__ vmax,
                                                                    const float *__restrict__ gamma,
                                                                    const float *__restrict__ beta, float Cn,
                                                                    const float2 *__restrict__ coef,
                                                                    float *__restrict__ dx,
                                                                    float2 *__restrict__ range_parts)
{
    pdl_wait();
    const ScanPos p = scan_pos<VEC>(C, tw);
    float rlo = INFINITY, rhi = -INFINITY;
    if (p.active) {
    const int rpb = kScanThreads / tw;
    float mu[VEC], s[VEC], g[VEC], b[VEC], lo[VEC], hi[VEC], m1[VEC], k2[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        mu[e] = mean[p.col + e];
        lo[e] = vmin[p.col + e]; hi[e] = vmax[p.col + e];
        s[e] = bn_scale(lo[e], hi[e], Cn);
        g[e] = gamma ? gamma[p.col + e] : 1.0f;
        b[e] = beta ? beta[p.col + e] : 0.0f;
        float2 cf = coef[p.col + e];
        m1[e] = cf.x; k2[e] = cf.y;
    }
    const int64_t step = (int64_t)gridDim.x * rpb;
    for (int64_t r0 = (int64_t)blockIdx.x * rpb + p.ty; r0 < rows; r0 += step * kScanUnroll) {
        VecF<VEC> vx[kScanUnroll], vd[kScanUnroll];
        bool ok[kScanUnroll];
#pragma unroll
        for (int u = 0; u < kScanUnroll; ++u) {
            int64_t r = r0 + u * step;
            ok[u] = r < rows;
            if (ok[u]) {
                if (VEC == 4) { vx[u].load_stream(x + (rows - 1 - r) * C + p.col); vd[u].load_stream(dy + (rows - 1 - r) * C + p.col); }
                else          { vx[u].load(x + r * C + p.col); vd[u].load(dy + r * C + p.col); }
            }
        }
#pragma unroll
        for (int u = 0; u < kScanUnroll; ++u)
            if (ok[u]) {
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float xv = vx[u].v[e];
                    float d = vd[u].v[e];
                    if (RELU && !(bn_y(bn_xhat(xv, mu[e], s[e]), g[e], b[e]) > 0.0f)) d = 0.0f;
                    vd[u].v[e] = bn_dx(d, bn_k2_ind(xv, lo[e], hi[e], k2[e]), s[e], g[e], m1[e]);
                    if (RANGE) { rlo = fminf(rlo, vd[u].v[e]); rhi = fmaxf(rhi, vd[u].v[e]); }
                }
                if (VEC == 4) vd[u].store_stream(dx + (rows - 1 - (r0 + u * step)) * C + p.col);
                else          vd[u].store(dx + (r0 + u * step) * C + p.col);
            }
    }
    }
    if (RANGE) {
        rlo = warp_min(rlo); rhi = warp_max(rhi);
        __shared__ float s_lo[kScanThreads / 32], s_hi[kScanThreads / 32];
        if ((threadIdx.x & 31) == 0) { s_lo[threadIdx.x >> 5] = rlo; s_hi[threadIdx.x >> 5] = rhi; }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kScanThreads / 32; ++w) { rlo = fminf(rlo, s_lo[w]); rhi = fmaxf(rhi, s_hi[w]); }
            range_parts[blockIdx.y * gridDim.x + blockIdx.x] = make_float2(rlo, rhi);
        }
    }
}

// ------------------------------------------------------------- few rows
// With few rows (a linear layer's minibatch, a late stage's last positions) a block takes CH = 16 channels whole: statistics and
// what follows from them in one launch, where the passes above need a launch for the partials and one to combine them -- 2 to 4 us
// each, which is what such a tensor costs.  Bound by latency: 512 threads, each row's 64 bytes by four of them, four rows in
// flight.  Up to kFewRows rows (16 per thread); beyond, one block per 16 channels walks too long (at 7220 x 160 the
// walk alone would take 17 us, the three launches take 12).  Eight channels (a sector of 32 bytes a row) where a
// block of 16 would give its threads more than one row and the blocks, code sums included, still fit the SMs once: half the walk
// and half the conversions per SM (forward 1024 x 1008 6.5 -> 5.1 us, 2048 x 1024 8.4 -> 6.7; backward 640 x 768 6.6 -> 6.1; with
// code sums beyond the SMs the 1024 x 1008 backward would go from 9.2 to 10.6).
constexpr int kFewThreads = 512, kFewRows = 2048;
template <int CH> constexpr int kFewHigh = kFewThreads / (CH / 4);        // rows taken at a time
static bool few_narrow(int64_t n, int64_t C, int beside) { return n > kFewHigh<16> && (C + 7) / 8 + beside <= sm_count(); }
static bool few_rows(int64_t n, int64_t C) { return n <= kFewRows && C % 4 == 0; }

// Sum (fp64), min and max over a block's rows, per channel: the 128 / CH lanes of a warp that hold the same four channels by
// shuffles (the first two steps halve the channels a lane still carries: four shuffles per quantity instead of twelve), then the warps in
// shared memory, one thread per quantity and channel (all threads adding up all warps took 6 us of a 64 x 64 tensor's backward).
// Every thread can then read its channels' results from the table: sums first, then (min, max) pairs.
template <int CH, int NS, int NM> struct FewTable { double sum[NS][CH]; float lo[NM][CH], hi[NM][CH]; };
template <int CH, int NS, int NM>      // channels; sums; (min, max) pairs
__device__ __forceinline__ const FewTable<CH, NS, NM> &few_reduce(double (&sum)[NS][4], float (&lo)[NM][4], float (&hi)[NM][4])
{
    constexpr int kWarps = kFewThreads / 32, kQuads = CH / 4;
    __shared__ double s_sum[NS][kWarps][CH];
    __shared__ float s_lo[NM][kWarps][CH], s_hi[NM][kWarps][CH];
    __shared__ FewTable<CH, NS, NM> t;
    static_assert((NS + 2 * NM) * CH <= kFewThreads, "a thread per quantity and channel");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool ba = lane & kQuads, bb = lane & (2 * kQuads);
    auto reduce = [&](auto (&v)[4], auto op) {             // of channel 2 * ba + bb over the lanes
        auto r0 = op(ba ? v[2] : v[0], __shfl_xor_sync(0xffffffffu, ba ? v[0] : v[2], kQuads));
        auto r1 = op(ba ? v[3] : v[1], __shfl_xor_sync(0xffffffffu, ba ? v[1] : v[3], kQuads));
        auto q = op(bb ? r1 : r0, __shfl_xor_sync(0xffffffffu, bb ? r0 : r1, 2 * kQuads));
#pragma unroll
        for (int m = 4 * kQuads; m < 32; m *= 2) q = op(q, __shfl_xor_sync(0xffffffffu, q, m));
        return q;
    };
    auto add = [](double a, double b) { return a + b; };
    auto mn = [](float a, float b) { return fminf(a, b); };
    auto mx = [](float a, float b) { return fmaxf(a, b); };
    const int ch = (lane & (kQuads - 1)) * 4 + (ba ? 2 : 0) + (bb ? 1 : 0);
#pragma unroll
    for (int k = 0; k < NS; ++k) { const double r = reduce(sum[k], add); if (lane < CH) s_sum[k][warp][ch] = r; }
#pragma unroll
    for (int k = 0; k < NM; ++k) {
        const float l = reduce(lo[k], mn), h = reduce(hi[k], mx);
        if (lane < CH) { s_lo[k][warp][ch] = l; s_hi[k][warp][ch] = h; }
    }
    __syncthreads();
    const int q = threadIdx.x / CH, c = threadIdx.x % CH;
    if (q < NS) {
        double r = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) r += s_sum[q][w][c];
        t.sum[q][c] = r;
    } else if (q < NS + NM) {
        float r = INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) r = fminf(r, s_lo[q - NS][w][c]);
        t.lo[q - NS][c] = r;
    } else if (q < NS + 2 * NM) {
        float r = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) r = fmaxf(r, s_hi[q - NS - NM][w][c]);
        t.hi[q - NS - NM][c] = r;
    }
    __syncthreads();
    return t;
}

// Forward: the rows wait in registers between the statistics and the normalisation (ROWS per thread, a power of two).
template <int CH, int ROWS>
__global__ void __launch_bounds__(kFewThreads) bn_fwd_few_kernel(const float *__restrict__ x, int rows, int C, const float *__restrict__ gamma,
                                                                 const float *__restrict__ beta, int relu, float Cn, float *__restrict__ y,
                                                                 float *__restrict__ mean, float *__restrict__ vmin, float *__restrict__ vmax)
{
    pdl_wait();
    constexpr int kQuads = CH / 4;
    const int col = (int)blockIdx.x * CH + (threadIdx.x % kQuads) * 4, ty = threadIdx.x / kQuads;
    const bool active = col < C;
    float4 v[ROWS];
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
        const int r = ty + u * kFewHigh<CH>;
        if (active && r < rows) v[u] = __ldg(reinterpret_cast<const float4 *>(x + (int64_t)r * C + col));
    }
    double sum[1][4];
    float lo[1][4], hi[1][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) { sum[0][e] = 0.0; lo[0][e] = INFINITY; hi[0][e] = -INFINITY; }
#pragma unroll
    for (int u = 0; u < ROWS; ++u)
        if (active && ty + u * kFewHigh<CH> < rows) {
            const float t[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { sum[0][e] += (double)t[e]; lo[0][e] = fminf(lo[0][e], t[e]); hi[0][e] = fmaxf(hi[0][e], t[e]); }
        }
    const FewTable<CH, 1, 1> &t1 = few_reduce<CH, 1, 1>(sum, lo, hi);
    if (!active) return;
    const int cl = (threadIdx.x % kQuads) * 4;
    float mu[4], s[4], g[4], b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float lo_e = t1.lo[0][cl + e], hi_e = t1.hi[0][cl + e];
        mu[e] = (float)(t1.sum[0][cl + e] / (double)rows);
        s[e] = bn_scale(lo_e, hi_e, Cn);
        g[e] = gamma ? gamma[col + e] : 1.0f; b[e] = beta ? beta[col + e] : 0.0f;
        if (ty == 0) { mean[col + e] = mu[e]; vmin[col + e] = lo_e; vmax[col + e] = hi_e; }
    }
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
        const int r = ty + u * kFewHigh<CH>;
        if (r >= rows) break;
        float t[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            t[e] = bn_y(bn_xhat(t[e], mu[e], s[e]), g[e], b[e]);
            if (relu) t[e] = fmaxf(t[e], 0.0f);
        }
        *reinterpret_cast<float4 *>(y + (int64_t)r * C + col) = make_float4(t[0], t[1], t[2], t[3]);
    }
}

// Backward: the channel's sums and the extremes of dy, and what bn_bwd_channel makes of them.  (blocks behind the channels: code
// sums that a later product needs; `zero`: cleared on the way)
template <int CH>
__global__ void __launch_bounds__(kFewThreads) bn_bwd_few_kernel(const float *__restrict__ dy, const float *__restrict__ x, int rows, int C,
                                                                 const float *__restrict__ mean, const float *__restrict__ vmin,
                                                                 const float *__restrict__ vmax, const float *__restrict__ gamma,
                                                                 const float *__restrict__ beta, int relu, float Cn, double Cnd,
                                                                 const BnBwdOut out, const ZeroJobs zero, const __grid_constant__ SumJobs J)
{
    pdl_wait();
    const int blocks = (C + CH - 1) / CH;
    if ((int)blockIdx.x >= blocks) {
        if (threadIdx.x < kSumThreads) code_sums_block(J, (int)blockIdx.x - blocks);
        return;
    }
    run_zero_jobs(zero, (int64_t)blockIdx.x * kFewThreads + threadIdx.x, (int64_t)blocks * kFewThreads);
    constexpr int kQuads = CH / 4;
    const int col = (int)blockIdx.x * CH + (threadIdx.x % kQuads) * 4, ty = threadIdx.x / kQuads;
    const bool active = col < C;
    constexpr int U = 4;
    float4 vx[U], vd[U];
    auto fetch = [&](int r0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = r0 + u * kFewHigh<CH>;
            if (r < rows && active) {
                vx[u] = __ldg(reinterpret_cast<const float4 *>(x + (int64_t)r * C + col));
                vd[u] = __ldg(reinterpret_cast<const float4 *>(dy + (int64_t)r * C + col));
            }
        }
    };
    fetch(ty);                            // (on their way while the channels' constants are)
    double sum[2][4];
    float lo[3][4], hi[3][4];             // ordinary positions, those at the channel's maximum, at its minimum
    float mu[4], s[4], g[4], b[4], cl[4], ch[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int c = active ? col + e : 0;
        sum[0][e] = sum[1][e] = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) { lo[k][e] = INFINITY; hi[k][e] = -INFINITY; }
        mu[e] = mean[c]; cl[e] = vmin[c]; ch[e] = vmax[c];
        s[e] = bn_scale(cl[e], ch[e], Cn);
        g[e] = gamma ? gamma[c] : 1.0f; b[e] = beta ? beta[c] : 0.0f;
    }
    for (int r0 = ty; r0 < rows && active; r0 += U * kFewHigh<CH>) {
        if (r0 != ty) fetch(r0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (r0 + u * kFewHigh<CH> >= rows) break;
            const float ax[4] = {vx[u].x, vx[u].y, vx[u].z, vx[u].w}, ad[4] = {vd[u].x, vd[u].y, vd[u].z, vd[u].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float xh = bn_xhat(ax[e], mu[e], s[e]);
                float d = ad[e];
                if (relu && !(bn_y(xh, g[e], b[e]) > 0.0f)) d = 0.0f;
                sum[0][e] += (double)d;
                sum[1][e] += (double)d * (double)xh;
                const bool ih = ax[e] == ch[e], il = ax[e] == cl[e];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (k == 0 ? ih == il : k == 1 ? ih && !il : il && !ih) { lo[k][e] = fminf(lo[k][e], d); hi[k][e] = fmaxf(hi[k][e], d); }
            }
        }
    }
    const FewTable<CH, 2, 3> &t = few_reduce<CH, 2, 3>(sum, lo, hi);
    // one thread per channel
    const int k = threadIdx.x, c = (int)blockIdx.x * CH + k;
    if (k >= CH || c >= C) return;
    const float ev[6] = {t.lo[0][k], t.hi[0][k], t.lo[1][k], t.hi[1][k], t.lo[2][k], t.hi[2][k]};
    bn_bwd_channel(c, t.sum[0][k], t.sum[1][k], rows, Cnd, gamma ? gamma[c] : 1.0f, beta ? beta[c] : 0.0f, mean[c], vmin[c], vmax[c], Cn,
                   out.chan_range ? ev : nullptr, out);
}

static int launch_bwd_few(const float *dy, const float *x, int64_t n, int64_t C, const float *gamma, const float *beta, int relu,
                          const float *mean, const float *vmin, const float *vmax, const BnBwdOut &out, const ZeroJobs &zero,
                          const SumJob *extra, int extra_count, cudaStream_t st)
{
    SumJobs J{};
    int sum_blocks = 0;
    if (extra_count) if (int rc = fill_sum_jobs(extra, extra_count, J, &sum_blocks)) return rc;
    const double Cnd = 1.0 / std::sqrt(2.0 * std::log((double)n));
    QBP_TRACE_BEGIN(st);
#define QBP_BN_FEW(CH_) launch(bn_bwd_few_kernel<CH_>, (int)((C + CH_ - 1) / CH_) + sum_blocks, kFewThreads, 0, st, dy, x, (int)n, (int)C, mean, vmin, \
                               vmax, gamma, beta, relu, (float)Cnd, Cnd, out, zero, J)
    if (few_narrow(n, C, sum_blocks)) QBP_BN_FEW(8); else QBP_BN_FEW(16);
#undef QBP_BN_FEW
    QBP_LAUNCH_OK("bn_bwd_few_kernel");
    return QBP_OK;
}

static size_t bn_ws_bytes(int64_t C)
{
    // forward: lo, hi (float) + sum (double) partials; backward: two double partials + coefficients
    // (... and, for the backward pass that also bifurcates, six float tables of dy extremes and the channels' ranges)
    size_t per = (size_t)kScanMaxStrips * (size_t)C;
    return 2 * align_up(per * sizeof(double), 256) + 2 * align_up(per * sizeof(float), 256) +
           align_up((size_t)C * sizeof(float2), 256) + 256 + align_up(6 * per * sizeof(float), 256) +
           2 * align_up((size_t)C * sizeof(float2), 256);
}

static int check_bn(const char *who, const void *a, const void *b, int64_t n, int64_t C, const void *ws, size_t ws_bytes)
{
    if (n < 2) return fail(QBP_ERR_INVALID_ARG, "%s: n must be at least 2 (C(1) is infinite)", who);
    if (C <= 0) return fail(QBP_ERR_INVALID_ARG, "%s: C must be positive", who);
    if (!a || !b) return fail(QBP_ERR_INVALID_ARG, "%s: NULL tensor", who);
    if (!ws || ws_bytes < bn_ws_bytes(C))
        return fail(QBP_ERR_WORKSPACE, "%s: workspace of %zu bytes needed, %zu given", who, bn_ws_bytes(C), ws_bytes);
    return QBP_OK;
}

// Upper bound on the (min, max) partials rangebn_bwd_impl writes: row strips x column slabs of the apply grid.
size_t rangebn_range_parts_capacity(int64_t C)
{
    // (vector columns may be single floats: C columns in slabs of kScanMaxTw)
    return (size_t)kScanMaxStrips * (size_t)((C + kScanMaxTw - 1) / kScanMaxTw + 1);
}

}  // namespace qbp

using namespace qbp;

extern "C" __attribute__((visibility("default"))) size_t qbp_rangebn_workspace_bytes(int64_t n, int64_t C)
{
    (void)n;
    return bn_ws_bytes(C > 0 ? C : 1);
}

namespace qbp {

// The apply pass (and what hangs on it) from per-channel mean / min / max that are already in save_*:
// the exact range of y and the next layer's 8-bit parameters when asked for, y and / or its 8-bit codes.
// n_stat: the rows the statistics were taken over (more than n_rows when several GPUs share a minibatch).
static int bn_fwd_apply_launch(const float *x, int64_t n_rows, int64_t n_stat, int64_t C, const float *gamma,
                               const float *beta, int relu, float *y, const float *save_mean, const float *save_min,
                               const float *save_max, qbp_qparams *out_range, const qbp_requant *rq, cudaStream_t st,
                               bool reverse, int64_t keep_head = 0, bool totals_cleared = false)
{
    const bool requant = rq != nullptr;
    if (requant && (!rq->q || !rq->qp)) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: the requantisation record needs q and qp");
    if (!y && !requant) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: neither y nor 8-bit codes wanted");
    const bool al = aligned16(x) && (!y || aligned16(y)) && (!requant || ((uintptr_t)rq->q & 3) == 0);
    const bool v4 = al && C % 4 == 0;
    const int bps = v4 ? (requant ? (relu ? blocks_per_sm<bn_apply_kernel<4, true, true>>(kScanThreads)
                                          : blocks_per_sm<bn_apply_kernel<4, false, true>>(kScanThreads))
                                  : (relu ? blocks_per_sm<bn_apply_kernel<4, true, false>>(kScanThreads)
                                          : blocks_per_sm<bn_apply_kernel<4, false, false>>(kScanThreads)))
                       : blocks_per_sm<bn_apply_kernel<1, true, true>>(kScanThreads);
    const ScanGeom ga = scan_geom(n_rows, C, al, bps);
    const dim3 grid_apply(ga.nbx, ga.slabs);
    const float Cn = (float)(1.0 / std::sqrt(2.0 * std::log((double)n_stat)));
    const bool own_range = requant && !out_range && C <= kBnOwnRangeMax;
    if ((out_range || requant) && !own_range) {
        QBP_TRACE_BEGIN(st);
        launch(bn_out_range_kernel, 1, 256, 0, st, save_mean, save_min, save_max, gamma, beta, (int)C, Cn, relu, out_range,
                                               requant ? rq->qp : nullptr, nullptr);
        QBP_LAUNCH_OK("bn_out_range_kernel");
    }
    BnRequant R{nullptr, nullptr, nullptr, 1, nullptr, own_range ? 1 : 0};
    bool fused_rowsum = false;
    if (requant) {
        R.rq = rq->qp; R.q = rq->q;
        // the row's lanes sit in one warp when the block is at most 32 vectors wide and one slab covers the row
        fused_rowsum = rq->row_sums && ga.tw <= 32 && ga.slabs == 1;
        if (fused_rowsum) { R.rowsum = rq->row_sums; R.rs_group = ga.tw; }
        if (rq->chan_sums) {
            if (n_rows >= (1ll << 22)) return fail(QBP_ERR_UNSUPPORTED_SHAPE, "rangebn_fwd: per-channel code totals for fewer than 2^22 rows");
            if (!totals_cleared)
                if (int rc = launch_clear(rq->chan_sums, 2 * C, st)) return rc;
            R.chansum = reinterpret_cast<unsigned long long *>(rq->chan_sums);
        }
    }
    QBP_TRACE_BEGIN(st);
#define QBP_BN_APPLY(V, RL, RQ) launch(bn_apply_kernel<V, RL, RQ>, grid_apply, kScanThreads, 0, st, x, n_rows, (int)C, ga.tw, save_mean, save_min, save_max, gamma, beta, Cn, y, R, reverse ? 1 : 0, keep_head)
    if (ga.vec == 4) {
        if (requant) { if (relu) QBP_BN_APPLY(4, true, true); else QBP_BN_APPLY(4, false, true); }
        else         { if (relu) QBP_BN_APPLY(4, true, false); else QBP_BN_APPLY(4, false, false); }
    } else {
        if (requant) { if (relu) QBP_BN_APPLY(1, true, true); else QBP_BN_APPLY(1, false, true); }
        else         { if (relu) QBP_BN_APPLY(1, true, false); else QBP_BN_APPLY(1, false, false); }
    }
#undef QBP_BN_APPLY
    QBP_LAUNCH_OK("bn_apply_kernel");
    if (requant && rq->row_sums && !fused_rowsum) return launch_rowsum(rq->q, true, n_rows, C, rq->row_sums, st);
    return QBP_OK;
}

// The statistics pass: partials per strip, then either mean / min / max (mean != NULL) or the raw sum / min / max.
static int bn_fwd_stats_launch(const float *x, int64_t n, int64_t C, float *mean, float *vmin, float *vmax, double *sum_out,
                               void *ws, size_t ws_bytes, cudaStream_t st)
{
    WsCarver w(ws, ws_bytes);
    double *psum = w.take<double>((size_t)kScanMaxStrips * C);
    w.take<double>((size_t)kScanMaxStrips * C);
    float *plo = w.take<float>((size_t)kScanMaxStrips * C);
    float *phi = w.take<float>((size_t)kScanMaxStrips * C);
    const bool al = aligned16(x);
    const bool v4 = al && C % 4 == 0;
    const ScanGeom g = scan_geom(n, C, al, v4 ? blocks_per_sm<bn_stats_kernel<4>>(kScanThreads)
                                              : blocks_per_sm<bn_stats_kernel<1>>(kScanThreads));
    const dim3 grid(g.nbx, g.slabs);
    QBP_TRACE_BEGIN(st);
    if (g.vec == 4) launch(bn_stats_kernel<4>, grid, kScanThreads, 0, st, x, n, (int)C, g.tw, plo, phi, psum, keep_from_row(n, 4 * C));
    else            launch(bn_stats_kernel<1>, grid, kScanThreads, 0, st, x, n, (int)C, g.tw, plo, phi, psum, keep_from_row(n, 4 * C));
    QBP_LAUNCH_OK("bn_stats_kernel");
    QBP_TRACE_BEGIN(st);
    launch(bn_stats_finalize_kernel, (int)C, 128, 0, st, plo, phi, psum, g.nbx, (int)C, n, mean, vmin, vmax, sum_out);
    QBP_LAUNCH_OK("bn_stats_finalize_kernel");
    return QBP_OK;
}

}  // namespace qbp

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_fwd_q8(const float *x, int64_t n, int64_t C, const float *gamma, const float *beta, int relu,
                               float *y, float *save_mean, float *save_min, float *save_max, qbp_qparams *out_range,
                               const qbp_requant *rq, void *ws, size_t ws_bytes, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    int rc = check_bn("rangebn_fwd", x, x, n, C, ws, ws_bytes);
    if (rc) return rc;
    if (!y && !rq) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: NULL tensor");
    if (!save_mean || !save_min || !save_max) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: NULL statistics buffer");
    if (!rq && !out_range && few_rows(n, C) && aligned16(x) && aligned16(y)) {
        const float Cn = (float)(1.0 / std::sqrt(2.0 * std::log((double)n)));
        QBP_TRACE_BEGIN(st);
#define QBP_BN_FEW(CH_, ROWS_) launch(bn_fwd_few_kernel<CH_, ROWS_>, (int)((C + CH_ - 1) / CH_), kFewThreads, 0, st, x, (int)n, (int)C, gamma, beta, \
                                      relu, Cn, y, save_mean, save_min, save_max)
        if (few_narrow(n, C, 0)) { if (n <= 4 * kFewHigh<8>) QBP_BN_FEW(8, 4); else QBP_BN_FEW(8, 8); }
        else if (n <= kFewHigh<16>)     QBP_BN_FEW(16, 1);
        else if (n <= 4 * kFewHigh<16>) QBP_BN_FEW(16, 4);
        else                            QBP_BN_FEW(16, 16);
#undef QBP_BN_FEW
        QBP_LAUNCH_OK("bn_fwd_few_kernel");
        return QBP_OK;
    }
    if ((rc = bn_fwd_stats_launch(x, n, C, save_mean, save_min, save_max, nullptr, ws, ws_bytes, st))) return rc;
    return bn_fwd_apply_launch(x, n, n, C, gamma, beta, relu, y, save_mean, save_min, save_max, out_range, rq, st, true, kKeepBytes / (4 * C));
}

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_fwd(const float *x, int64_t n, int64_t C, const float *gamma, const float *beta, int relu,
                               float *y, float *save_mean, float *save_min, float *save_max, qbp_qparams *out_range,
                               void *ws, size_t ws_bytes, void *stream)
{
    if (!y) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: NULL tensor");
    return qbp_rangebn_fwd_q8(x, n, C, gamma, beta, relu, y, save_mean, save_min, save_max, out_range, nullptr, ws, ws_bytes, stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_fwd_stats(const float *x, int64_t n, int64_t C, double *col_sum, float *col_min,
                               float *col_max, void *ws, size_t ws_bytes, void *stream)
{
    // (n = 1 is a valid share of a larger minibatch: the n >= 2 rule applies to n_stat of the apply call)
    if (n < 1 || C <= 0) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd_stats: n and C must be positive");
    if (!x || !col_sum || !col_min || !col_max) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd_stats: NULL argument");
    if (!ws || ws_bytes < bn_ws_bytes(C))
        return fail(QBP_ERR_WORKSPACE, "rangebn_fwd_stats: workspace of %zu bytes needed, %zu given", bn_ws_bytes(C), ws_bytes);
    return bn_fwd_stats_launch(x, n, C, nullptr, col_min, col_max, col_sum, ws, ws_bytes, (cudaStream_t)stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_fwd_apply(const float *x, int64_t n_rows, int64_t n_stat, int64_t C, const double *col_sum,
                               const float *col_min, const float *col_max, const float *gamma, const float *beta, int relu,
                               float *y, float *save_mean, float *save_min, float *save_max, qbp_qparams *out_range,
                               const qbp_requant *rq, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (n_rows < 1 || n_stat < n_rows || C <= 0) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd_apply: needs 1 <= n_rows <= n_stat, C > 0");
    if (n_stat < 2) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd_apply: n_stat must be at least 2 (C(1) is infinite)");
    if (!x || !col_sum || !col_min || !col_max || !save_mean || !save_min || !save_max)
        return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd_apply: NULL argument");
    QBP_TRACE_BEGIN(st);
    launch(bn_mean_from_sum_kernel, (int)((C + 255) / 256), 256, 0, st, col_sum, col_min, col_max, (int)C, n_stat, save_mean, save_min, save_max);
    QBP_LAUNCH_OK("bn_mean_from_sum_kernel");
    // (nothing kept for a backward call, which here comes after other layers: 103 MB statistics + apply 55.4 us with it, 53.2 without)
    return bn_fwd_apply_launch(x, n_rows, n_stat, C, gamma, beta, relu, y, save_mean, save_min, save_max, out_range, rq, st, true, 0);
}

// The statistics half of the recompute fusion (a convolution run twice: once for the statistics, once to write
// the normalised output as 8-bit codes): from the partials the first run left, the saved statistics, the 8-bit
// parameters of the output and, per channel, (mean, scale, gamma, beta) for the second run's epilogue.
int qbp::rangebn_fold_from_parts(int64_t n, int64_t C, const float *gamma, const float *beta, int relu, float *save_mean,
                                 float *save_min, float *save_max, const ColStatParts &parts, qbp_qparams *qp8_out,
                                 float4 *fold, cudaStream_t st)
{
    if (!save_mean || !save_min || !save_max || !parts.lo || !parts.hi || !parts.sum || parts.rows <= 0 || !qp8_out || !fold)
        return fail(QBP_ERR_INVALID_ARG, "rangebn: NULL argument");
    if (n < 2 || C <= 0) return fail(QBP_ERR_INVALID_ARG, "rangebn: needs n >= 2 rows");
    const float Cn = (float)(1.0 / std::sqrt(2.0 * std::log((double)n)));
    QBP_TRACE_BEGIN(st);
    launch(bn_stats_finalize_kernel, (int)C, 128, 0, st, parts.lo, parts.hi, parts.sum, parts.rows, (int)C, n, save_mean, save_min, save_max, nullptr);
    QBP_LAUNCH_OK("bn_stats_finalize_kernel");
    QBP_TRACE_BEGIN(st);
    launch(bn_out_range_kernel, 1, 256, 0, st, save_mean, save_min, save_max, gamma, beta, (int)C, Cn, relu, nullptr, qp8_out, fold);
    QBP_LAUNCH_OK("bn_out_range_kernel");
    return QBP_OK;
}

// Forward from per-column partials of x that its producer left (rows of [C]: sum, min, max), without a statistics
// pass over x: finalize, then the apply pass.
int qbp::rangebn_fwd_from_parts(const float *x, int64_t n, int64_t C, const float *gamma, const float *beta, int relu,
                                float *y, float *save_mean, float *save_min, float *save_max, const ColStatParts &parts,
                                qbp_qparams *out_range, const qbp_requant *rq, cudaStream_t st, bool totals_cleared)
{
    if (!x || !save_mean || !save_min || !save_max || !parts.lo || !parts.hi || !parts.sum || parts.rows <= 0)
        return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: NULL tensor");
    if (n < 2 || C <= 0) return fail(QBP_ERR_INVALID_ARG, "rangebn_fwd: needs n >= 2 rows");
    QBP_TRACE_BEGIN(st);
    launch(bn_stats_finalize_kernel, (int)C, 128, 0, st, parts.lo, parts.hi, parts.sum, parts.rows, (int)C, n, save_mean, save_min, save_max, nullptr);
    QBP_LAUNCH_OK("bn_stats_finalize_kernel");
    // (the product that left the statistics has just written x: its tail is in the L2)
    return bn_fwd_apply_launch(x, n, n, C, gamma, beta, relu, y, save_mean, save_min, save_max, out_range, rq, st, true, 0, totals_cleared);
}

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_bwd(const float *dy, const float *x, int64_t n, int64_t C, const float *gamma,
                               const float *beta, int relu, const float *save_mean, const float *save_min,
                               const float *save_max, float *dx, float *dgamma, float *dbeta, void *ws,
                               size_t ws_bytes, void *stream)
{
    return rangebn_bwd_impl(dy, x, n, C, gamma, beta, relu, save_mean, save_min, save_max, dx, dgamma, dbeta, ws, ws_bytes,
                            nullptr, nullptr, (cudaStream_t)stream);
}

namespace qbp {

static int bn_bwd_stats_launch(const float *dy, const float *x, int64_t n_rows, int64_t n_stat, int64_t C, const float *gamma,
                               const float *beta, int relu, const float *save_mean, const float *save_min,
                               const float *save_max, float *dgamma, float *dbeta, float2 *coef, double *sum_dy,
                               double *sum_dyx, double *pa, double *pb, cudaStream_t st, float *ext = nullptr,
                               float2 *chan_range = nullptr, float2 *relu_thr = nullptr, const ZeroJobs &zero = ZeroJobs{},
                               const SumJob *extra = nullptr, int extra_count = 0, bool keep_tail = true)
{
    const bool al = aligned16(x) && aligned16(dy);
    const bool v4 = al && C % 4 == 0;
    const ScanGeom g = scan_geom(n_rows, C, al, v4 ? (ext ? blocks_per_sm<bn_bwd_stats_kernel<4, true, true>>(kScanThreads)
                                                          : relu ? blocks_per_sm<bn_bwd_stats_kernel<4, true, false>>(kScanThreads)
                                                                 : blocks_per_sm<bn_bwd_stats_kernel<4, false, false>>(kScanThreads))
                                                   : blocks_per_sm<bn_bwd_stats_kernel<1, true, false>>(kScanThreads));
    const dim3 grid(g.nbx, g.slabs);
    const double Cnd = 1.0 / std::sqrt(2.0 * std::log((double)n_stat));
    const float Cn = (float)Cnd;
    const int64_t keep_from = keep_tail ? keep_from_row(n_rows, 8 * C) : n_rows;
    QBP_TRACE_BEGIN(st);
#define QBP_BN_BSTATS(V, R, E) launch(bn_bwd_stats_kernel<V, R, E>, grid, kScanThreads, 0, st, dy, x, n_rows, (int)C, g.tw, save_mean, save_min, save_max, gamma, beta, Cn, pa, pb, ext, zero, keep_from)
    if (ext) {
        if (g.vec != 4) return fail(QBP_ERR_UNSUPPORTED_SHAPE, "rangebn_bwd: the pass with dy extremes needs aligned tensors and C a multiple of 4");
        if (relu) QBP_BN_BSTATS(4, true, true); else QBP_BN_BSTATS(4, false, true);
    } else if (g.vec == 4) { if (relu) QBP_BN_BSTATS(4, true, false); else QBP_BN_BSTATS(4, false, false); }
    else                   { if (relu) QBP_BN_BSTATS(1, true, false); else QBP_BN_BSTATS(1, false, false); }
#undef QBP_BN_BSTATS
    QBP_LAUNCH_OK("bn_bwd_stats_kernel");
    QBP_TRACE_BEGIN(st);
    SumJobs J{};
    int sum_blocks = 0;
    if (extra_count) if (int rc = fill_sum_jobs(extra, extra_count, J, &sum_blocks)) return rc;
#define QBP_BN_BFIN(T) launch(bn_bwd_finalize_kernel<T>, (int)C + sum_blocks, T, 0, st, pa, pb, g.nbx, (int)C, n_stat, gamma, Cnd, dgamma, dbeta, coef, sum_dy, sum_dyx, ext, save_min, save_max, Cn, chan_range, save_mean, beta, relu_thr, J)
    if (sum_blocks || g.nbx > 256) QBP_BN_BFIN(kSumThreads); else if (g.nbx > 128) QBP_BN_BFIN(128); else QBP_BN_BFIN(64);
#undef QBP_BN_BFIN
    QBP_LAUNCH_OK("bn_bwd_finalize_kernel");
    return QBP_OK;
}

static int bn_bwd_apply_launch(const float *dy, const float *x, int64_t n_rows, int64_t n_stat, int64_t C, const float *gamma,
                               const float *beta, int relu, const float *save_mean, const float *save_min,
                               const float *save_max, const float2 *coef, float *dx, float2 *range_parts, int *nparts,
                               cudaStream_t st)
{
    const bool al = aligned16(x) && aligned16(dy) && aligned16(dx);
    const bool v4 = al && C % 4 == 0;
    const ScanGeom ga = scan_geom(n_rows, C, al, v4 ? (relu ? blocks_per_sm<bn_bwd_apply_kernel<4, true, true>>(kScanThreads)
                                                            : blocks_per_sm<bn_bwd_apply_kernel<4, false, true>>(kScanThreads))
                                                    : blocks_per_sm<bn_bwd_apply_kernel<1, true, true>>(kScanThreads));
    const dim3 grid_apply(ga.nbx, ga.slabs);
    const float Cn = (float)(1.0 / std::sqrt(2.0 * std::log((double)n_stat)));
    QBP_TRACE_BEGIN(st);
#define QBP_BN_BAPPLY(V, R, G) launch(bn_bwd_apply_kernel<V, R, G>, grid_apply, kScanThreads, 0, st, dy, x, n_rows, (int)C, ga.tw, save_mean, save_min, save_max, gamma, beta, Cn, coef, dx, range_parts)
    if (range_parts) {
        if (ga.vec == 4) { if (relu) QBP_BN_BAPPLY(4, true, true); else QBP_BN_BAPPLY(4, false, true); }
        else             { if (relu) QBP_BN_BAPPLY(1, true, true); else QBP_BN_BAPPLY(1, false, true); }
        if (nparts) *nparts = (int)(grid_apply.x * grid_apply.y);
    } else {
        if (ga.vec == 4) { if (relu) QBP_BN_BAPPLY(4, true, false); else QBP_BN_BAPPLY(4, false, false); }
        else             { if (relu) QBP_BN_BAPPLY(1, true, false); else QBP_BN_BAPPLY(1, false, false); }
    }
#undef QBP_BN_BAPPLY
    QBP_LAUNCH_OK("bn_bwd_apply_kernel");
    return QBP_OK;
}

// Whether the statistics of rangebn_bwd_bifurcate_impl are one launch: what it clears is then not clear before `extra` runs.
bool rangebn_bwd_one_launch(int64_t n, int64_t C) { return few_rows(n, C); }

// Whether rangebn_bwd_bifurcate_impl takes these tensors.  (Philox blocks below 2^32: more elements do not fit the device)
bool rangebn_bwd_bifurcate_supported(const float *dy, const float *x, const float *g_out, int64_t n, int64_t C)
{
    return aligned16(x) && aligned16(dy) && (!g_out || aligned16(g_out)) && C % 4 == 0 && n >= 2 && n * C < (1ll << 34);
}

// Range BN backward and the bifurcation of its result in two passes over (dy, x): statistics with the extremes of dy
// (from which the exact range of the gradient follows), then the pass that computes the gradient and writes its 8-bit
// copy, the limbs of its 16-bit copy and the rows' code sums -- and the fp32 gradient only when g_out is given.
int rangebn_bwd_bifurcate_impl(const float *dy, const float *x, int64_t n, int64_t C, const float *gamma, const float *beta,
                               int relu, const float *save_mean, const float *save_min, const float *save_max, float *g_out,
                               float *dgamma, float *dbeta, uint64_t seed, uint32_t id8, uint32_t id16, int8_t *q8,
                               qbp_qparams *qp8, int32_t *row_sums8, int8_t *hi, uint8_t *lo, qbp_qparams *qp16, bool lo_signed,
                               void *ws, size_t ws_bytes, cudaStream_t st, int64_t *tot16, void *clear,
                               int64_t clear_words, const SumJob *extra, int extra_count)
{
    int rc = check_bn("rangebn_bwd", dy, x, n, C, ws, ws_bytes);
    if (rc) return rc;
    if (!rangebn_bwd_bifurcate_supported(dy, x, g_out, n, C) || ((uintptr_t)q8 & 3) || ((uintptr_t)hi & 3) || ((uintptr_t)lo & 3))
        return fail(QBP_ERR_UNSUPPORTED_SHAPE, "rangebn_bwd (bifurcating): shape or alignment not taken");
    WsCarver w(ws, ws_bytes);
    double *pa = w.take<double>((size_t)kScanMaxStrips * C);
    double *pb = w.take<double>((size_t)kScanMaxStrips * C);
    w.take<float>((size_t)kScanMaxStrips * C);
    w.take<float>((size_t)kScanMaxStrips * C);
    float2 *coef = w.take<float2>((size_t)C);
    w.take<char>(256);
    float *ext = w.take<float>(6 * (size_t)kScanMaxStrips * C);
    float2 *chan_range = w.take<float2>((size_t)C);
    float2 *relu_thr = w.take<float2>((size_t)C);
    // (kBabBlocks resident blocks per SM, by the kernel's launch bounds and its ring, whatever the instance)
    const ScanGeom ga = scan_geom(n, C, true, kBabBlocks);
    // each row's code sum by shuffles over the row's lanes of a warp; a row that spans several warps or blocks is
    // added up from its pieces (integer atomics on the zeroed sums: the result does not depend on the order)
    ZeroJobs zero{};
    if (row_sums8 && (ga.tw > 32 || ga.slabs > 1) && (rc = zero.add(row_sums8, n))) return rc;
    if ((rc = zero.add(clear, clear_words))) return rc;
    if (few_rows(n, C)) {
        if ((rc = launch_bwd_few(dy, x, n, C, gamma, beta, relu, save_mean, save_min, save_max,
                                 BnBwdOut{dgamma, dbeta, coef, chan_range, relu ? relu_thr : nullptr}, zero, extra, extra_count, st)))
            return rc;
    } else if ((rc = bn_bwd_stats_launch(dy, x, n, n, C, gamma, beta, relu, save_mean, save_min, save_max, dgamma, dbeta, coef, nullptr,
                                  nullptr, pa, pb, st, ext, chan_range, relu ? relu_thr : nullptr, zero, extra, extra_count, g_out != nullptr)))
        return rc;
    const RangeSrc range{chan_range, (int)C, nullptr, qp8, qp16};
    const dim3 grid(ga.nbx, ga.slabs);
    const float Cn = (float)(1.0 / std::sqrt(2.0 * std::log((double)n)));
    const PhiloxKeys keys = philox_keys_host(seed);
    const uint32_t flip = lo_signed ? 0x80808080u : 0u;
    QBP_TRACE_BEGIN(st);
#define QBP_BN_BAB(R, G, T, O)                                                                                          \
    do {                                                                                                                \
        static PerDeviceOnce once_;                                                                                     \
        QBP_SMEM_OPT_IN(once_, (bn_bwd_apply_bifurcate_kernel<R, G, T, O>), kBabRingBytes);                             \
        launch(bn_bwd_apply_bifurcate_kernel<R, G, T, O>, grid, kScanThreads, kBabRingBytes, st,                        \
               reinterpret_cast<const float4 *>(dy), reinterpret_cast<const float4 *>(x), (uint32_t)n, (int)C, ga.tw,   \
               save_min, save_max, gamma, Cn, coef, reinterpret_cast<float4 *>(g_out), range, id8, id16, keys,          \
               reinterpret_cast<uint32_t *>(q8), reinterpret_cast<uint32_t *>(hi), reinterpret_cast<uint32_t *>(lo),    \
               flip, row_sums8, reinterpret_cast<unsigned long long *>(tot16), relu_thr);                               \
    } while (0)
#define QBP_BN_BAB1(R, G, T) do { if (id8 == id16) QBP_BN_BAB(R, G, T, true); else QBP_BN_BAB(R, G, T, false); } while (0)
#define QBP_BN_BAB2(R, G) do { if (tot16) QBP_BN_BAB1(R, G, true); else QBP_BN_BAB1(R, G, false); } while (0)
    if (g_out) { if (relu) QBP_BN_BAB2(true, true); else QBP_BN_BAB2(false, true); }
    else       { if (relu) QBP_BN_BAB2(true, false); else QBP_BN_BAB2(false, false); }
#undef QBP_BN_BAB2
#undef QBP_BN_BAB1
#undef QBP_BN_BAB
    QBP_LAUNCH_OK("bn_bwd_apply_bifurcate_kernel");
    return QBP_OK;
}

}  // namespace qbp

// range_parts (nullable, room for rangebn_range_parts_capacity(C) entries) receives one (min, max) of dx per
// block of the apply pass; *nparts their count.
int qbp::rangebn_bwd_impl(const float *dy, const float *x, int64_t n, int64_t C, const float *gamma, const float *beta,
                          int relu, const float *save_mean, const float *save_min, const float *save_max, float *dx,
                          float *dgamma, float *dbeta, void *ws, size_t ws_bytes, float2 *range_parts, int *nparts,
                          cudaStream_t st)
{
    int rc = check_bn("rangebn_bwd", x, dy, n, C, ws, ws_bytes);
    if (rc) return rc;
    if (!dx || !save_mean || !save_min || !save_max) return fail(QBP_ERR_INVALID_ARG, "rangebn_bwd: NULL tensor");
    WsCarver w(ws, ws_bytes);
    double *pa = w.take<double>((size_t)kScanMaxStrips * C);
    double *pb = w.take<double>((size_t)kScanMaxStrips * C);
    w.take<float>((size_t)kScanMaxStrips * C);
    w.take<float>((size_t)kScanMaxStrips * C);
    float2 *coef = w.take<float2>((size_t)C);
    if (few_rows(n, C) && aligned16(x) && aligned16(dy)) {
        if ((rc = launch_bwd_few(dy, x, n, C, gamma, beta, relu, save_mean, save_min, save_max, BnBwdOut{dgamma, dbeta, coef, nullptr, nullptr},
                                 ZeroJobs{}, nullptr, 0, st)))
            return rc;
    } else if ((rc = bn_bwd_stats_launch(dy, x, n, n, C, gamma, beta, relu, save_mean, save_min, save_max, dgamma, dbeta, coef,
                                  nullptr, nullptr, pa, pb, st)))
        return rc;
    return bn_bwd_apply_launch(dy, x, n, n, C, gamma, beta, relu, save_mean, save_min, save_max, coef, dx, range_parts, nparts, st);
}

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_bwd_stats(const float *dy, const float *x, int64_t n_rows, int64_t n_stat, int64_t C,
                               const float *gamma, const float *beta, int relu, const float *save_mean,
                               const float *save_min, const float *save_max, double *sum_dy, double *sum_dyxhat,
                               void *ws, size_t ws_bytes, void *stream)
{
    if (n_rows < 1 || n_stat < n_rows || n_stat < 2 || C <= 0)
        return fail(QBP_ERR_INVALID_ARG, "rangebn_bwd_stats: needs 1 <= n_rows <= n_stat, n_stat >= 2, C > 0");
    if (!dy || !x || !save_mean || !save_min || !save_max || !sum_dy || !sum_dyxhat)
        return fail(QBP_ERR_INVALID_ARG, "rangebn_bwd_stats: NULL argument");
    if (!ws || ws_bytes < bn_ws_bytes(C))
        return fail(QBP_ERR_WORKSPACE, "rangebn_bwd_stats: workspace of %zu bytes needed, %zu given", bn_ws_bytes(C), ws_bytes);
    WsCarver w(ws, ws_bytes);
    double *pa = w.take<double>((size_t)kScanMaxStrips * C);
    double *pb = w.take<double>((size_t)kScanMaxStrips * C);
    return bn_bwd_stats_launch(dy, x, n_rows, n_stat, C, gamma, beta, relu, save_mean, save_min, save_max, nullptr, nullptr,
                               nullptr, sum_dy, sum_dyxhat, pa, pb, (cudaStream_t)stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_rangebn_bwd_apply(const float *dy, const float *x, int64_t n_rows, int64_t n_stat, int64_t C,
                               const float *gamma, const float *beta, int relu, const float *save_mean,
                               const float *save_min, const float *save_max, const double *sum_dy,
                               const double *sum_dyxhat, float *dx, float *dgamma, float *dbeta, void *ws,
                               size_t ws_bytes, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (n_rows < 1 || n_stat < n_rows || n_stat < 2 || C <= 0)
        return fail(QBP_ERR_INVALID_ARG, "rangebn_bwd_apply: needs 1 <= n_rows <= n_stat, n_stat >= 2, C > 0");
    if (!dy || !x || !dx || !save_mean || !save_min || !save_max || !sum_dy || !sum_dyxhat)
        return fail(QBP_ERR_INVALID_ARG, "rangebn_bwd_apply: NULL argument");
    if (!ws || ws_bytes < bn_ws_bytes(C))
        return fail(QBP_ERR_WORKSPACE, "rangebn_bwd_apply: workspace of %zu bytes needed, %zu given", bn_ws_bytes(C), ws_bytes);
    WsCarver w(ws, ws_bytes);
    w.take<double>((size_t)kScanMaxStrips * C);
    w.take<double>((size_t)kScanMaxStrips * C);
    w.take<float>((size_t)kScanMaxStrips * C);
    w.take<float>((size_t)kScanMaxStrips * C);
    float2 *coef = w.take<float2>((size_t)C);
    const double Cnd = 1.0 / std::sqrt(2.0 * std::log((double)n_stat));
    QBP_TRACE_BEGIN(st);
    launch(bn_bwd_coef_kernel, (int)((C + 255) / 256), 256, 0, st, sum_dy, sum_dyxhat, (int)C, n_stat, gamma, Cnd, dgamma, dbeta, coef);
    QBP_LAUNCH_OK("bn_bwd_coef_kernel");
    return bn_bwd_apply_launch(dy, x, n_rows, n_stat, C, gamma, beta, relu, save_mean, save_min, save_max, coef, dx, nullptr, nullptr, st);
}
