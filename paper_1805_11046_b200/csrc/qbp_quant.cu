// Range quantiser kernels (Section 4 "Quantization methods", Appendix B):
// min/max range scan, scale / zero-point, nearest and stochastic rounding to
// 8 and 16 bits, byte-limb split of the 16-bit codes, and the fused
// "bifurcation" that writes the 8-bit and 16-bit copies of a gradient from
// one read.  All of it is HBM-bound streaming work: 16-byte loads, 4 loads in
// flight per thread, warp-shuffle + shared-memory reductions, grids sized to
// fill every SM.  Also hosts the library's error-reporting state.
#include "qbp_colscan.cuh"
#include "qbp_mma.cuh"
#include "qbp_pair.cuh"
#include "qbp_sums.cuh"

#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

namespace qbp {

// ------------------------------------------------------------ error state
static thread_local char g_err[512] = "";

void set_error(const char *fmt, ...)
{
    va_list ap; va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}
int fail(int status, const char *fmt, ...)
{
    va_list ap; va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return status;
}
int sm_count()
{
    static thread_local int cached_dev = -1, cached = 148;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 148; }
    if (dev != cached_dev) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) cached = n;
        else cudaGetLastError();
        cached_dev = dev;
    }
    return cached;
}

// ------------------------------------------------------------ launch tracing
struct TraceRec { const char *name; cudaEvent_t a, b; };
static bool g_trace_on = false;
static std::vector<TraceRec> g_trace;
static std::vector<cudaEvent_t> g_event_pool;

static cudaEvent_t pool_event()
{
    if (!g_event_pool.empty()) { cudaEvent_t e = g_event_pool.back(); g_event_pool.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}
bool trace_is_on() { return g_trace_on; }
void trace_begin(cudaStream_t st)
{
    if (!g_trace_on) return;
    TraceRec r{nullptr, pool_event(), pool_event()};
    cudaEventRecord(r.a, st);
    g_trace.push_back(r);
}
void trace_end(const char *name, cudaStream_t st)
{
    if (!g_trace_on || g_trace.empty() || g_trace.back().name) return;
    g_trace.back().name = name;
    cudaEventRecord(g_trace.back().b, st);
}

constexpr int kThreads = 256;
constexpr int kUnroll = 4;
constexpr int kRangeUnroll = 8;          // loads in flight per thread of the read-only range scan
constexpr int kMaxParts = 4096;          // upper bound on per-tensor scan blocks

// ------------------------------------------------------- per-tensor range
// keep_rev: the tensor is walked from its end with loads that leave the lines in the L2 -- where nearest rounding follows from the
// front, bound by HBM, and so finds the first 100 MB there (103 MB 38.2 -> 35.4 us, 206 MB 73.2 -> 69.7).  Stochastic rounding is
// bound by the integer pipes and only pays for the slower scan (53.6 -> 55.5).
// Up to two tensors in one launch (a layer's weights, b, beside its activation, a): the first b.blocks blocks take b.
struct ScanJob { const float *x; int64_t n; float2 *parts; int blocks, keep_rev; };
template <int VEC>
__global__ void __launch_bounds__(kThreads) range_partial_kernel(const __grid_constant__ ScanJob a, const __grid_constant__ ScanJob b,
                                                                 const __grid_constant__ ZeroJobs zero)
{
    pdl_wait();
    const bool second = (int)blockIdx.x < b.blocks;
    const ScanJob &J = second ? b : a;
    const int block = second ? (int)blockIdx.x : (int)blockIdx.x - b.blocks;
    run_zero_jobs(zero, (int64_t)blockIdx.x * kThreads + threadIdx.x, (int64_t)gridDim.x * kThreads);
    const float *__restrict__ x = J.x;
    float lo = INFINITY, hi = -INFINITY;
    const int64_t nv = J.n / VEC;
    const int64_t stride = (int64_t)J.blocks * kThreads * kRangeUnroll;
    for (int64_t base = (int64_t)block * kThreads * kRangeUnroll; base < nv; base += stride) {
        VecF<VEC> v[kRangeUnroll];
        bool ok[kRangeUnroll];
#pragma unroll
        for (int u = 0; u < kRangeUnroll; ++u) {
            int64_t i = base + u * kThreads + threadIdx.x;
            ok[u] = i < nv;
            if (ok[u]) { if (J.keep_rev) v[u].load(x + (nv - 1 - i) * VEC); else v[u].load_stream(x + i * VEC); }
        }
#pragma unroll
        for (int u = 0; u < kRangeUnroll; ++u)
            if (ok[u]) {
#pragma unroll
                for (int e = 0; e < VEC; ++e) { lo = fminf(lo, v[u].v[e]); hi = fmaxf(hi, v[u].v[e]); }
            }
    }
    if (block == 0 && threadIdx.x == 0)
        for (int64_t i = nv * VEC; i < J.n; ++i) { lo = fminf(lo, x[i]); hi = fmaxf(hi, x[i]); }
    const float2 r = block_min_max(lo, hi);
    if (threadIdx.x == 0) J.parts[block] = r;
}

// The parameters of an empty tensor.
__global__ void empty_qparams_kernel(qbp_qparams *qp8, qbp_qparams *qp16)
{
    pdl_wait();
    if (qp8) *qp8 = make_qparams(0.0f, 0.0f, 8);
    if (qp16) *qp16 = make_qparams(0.0f, 0.0f, 16);
}

// ---------------------------------------------- chunk-averaged clamping values
// Appendix B, activations: the clamping values are the averages, over K chunks of the tensor, of the chunks'
// minima and maxima.  blockIdx.y = chunk (equal contiguous runs of n_chunk elements), blockIdx.x = block inside it.
template <int VEC>
__global__ void __launch_bounds__(kThreads) chunk_range_partial_kernel(const float *__restrict__ x, int64_t n_chunk,
                                                                       float2 *__restrict__ partials)
{
    pdl_wait();
    x += (int64_t)blockIdx.y * n_chunk;
    float lo = INFINITY, hi = -INFINITY;
    const int64_t nv = n_chunk / VEC;              // (VEC = 4 only when n_chunk is a multiple of 4)
    const int64_t stride = (int64_t)gridDim.x * kThreads * kRangeUnroll;
    for (int64_t base = (int64_t)blockIdx.x * kThreads * kRangeUnroll; base < nv; base += stride) {
        VecF<VEC> v[kRangeUnroll];
        bool ok[kRangeUnroll];
#pragma unroll
        for (int u = 0; u < kRangeUnroll; ++u) {
            int64_t i = base + u * kThreads + threadIdx.x;
            ok[u] = i < nv;
            if (ok[u]) v[u].load_stream(x + i * VEC);
        }
#pragma unroll
        for (int u = 0; u < kRangeUnroll; ++u)
            if (ok[u]) {
#pragma unroll
                for (int e = 0; e < VEC; ++e) { lo = fminf(lo, v[u].v[e]); hi = fmaxf(hi, v[u].v[e]); }
            }
    }
    lo = warp_min(lo); hi = warp_max(hi);
    __shared__ float s_lo[kThreads / 32], s_hi[kThreads / 32];
    if ((threadIdx.x & 31) == 0) { s_lo[threadIdx.x >> 5] = lo; s_hi[threadIdx.x >> 5] = hi; }
    __syncthreads();
    if (threadIdx.x < 32) {
        lo = threadIdx.x < kThreads / 32 ? s_lo[threadIdx.x] : INFINITY;
        hi = threadIdx.x < kThreads / 32 ? s_hi[threadIdx.x] : -INFINITY;
        lo = warp_min(lo); hi = warp_max(hi);
        if (threadIdx.x == 0) partials[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = make_float2(lo, hi);
    }
}

// One block: every chunk's (min, max) from its blocks' partials (a warp per chunk, the lanes stride over the
// chunk's blocks), then the two averages, added up in chunk order in double by one thread (the order is part of
// the result: the result depends on it, and the CPU check adds them up the same way).
__global__ void __launch_bounds__(kThreads) chunk_range_finalize_kernel(const float2 *__restrict__ partials, int chunks,
                                                                        int blocks_per_chunk, float2 *__restrict__ per_chunk,
                                                                        qbp_qparams *__restrict__ out)
{
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = warp; k < chunks; k += kThreads / 32) {
        float lo = INFINITY, hi = -INFINITY;
        for (int b = lane; b < blocks_per_chunk; b += 32) {
            const float2 p = partials[(int64_t)k * blocks_per_chunk + b];
            lo = fminf(lo, p.x); hi = fmaxf(hi, p.y);
        }
        lo = warp_min(lo); hi = warp_max(hi);
        if (lane == 0) per_chunk[k] = make_float2(lo, hi);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double slo = 0.0, shi = 0.0;
        for (int k = 0; k < chunks; ++k) { slo += (double)per_chunk[k].x; shi += (double)per_chunk[k].y; }
        qbp_qparams r;
        r.scale = 0.0f; r.zero_point = 0;
        r.vmin = (float)(slo / (double)chunks); r.vmax = (float)(shi / (double)chunks);
        *out = r;
    }
}

// Parameters from clamping values the caller already has (one thread each).
__global__ void qparams_from_range_kernel(const qbp_qparams *__restrict__ in, int count, int bits,
                                          qbp_qparams *__restrict__ out)
{
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = make_qparams(in[i].vmin, in[i].vmax, bits);
}

// ------------------------------------------------------ per-channel range
template <int VEC>
__global__ void __launch_bounds__(kScanThreads) chan_range_partial_kernel(const float *__restrict__ x, int64_t rows,
                                                                          int C, int tw, float *__restrict__ part_lo,
                                                                          float *__restrict__ part_hi)
{
    pdl_wait();
    const ScanPos p = scan_pos<VEC>(C, tw);
    const int rpb = kScanThreads / tw;
    float lo[VEC], hi[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) { lo[e] = INFINITY; hi[e] = -INFINITY; }
    if (p.active) {
        const int64_t step = (int64_t)gridDim.x * rpb;
        for (int64_t r0 = (int64_t)blockIdx.x * rpb + p.ty; r0 < rows; r0 += step * kScanUnroll) {
            VecF<VEC> v[kScanUnroll];
            bool ok[kScanUnroll];
#pragma unroll
            for (int u = 0; u < kScanUnroll; ++u) {
                int64_t r = r0 + u * step;
                ok[u] = r < rows;
                if (ok[u]) v[u].load_stream(x + r * C + p.col);
            }
#pragma unroll
            for (int u = 0; u < kScanUnroll; ++u)
                if (ok[u]) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) { lo[e] = fminf(lo[e], v[u].v[e]); hi[e] = fmaxf(hi[e], v[u].v[e]); }
                }
        }
    }
    __shared__ float s_lo[kScanThreads * VEC], s_hi[kScanThreads * VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) { s_lo[threadIdx.x * VEC + e] = lo[e]; s_hi[threadIdx.x * VEC + e] = hi[e]; }
    __syncthreads();
    if (p.ty == 0 && p.active) {
        for (int y = 1; y < rpb; ++y)
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                lo[e] = fminf(lo[e], s_lo[(y * tw + p.tx) * VEC + e]);
                hi[e] = fmaxf(hi[e], s_hi[(y * tw + p.tx) * VEC + e]);
            }
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            part_lo[(int64_t)blockIdx.x * C + p.col + e] = lo[e];
            part_hi[(int64_t)blockIdx.x * C + p.col + e] = hi[e];
        }
    }
}

// One warp per channel over the strip partials.
__global__ void __launch_bounds__(kThreads) chan_range_finalize_kernel(const float *__restrict__ part_lo,
                                                                       const float *__restrict__ part_hi, int nparts,
                                                                       int C, int bits, qbp_qparams *__restrict__ qp)
{
    pdl_wait();
    int c = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    if (c >= C) return;
    float lo = INFINITY, hi = -INFINITY;
    for (int i = threadIdx.x & 31; i < nparts; i += 32) {
        lo = fminf(lo, part_lo[(int64_t)i * C + c]);
        hi = fmaxf(hi, part_hi[(int64_t)i * C + c]);
    }
    lo = warp_min(lo); hi = warp_max(hi);
    if ((threadIdx.x & 31) == 0) qp[c] = make_qparams(lo, hi, bits);
}

// ------------------------------------------------------------ quantisation
struct QuantOut {
    int8_t *q8;      // 8-bit codes (nullable)
    int16_t *q16;    // 16-bit codes (nullable)
    int8_t *hi;      // high byte of the 16-bit code (nullable)
    uint8_t *lo;     // low byte (nullable)
    // Sums of the stored 8-bit codes over each row of `cols` (nullable; vector path only).  rs_group lanes (a power of two that
    // divides cols / 4, at most 32) add up.  rs_shift >= 0: they are a whole row, cols / 4 = 2^rs_shift.  Else the sums are zero
    // beforehand and pieces are added: per group, or (rs_group 0: 128 columns or more, no multiple of 128) per warp, whose 128
    // elements meet at most two (in groups of the four lanes that divide 4080 columns the atomics of 4096 such rows took 40 us).
    int32_t *rowsum8;
    int rs_group, rs_shift;
    FastDiv rs_div;             // by cols / 4
    // Per-channel totals of the stored codes over all rows, added (64-bit atomics) to chansum8 [cols] / chansum16
    // [cols] (nullable; vector path, per tensor, cols / 4 a power of two <= 256: a thread then keeps its four
    // channels for its whole life).  The weight gradient's zero-point terms are built from such totals.
    unsigned long long *chansum8, *chansum16;
    // 0x80808080: the low bytes are stored with their top bit flipped, i.e. as the signed bytes lo - 128 (the weight
    // gradient then runs both limbs as one s8 x s8 product); 0: plain unsigned low bytes.
    uint32_t lo_flip;
};

static QuantOut quant_out(int8_t *q8, int16_t *q16, int8_t *hi, uint8_t *lo, uint32_t lo_flip = 0u)
{
    QuantOut o{};
    o.q8 = q8; o.q16 = q16; o.hi = hi; o.lo = lo; o.lo_flip = lo_flip;
    return o;
}

// Column sums beside the codes of a quantising launch's second tensor (NULL: not wanted).
struct StripJob { int64_t rows; int pieces; int32_t *col_sums; };

// One tensor of a quantising launch.
struct QuantJob {
    const float *x; int64_t n; int cols;
    RangeSrc r;                  // per channel: the records [cols] at r.qp8 / r.qp16
    uint32_t id8, id16; QuantOut o; int smem_cols; uint64_t index_base;
};

// Scalar path: unaligned tensors, per-element tails.  One Philox block per element.
template <bool SR>
__device__ __forceinline__ void quantize_scalar(const QuantJob &J, int64_t i, bool perch, const QParamsReg &t8, const QParamsReg &t16,
                                                const PhiloxKeys &key)
{
    const QuantOut &o = J.o;
    const uint32_t id8 = J.id8, id16 = J.id16;
    const int c = perch ? (int)(i % J.cols) : 0;
    const float v = J.x[i];
    const uint64_t j = ((uint64_t)i + J.index_base) >> 2;          // (index_base is a multiple of 4: word i & 3 is unchanged)
    if (o.q8) {
        const QParamsReg p = perch ? qparams_reg(J.r.qp8[c], 8) : t8;
        uint32_t rnd = 0;
        if (SR) {
            uint4 b = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)(j >> 32), id8, 0u), key);
            const uint32_t w[4] = {b.x, b.y, b.z, b.w};
            rnd = w[i & 3];
        }
        o.q8[i] = (int8_t)(quantize_code<SR>(v, p.inv, p.zp_u, 255.0f, rnd) - 128);
    }
    if (o.q16 || o.hi || o.lo) {
        const QParamsReg p = perch ? qparams_reg(J.r.qp16[c], 16) : t16;
        uint32_t rnd = 0;
        if (SR) {
            uint4 b = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)(j >> 32), id16, 0u), key);
            const uint32_t w[4] = {b.x, b.y, b.z, b.w};
            rnd = w[i & 3];
        }
        int s = quantize_code<SR>(v, p.inv, p.zp_u, 65535.0f, rnd) - 32768;
        if (o.q16) o.q16[i] = (int16_t)s;
        if (o.hi) o.hi[i] = (int8_t)(s >> 8);
        if (o.lo) o.lo[i] = (uint8_t)((s & 0xFF) ^ (o.lo_flip & 0xFF));
    }
}

// Four codes (low bytes of c[0..3]) into one word.
__device__ __forceinline__ uint32_t pack_bytes0(const uint32_t (&c)[4])
{
    return __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
}
// The top bytes of c[0..3] into one word.
__device__ __forceinline__ uint32_t pack_bytes3(const uint32_t (&c)[4])
{
    return __byte_perm(__byte_perm(c[0], c[1], 0x0073), __byte_perm(c[2], c[3], 0x0073), 0x5410);
}
// The second bytes of c[0..3] into one word.
__device__ __forceinline__ uint32_t pack_bytes1(const uint32_t (&c)[4])
{
    return __byte_perm(__byte_perm(c[0], c[1], 0x0051), __byte_perm(c[2], c[3], 0x0051), 0x5410);
}
// The third bytes of c[0..3] into one word.
__device__ __forceinline__ uint32_t pack_bytes2(const uint32_t (&c)[4])
{
    return __byte_perm(__byte_perm(c[0], c[1], 0x0062), __byte_perm(c[2], c[3], 0x0062), 0x5410);
}

// A warp's share of the row sums: lane l has the codes of vector j = j of lane 0 + l (ok: inside the tensor), sum their sum.
__device__ __forceinline__ void put_row_sum_group(const QuantOut &o, int64_t j, bool ok, int sum)          // rs_group > 0
{
    // (groups are aligned: the lane index is j mod 32)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        if (off < o.rs_group) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (ok && (threadIdx.x & (o.rs_group - 1)) == 0) {
        if (o.rs_shift >= 0) o.rowsum8[j >> o.rs_shift] = sum;
        else                 atomicAdd(o.rowsum8 + o.rs_div.div((int)j), sum);
    }
}
__device__ __forceinline__ void put_row_sum_wide(const QuantOut &o, int64_t j, int sum)                    // rs_group == 0
{
    const int row = o.rs_div.div((int)j), first = __shfl_sync(0xffffffffu, row, 0);
    const int all = __reduce_add_sync(0xffffffffu, sum), here = __reduce_add_sync(0xffffffffu, row == first ? sum : 0);
    if ((threadIdx.x & 31) == 0) {
        if (here) atomicAdd(o.rowsum8 + first, here);
        if (all != here) atomicAdd(o.rowsum8 + first + 1, all - here);
    }
}

// PERCH is a template parameter so that the per-tensor instance (the hot one: it is bound by its instruction
// count when rounding stochastically) carries none of the per-channel parameter handling.
// TOTALS: the instance that also leaves the per-channel totals (the others carry none of that work).
// J32: every Philox block index is below 2^32 (the first two rounds then have constant halves).  Four blocks per SM.
template <bool SR, int VEC, bool PERCH, bool TOTALS, bool J32>
__device__ __forceinline__ void quantize_body(const QuantJob &J, const PhiloxKeys &keys, int block, int blocks)
{
    const float *__restrict__ x = J.x;
    const int64_t n = J.n;
    const int cols = J.cols, smem_cols = J.smem_cols;
    const QuantOut &o = J.o;
    const uint32_t id8 = J.id8, id16 = J.id16;
    const uint64_t index_base = J.index_base;
    const bool want8 = o.q8 != nullptr, want16 = o.q16 || o.hi || o.lo;
    QParamsReg p8 = {0, 0}, p16 = {0, 0};
    if (!PERCH) resolve_range(J.r, want8, want16, block == 0, p8, p16);
    const QParamsReg t8 = p8, t16 = p16;
    if (VEC == 1) {
        const int64_t stride = (int64_t)blocks * kThreads;
        for (int64_t i = (int64_t)block * kThreads + threadIdx.x; i < n; i += stride) quantize_scalar<SR>(J, i, PERCH, t8, t16, keys);
        return;
    }
    // per channel: (1/scale, zero-point) of every channel once per block in shared memory (when the launcher
    // gave it room), instead of a division per element
    extern __shared__ float2 s_qp[];                         // [cols] for 8 bits, then [cols] for 16 bits
    const bool table = PERCH && smem_cols > 0;
    if (table) {
        for (int c = threadIdx.x; c < cols; c += kThreads) {
            if (want8)  { QParamsReg t = qparams_reg(J.r.qp8[c], 8);   s_qp[c] = make_float2(t.inv, t.zp_u); }
            if (want16) { QParamsReg t = qparams_reg(J.r.qp16[c], 16); s_qp[cols + c] = make_float2(t.inv, t.zp_u); }
        }
        __syncthreads();
    }
    if (!PERCH) {
        // the stochastic codes are taken in fixed point with 16 fraction bits: fold the factor into the parameters
        if (SR) { p8.inv *= 65536.0f; p8.zp_u *= 65536.0f; p16.inv *= 65536.0f; p16.zp_u *= 65536.0f; }
    }
    // both copies of a gradient under one tensor id: one Philox block serves the two (disjoint halves of each word)
    const bool one_block = want8 && want16 && id8 == id16;
    int cs8[4] = {0, 0, 0, 0};                               // this thread's channels: totals of the stored 8-bit codes
    int cs16[4] = {0, 0, 0, 0};                              // ... and of the stored 16-bit codes (fewer than 65536 per thread)
    const int64_t nv = n >> 2;
    const int64_t stride = (int64_t)blocks * kThreads * kUnroll;
    for (int64_t base = (int64_t)block * kThreads * kUnroll; base < nv; base += stride) {
        float4 v[kUnroll];
        bool ok[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            int64_t j = base + u * kThreads + threadIdx.x;
            ok[u] = j < nv;
            // nearest rounding follows a range scan of the same (large) tensor and is bound by HBM: evict-first loads;
            // the stochastic instance is bound by arithmetic and often finds the tail of its input in the L2
            if (ok[u]) v[u] = SR ? __ldg(reinterpret_cast<const float4 *>(x) + j) : __ldcs(reinterpret_cast<const float4 *>(x) + j);
        }
        int rs[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) rs[u] = 0;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (!ok[u]) continue;
            const int64_t j = base + u * kThreads + threadIdx.x;
            const float xs[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
            const int c0 = PERCH ? (int)((j << 2) % cols) : 0;
            uint4 b8 = make_uint4(0, 0, 0, 0), b16 = b8;
            if (SR) {
                // counter = the block's index in the whole tensor (a shard of a larger tensor starts at index_base)
                const uint64_t jb = (uint64_t)j + (index_base >> 2);
                if (want8) b8 = philox4x32_10(make_uint4((uint32_t)jb, J32 ? 0u : (uint32_t)(jb >> 32), id8, 0u), keys);
                if (want16) b16 = one_block ? b8 : philox4x32_10(make_uint4((uint32_t)jb, J32 ? 0u : (uint32_t)(jb >> 32), id16, 0u), keys);
            }
            if (want8) {
                const uint32_t r[4] = {b8.x, b8.y, b8.z, b8.w};
                uint32_t c[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (PERCH) {
                        if (table) { const float2 t = s_qp[c0 + e]; p8.inv = t.x; p8.zp_u = t.y; }
                        else p8 = qparams_reg(J.r.qp8[c0 + e], 8);
                        if (SR) { p8.inv *= 65536.0f; p8.zp_u *= 65536.0f; }
                    }
                    c[e] = SR ? quantize_sr8_byte2(xs[e], p8.inv, p8.zp_u, r[e])
                              : (uint32_t)quantize_code<SR>(xs[e], p8.inv, p8.zp_u, 255.0f, r[e]);
                }
                const uint32_t packed = SR ? pack_bytes2(c) : pack_bytes0(c) ^ 0x80808080u;       // stored = unsigned code - 128
                reinterpret_cast<uint32_t *>(o.q8)[j] = packed;
                if (o.rowsum8) rs[u] = __dp4a((int)packed, 0x01010101, 0);
                if (TOTALS && o.chansum8) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) cs8[e] = __dp4a((int)packed, 1 << (8 * e), cs8[e]);
                }
            }
            if (want16) {
                const uint32_t r[4] = {b16.x, b16.y, b16.z, b16.w};
                uint32_t c[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (PERCH) {
                        if (table) { const float2 t = s_qp[cols + c0 + e]; p16.inv = t.x; p16.zp_u = t.y; }
                        else p16 = qparams_reg(J.r.qp16[c0 + e], 16);
                        if (SR) { p16.inv *= 65536.0f; p16.zp_u *= 65536.0f; }
                    }
                    // (stochastic: the code sits in the upper half of the word, i.e. bytes 3 and 2)
                    c[e] = SR ? quantize_sr16_top_half(xs[e], p16.inv, p16.zp_u, r[e])
                              : (uint32_t)quantize_code<SR>(xs[e], p16.inv, p16.zp_u, 65535.0f, r[e]);
                }
                if (TOTALS && o.chansum16) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) cs16[e] += SR ? (int)c[e] >> 16 : (int)c[e] - 32768;
                }
                // stored = unsigned code - 32768: flip the top bit of every code (of every high byte)
                if (o.q16)
                    reinterpret_cast<uint2 *>(o.q16)[j] = make_uint2(__byte_perm(c[0], c[1], SR ? 0x7632 : 0x5410) ^ (SR ? 0u : 0x80008000u),
                                                                     __byte_perm(c[2], c[3], SR ? 0x7632 : 0x5410) ^ (SR ? 0u : 0x80008000u));
                if (SR && o.hi && o.lo) {
                    // (low, low, high, high) bytes of two codes each, then the two words: four permutes for both limbs
                    const uint32_t t01 = __byte_perm(c[0], c[1], 0x7362), t23 = __byte_perm(c[2], c[3], 0x7362);
                    reinterpret_cast<uint32_t *>(o.hi)[j] = __byte_perm(t01, t23, 0x7632);
                    reinterpret_cast<uint32_t *>(o.lo)[j] = __byte_perm(t01, t23, 0x5410) ^ o.lo_flip;
                } else {
                    if (o.hi) reinterpret_cast<uint32_t *>(o.hi)[j] = SR ? pack_bytes3(c) : pack_bytes1(c) ^ 0x80808080u;
                    if (o.lo) reinterpret_cast<uint32_t *>(o.lo)[j] = (SR ? pack_bytes2(c) : pack_bytes0(c)) ^ o.lo_flip;
                }
            }
        }
        if (o.rowsum8 && o.rs_group) {
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) put_row_sum_group(o, base + u * kThreads + threadIdx.x, ok[u], rs[u]);
        } else if (o.rowsum8) {
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) put_row_sum_wide(o, base + u * kThreads + threadIdx.x, rs[u]);
        }
    }
    if (block == 0 && threadIdx.x == 0)
        for (int64_t i = nv << 2; i < n; ++i) quantize_scalar<SR>(J, i, PERCH, t8, t16, keys);
    if (TOTALS && !PERCH && (o.chansum8 || o.chansum16)) {
        // (cols / 4 divides the block size and the grid stride: the thread's channels are 4 * (threadIdx.x mod cols / 4) ...)
        // (a block sees fewer than 65536 rows -- the launcher's rule -- so its totals fit int32)
        int *s_cs = reinterpret_cast<int *>(s_qp);           // [cols] 8-bit totals, then [cols] 16-bit ones
        for (int c = threadIdx.x; c < 2 * cols; c += kThreads) s_cs[c] = 0;
        __syncthreads();
        const int c0 = 4 * (threadIdx.x & ((cols >> 2) - 1));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (o.chansum8 && cs8[e]) atomicAdd(&s_cs[c0 + e], cs8[e]);
            if (o.chansum16) atomicAdd(&s_cs[cols + c0 + e], cs16[e]);
        }
        __syncthreads();
        for (int c = threadIdx.x; c < cols; c += kThreads) {
            if (o.chansum8 && s_cs[c]) atomicAdd(o.chansum8 + c, (unsigned long long)(long long)s_cs[c]);
            if (o.chansum16 && s_cs[cols + c]) atomicAdd(o.chansum16 + c, (unsigned long long)(long long)s_cs[cols + c]);
        }
    }
}

template <bool SR, int VEC, bool PERCH, bool TOTALS, bool J32>
__global__ void __launch_bounds__(kThreads, 4) quantize_kernel(const __grid_constant__ QuantJob J, const __grid_constant__ PhiloxKeys keys)
{
    pdl_wait();
    quantize_body<SR, VEC, PERCH, TOTALS, J32>(J, keys, (int)blockIdx.x, (int)gridDim.x);
}

// A gradient's 8-bit copy and the byte limbs of its 16-bit copy, nothing else (the usual bifurcation): the integer pipes bound
// it, so the general body's checks and 64-bit indices are left out (26 instructions per element instead of 39) and four blocks
// share an SM.  25.7 M elements with a range that is known: 50 -> 37 us (4.9 TB/s).  Not better: two vectors per thread with
// six blocks (41) or with the next two fetched ahead (41).
// ONE: both copies have one tensor id and share their Philox blocks.
template <bool ONE>
__global__ void __launch_bounds__(kThreads, 4) bifurcate_kernel(const __grid_constant__ QuantJob J, const __grid_constant__ PhiloxKeys keys)
{
    pdl_wait();
    QParamsReg p8 = {0, 0}, p16 = {0, 0};
    resolve_range(J.r, true, true, blockIdx.x == 0, p8, p16);
    const QParamsReg t8 = p8, t16 = p16;
    const float inv8 = p8.inv * 65536.0f, zp8 = p8.zp_u * 65536.0f, inv16 = p16.inv * 65536.0f, zp16 = p16.zp_u * 65536.0f;
    const float4 *const x = reinterpret_cast<const float4 *>(J.x);
    uint32_t *const q8 = reinterpret_cast<uint32_t *>(J.o.q8), *const hi = reinterpret_cast<uint32_t *>(J.o.hi), *const lo = reinterpret_cast<uint32_t *>(J.o.lo);
    const uint32_t nv = (uint32_t)(J.n >> 2), first = (uint32_t)(J.index_base >> 2);
    auto work = [&](const float4 &f, uint32_t j) {
        const float v[4] = {f.x, f.y, f.z, f.w};
        const uint4 r8 = philox4x32_10(make_uint4(j + first, 0u, J.id8, 0u), keys);
        const uint4 r16 = ONE ? r8 : philox4x32_10(make_uint4(j + first, 0u, J.id16, 0u), keys);
        uint32_t c16[4];
        const BifWords w = bifurcate4(v, inv8, zp8, inv16, zp16, r8, r16, J.o.lo_flip, c16);
        q8[j] = w.q8; hi[j] = w.hi; lo[j] = w.lo;
    };
    constexpr uint32_t kStep = kThreads * kUnroll;
    for (uint64_t base = (uint64_t)blockIdx.x * kStep; base < nv; base += (uint64_t)gridDim.x * kStep) {
        const uint32_t j = (uint32_t)base + threadIdx.x;
        if (base + kStep <= nv) {
            float4 v[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) v[u] = __ldg(x + (j + u * kThreads));
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) work(v[u], j + u * kThreads);
        } else {
#pragma unroll 1
            for (int u = 0; u < kUnroll; ++u)
                if (base + u * kThreads + threadIdx.x < nv) work(__ldg(x + (j + u * kThreads)), j + u * kThreads);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (int64_t i = (int64_t)nv << 2; i < J.n; ++i) quantize_scalar<true>(J, i, false, t8, t16, keys);
}

// A matrix [rows x cols] (cols a multiple of 4) quantised to 8 bits by nearest rounding, with the sums of its columns in pieces of
// its rows: block = (strip of 64 columns, piece), 16 rows at a time, four of them in flight per thread.
__device__ __forceinline__ void quantize_strip(const QuantJob &J, const StripJob &S, int block)
{
    QParamsReg p8 = {0, 0}, none = {0, 0};
    resolve_range(J.r, true, false, block == 0, p8, none);
    const int cv = J.cols >> 2, strips = (cv + 15) >> 4, strip = block % strips, piece = block / strips;
    const int v = strip * 16 + (threadIdx.x & 15), ty = threadIdx.x >> 4;
    const int64_t r_begin = S.rows * piece / S.pieces, r_end = S.rows * (piece + 1) / S.pieces;
    int acc[4] = {0, 0, 0, 0};
    for (int64_t r = r_begin + ty; r < r_end && v < cv; r += 16 * kUnroll) {
        float4 f[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            if (r + 16 * u < r_end) f[u] = __ldcs(reinterpret_cast<const float4 *>(J.x) + (r + 16 * u) * cv + v);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (r + 16 * u >= r_end) break;
            const float e4[4] = {f[u].x, f[u].y, f[u].z, f[u].w};
            uint32_t c[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                c[e] = (uint32_t)quantize_code<false>(e4[e], p8.inv, p8.zp_u, 255.0f, 0u);
                acc[e] += (int)c[e] - 128;
            }
            reinterpret_cast<uint32_t *>(J.o.q8)[(r + 16 * u) * cv + v] = pack_bytes0(c) ^ 0x80808080u;
        }
    }
    __shared__ int s_acc[kThreads / 32][64];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 16);              // (a warp holds two rows)
        if ((threadIdx.x & 31) < 16) s_acc[threadIdx.x >> 5][(threadIdx.x & 15) * 4 + e] = acc[e];
    }
    __syncthreads();
    const int col = strip * 64 + (int)threadIdx.x;
    if (threadIdx.x < 64 && col < J.cols) {
        int sum = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) sum += s_acc[w][threadIdx.x];
        S.col_sums[(int64_t)piece * J.cols + col] = sum;
    }
}

// A layer's weights (the first b_blocks blocks; with the sums of their columns when S.col_sums is given) and activation in one
// launch; nearest rounding, per tensor.
template <bool TOTALS>
__global__ void __launch_bounds__(kThreads) quantize_pair_kernel(const __grid_constant__ QuantJob a, const __grid_constant__ QuantJob b, int b_blocks,
                                                                 const __grid_constant__ StripJob S)
{
    pdl_wait();
    const PhiloxKeys none = {};
    if ((int)blockIdx.x >= b_blocks) quantize_body<false, 4, false, TOTALS, false>(a, none, (int)blockIdx.x - b_blocks, (int)gridDim.x - b_blocks);
    else if (!TOTALS && S.col_sums)  quantize_strip(b, S, (int)blockIdx.x);
    else                             quantize_body<false, 4, false, false, false>(b, none, (int)blockIdx.x, b_blocks);
}

// A layer's activation and weights, each of at most kSmallElems elements: range, codes and their sums in one launch.  A tensor is a
// cluster of eight CTAs that holds it in registers (two float4 a thread); their ranges meet in distributed shared memory.  What the
// sums are added to is cleared before the cluster's barrier.  (A scan and a quantiser are two launches of 2 and 4 us for such tensors,
// of which the reading is a fraction: the layer of 64 x 256 -> 128 33.4 -> 32.3 us a step.  Not for larger tensors, whose bytes eight
// SMs take too long to read: weights of 147 K elements 6.7 us against 6.4, the layer of 512 x 512 -> 512 53.0 against 51.9.)
// colsum [cols]: column sums, 32 bits, added to the first of `pieces` rows; o.chansum8: 64 bits.
struct SmallOperand { const float *x; int n4, cols; QuantOut o; qbp_qparams *qp; int32_t *colsum; int pieces; };
struct SmallJob { SmallOperand op[2]; ZeroJobs zero; };
constexpr int kSmallCtas = 8, kSmallThreads = 1024, kSmallVecs = 2, kSmallMaxCols = 8192;
constexpr int64_t kSmallElems = 4ll * kSmallCtas * kSmallThreads * kSmallVecs;
__device__ __forceinline__ void quantize_small_body(const SmallJob &J)
{
    extern __shared__ int s_cols[];                          // [cols] when column sums or totals are wanted
    __shared__ float2 s_range;
    const SmallOperand &op = J.op[blockIdx.x / kSmallCtas];
    const QuantOut &o = op.o;
    const int rank = (int)cluster_ctarank(), t = rank * kSmallThreads + (int)threadIdx.x;
    constexpr int kAll = kSmallCtas * kSmallThreads;
    const bool columns = op.colsum || o.chansum8;
    float4 v[kSmallVecs];
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int k = 0; k < kSmallVecs; ++k)
        if (t + k * kAll < op.n4) v[k] = __ldg(reinterpret_cast<const float4 *>(op.x) + t + k * kAll);
    if (blockIdx.x < kSmallCtas) run_zero_jobs(J.zero, t, kAll);
    if (o.rowsum8 && o.rs_shift < 0)
        for (int i = t; i < op.n4 / (op.cols >> 2); i += kAll) o.rowsum8[i] = 0;
    if (op.colsum)
        for (int i = t; i < op.pieces * op.cols; i += kAll) op.colsum[i] = 0;
    if (o.chansum8)
        for (int i = t; i < op.cols; i += kAll) o.chansum8[i] = 0;
    if (columns)
        for (int i = threadIdx.x; i < op.cols; i += kSmallThreads) s_cols[i] = 0;
#pragma unroll
    for (int k = 0; k < kSmallVecs; ++k)
        if (t + k * kAll < op.n4) {
            lo = fminf(fminf(lo, fminf(v[k].x, v[k].y)), fminf(v[k].z, v[k].w));
            hi = fmaxf(fmaxf(hi, fmaxf(v[k].x, v[k].y)), fmaxf(v[k].z, v[k].w));
        }
    const float2 mine = block_min_max(lo, hi);
    if (threadIdx.x == 0) s_range = mine;
    __syncthreads();
    cluster_sync_all();
    {
        const int lane = threadIdx.x & 31;
        float2 r = make_float2(INFINITY, -INFINITY);
        if (lane < kSmallCtas) {
            const uint32_t at = map_to_cta(&s_range, (uint32_t)lane);
            asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(at) : "memory");
        }
        lo = warp_min(r.x); hi = warp_max(r.y);
    }
    // (a CTA's range may be read until all have read it: the wait for this is at the end)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const qbp_qparams qp = make_qparams(lo, hi, 8);
    if (t == 0) *op.qp = qp;
    const QParamsReg p = qparams_reg(qp, 8);
    const int cv = op.cols >> 2;
#pragma unroll
    for (int k = 0; k < kSmallVecs; ++k) {
        const int j = t + k * kAll;
        if (j - (int)(threadIdx.x & 31) >= op.n4) break;     // (the warp's)
        const bool ok = j < op.n4;
        int sum = 0;
        if (ok) {
            const float e4[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
            uint32_t c[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) c[e] = (uint32_t)quantize_code<false>(e4[e], p.inv, p.zp_u, 255.0f, 0u);
            const uint32_t packed = pack_bytes0(c) ^ 0x80808080u;
            reinterpret_cast<uint32_t *>(o.q8)[j] = packed;
            sum = __dp4a((int)packed, 0x01010101, 0);
            if (columns) {
                const int c0 = (j % cv) * 4;
#pragma unroll
                for (int e = 0; e < 4; ++e) atomicAdd(&s_cols[c0 + e], (int)c[e] - 128);
            }
        }
        if (o.rowsum8) { if (o.rs_group) put_row_sum_group(o, j, ok, sum); else put_row_sum_wide(o, j, sum); }
    }
    if (columns) {
        __syncthreads();
        for (int i = threadIdx.x; i < op.cols; i += kSmallThreads) {
            const int sum = s_cols[i];
            if (sum && op.colsum) atomicAdd(op.colsum + i, sum);
            if (sum && o.chansum8) atomicAdd(o.chansum8 + i, (unsigned long long)(long long)sum);
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads, 1) operands_prep_kernel(const __grid_constant__ SmallJob J)
{
    pdl_wait();
    quantize_small_body(J);
}

// Regions cleared between two kernels (see launch_clear).
__global__ void __launch_bounds__(kThreads) clear_kernel(const __grid_constant__ ZeroJobs zero)
{
    pdl_wait();
    run_zero_jobs(zero, (int64_t)blockIdx.x * kThreads + threadIdx.x, (int64_t)gridDim.x * kThreads);
}

// The sums of up to eight code tensors in a launch of their own (see qbp_sums.cuh).
template <bool BESIDE>
__global__ void __launch_bounds__(kSumThreads) code_sums_kernel(const __grid_constant__ SumJobs J)
{
    if (!BESIDE) pdl_trigger();          // (see launch(); without a look at a parameter, which cost every small product 0.3 us)
    pdl_wait();
    if (BESIDE) pdl_trigger();
    run_zero_jobs(J.zero, (int64_t)blockIdx.x * kSumThreads + threadIdx.x, (int64_t)gridDim.x * kSumThreads);
    code_sums_block(J, (int)blockIdx.x);
}

// ----------------------------------------------------------------- launchers
// Pieces of the rows in a column sum: enough blocks for four per SM, at least 128 rows each, at most 16 pieces (the reader adds
// them up) -- but at most 2^22 rows each, so that a piece fits int32 (255 * 2^22 < 2^31).
int sum_pieces(int64_t rows, int64_t cols)
{
    const int64_t strips = (cols + 127) / 128;
    int64_t p = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(4ll * sm_count() / strips, 16), rows / 128));
    return (int)std::max<int64_t>(p, (rows >> 22) + 1);
}

// The same for the long edges of N images (always added up by atomics): some 256 positions of the longest edge each, at most 64; of
// short edges up to four, as long as a block of `high` rows has all of its piece in flight at once.  (256 images of 56 x 56: with
// 16 pieces of 896 positions the layer took 530 us, with 56 526; of 14 x 14, 256 channels: 14 pieces 250.5, 28 of them 254.)
static int edge_pieces(int64_t rows, int H, int W, int high)
{
    const int64_t longest = rows / ((int64_t)H * W) * std::max(H, W);
    const int64_t p = std::max<int64_t>(std::min<int64_t>(64, longest / 256), std::min<int64_t>(4, longest / (4 * high)));
    return (int)std::max<int64_t>(std::max<int64_t>(1, p), (longest >> 22) + 1);
}
// ... and for their corners: one position per image.
static int corner_pieces(int64_t images)
{
    return (int)std::max<int64_t>(std::max<int64_t>(1, std::min<int64_t>(64, images / 256)), (images >> 22) + 1);
}

int fill_sum_jobs(const SumJob *jobs, int count, SumJobs &J, int *blocks)
{
    // (sums over rows first: their blocks run longest; those along rows fill the machine behind them)
    int first = 0, order[kMaxSumJobs], n = 0;
    for (int pass = 0; pass < 2; ++pass)
        for (int i = 0; i < count; ++i)
            if ((jobs[i].kind == kSumRows) == (pass == 1)) order[n++] = i;
    for (int i = 0; i < count; ++i) {
        const SumJob &s = jobs[order[i]];
        if (s.cols % 16 || !aligned16(s.q)) return fail(QBP_ERR_INVALID_ARG, "code sums need 16-byte aligned rows (cols %% 16 == 0)");
        SumJobDev &j = J.j[i];
        j.q = static_cast<const uint8_t *>(s.q); j.rows = s.rows; j.cols = (int)s.cols; j.kind = s.kind; j.out = s.out; j.out64 = s.out64;
        j.flip = s.is_signed ? 0u : 0x80808080u; j.first = first; j.G = 1; j.pieces = j.corner_pieces = 1; j.H = s.H; j.W = s.W;
        while ((16 << j.lg_log2) < s.cols && j.lg_log2 < 3) ++j.lg_log2;
        const int strips = (int)((s.cols / 16 + (1 << j.lg_log2) - 1) >> j.lg_log2);
        if (s.kind == kSumRows) {
            while (j.G < 32 && j.G < s.cols / 16) j.G <<= 1;
            const int64_t groups = kSumThreads / j.G;
            j.blocks = (int)std::max<int64_t>(1, std::min<int64_t>((s.rows + groups - 1) / groups, 4ll * sm_count()));
        } else {
            j.pieces = s.kind == kSumEdges ? edge_pieces(s.rows, s.H, s.W, kSumThreads >> j.lg_log2) : sum_pieces(s.rows, s.cols);
            // added up by atomics, nobody reads the pieces one by one: as many blocks as the rows give work to (the sums of
            // 200704 x 128 codes: 31 us with 16 pieces, 16 so)
            if (s.out64 && s.kind == kSumCols) j.pieces = (int)std::max<int64_t>(j.pieces, std::min<int64_t>(4ll * sm_count() / strips, s.rows / 128));
            if (s.kind == kSumEdges) j.corner_pieces = corner_pieces(s.rows / ((int64_t)s.H * s.W));
            j.blocks = strips * (s.kind == kSumCols ? j.pieces : 4 * (j.pieces + j.corner_pieces));
        }
        first += j.blocks;
    }
    J.count = count;
    *blocks = first;
    return QBP_OK;
}

int launch_clear(void *p, int64_t words, cudaStream_t st)
{
    if (words <= 0) return QBP_OK;
    ZeroJobs zero{};
    if (int rc = zero.add(p, words)) return rc;
    const int grid = (int)std::min<int64_t>(sm_count(), (words + kThreads - 1) / kThreads);
    QBP_TRACE_BEGIN(st);
    launch(clear_kernel, grid, kThreads, 0, st, zero);
    QBP_LAUNCH_OK("clear_kernel");
    return QBP_OK;
}

int launch_code_sums(const SumJob *jobs, int count, cudaStream_t st, const ZeroJobs &zero, bool *beside)
{
    if (beside) *beside = false;
    if (count == 0) {
        for (int k = 0; k < zero.count; ++k)
            if (int rc = launch_clear(zero.p[k], zero.words[k], st)) return rc;
        return QBP_OK;
    }
    SumJobs J{};
    int blocks = 0;
    if (int rc = fill_sum_jobs(jobs, count, J, &blocks)) return rc;
    J.zero = zero;
    int64_t bytes = 0;
    for (int i = 0; i < count; ++i) bytes += jobs[i].rows * jobs[i].cols;
    const bool ahead = beside && bytes >= kSumsBesideMin && bytes <= kSumsBesideMax;
    if (beside) *beside = ahead;
    QBP_TRACE_BEGIN(st);
    if (ahead) launch(code_sums_kernel<true>, blocks, kSumThreads, 0, st, J);
    else       launch(code_sums_kernel<false>, blocks, kSumThreads, 0, st, J);
    QBP_LAUNCH_OK("code_sums_kernel");
    return QBP_OK;
}

// One wave: `bps` resident blocks per SM (the kernel's occupancy), never more blocks than work groups.
static int grid_for(int bps, int64_t n_groups)
{
    int64_t want = (int64_t)sm_count() * bps;
    int64_t g = n_groups < want ? n_groups : want;
    return (int)(g < 1 ? 1 : g);
}

// Blocks of the scan of one tensor: one wave at most.
static int scan_blocks(int64_t n, bool vec)
{
    if (n <= 0) return 0;
    const int64_t per_block = (int64_t)kThreads * kRangeUnroll * (vec ? 4 : 1);
    const int g = grid_for(vec ? blocks_per_sm<range_partial_kernel<4>>(kThreads) : blocks_per_sm<range_partial_kernel<1>>(kThreads), (n + per_block - 1) / per_block);
    return std::min(g, kMaxParts);
}

// Leaves *nparts (min, max) pairs of the n elements at `partials`.
static int launch_range(const float *x, int64_t n, float2 *partials, int *nparts, cudaStream_t st, const ZeroJobs &zero = ZeroJobs{},
                        bool nearest = false)
{
    const bool vec = aligned16(x);
    const ScanJob a{x, n, partials, scan_blocks(n, vec), nearest ? 1 : 0}, none{};
    *nparts = a.blocks;
    if (a.blocks == 0) return QBP_OK;
    QBP_TRACE_BEGIN(st);
    if (vec) launch(range_partial_kernel<4>, a.blocks, kThreads, 0, st, a, none, zero);
    else     launch(range_partial_kernel<1>, a.blocks, kThreads, 0, st, a, none, zero);
    QBP_LAUNCH_OK("range_partial_kernel");
    return QBP_OK;
}

// The per-tensor scan for callers in other files.
size_t range_scan_ws_bytes() { return align_up(sizeof(float2) * kMaxParts, 256); }
int range_scan(const float *x, int64_t n, void *ws, size_t ws_bytes, int *nparts, cudaStream_t st)
{
    if (!ws || ws_bytes < range_scan_ws_bytes()) return fail(QBP_ERR_WORKSPACE, "range scan: workspace too small");
    return launch_range(x, n, static_cast<float2 *>(ws), nparts, st);
}

static int launch_empty_qparams(qbp_qparams *qp8, qbp_qparams *qp16, cudaStream_t st)
{
    QBP_TRACE_BEGIN(st);
    launch(empty_qparams_kernel, 1, 1, 0, st, qp8, qp16);
    QBP_LAUNCH_OK("empty_qparams_kernel");
    return QBP_OK;
}

static int launch_chan_range(const float *x, int64_t rows, int64_t cols, int bits, float *part_lo, float *part_hi,
                             qbp_qparams *qp, cudaStream_t st)
{
    const bool v4 = aligned16(x) && cols % 4 == 0;
    ScanGeom g = scan_geom(rows, cols, aligned16(x), v4 ? blocks_per_sm<chan_range_partial_kernel<4>>(kScanThreads)
                                                        : blocks_per_sm<chan_range_partial_kernel<1>>(kScanThreads));
    int nparts = 0;
    if (rows > 0) {
        nparts = g.nbx;
        dim3 grid(g.nbx, g.slabs);
        QBP_TRACE_BEGIN(st);
        if (g.vec == 4) launch(chan_range_partial_kernel<4>, grid, kScanThreads, 0, st, x, rows, (int)cols, g.tw, part_lo, part_hi);
        else            launch(chan_range_partial_kernel<1>, grid, kScanThreads, 0, st, x, rows, (int)cols, g.tw, part_lo, part_hi);
        QBP_LAUNCH_OK("chan_range_partial_kernel");
    }
    QBP_TRACE_BEGIN(st);
    launch(chan_range_finalize_kernel, (int)((cols + 7) / 8), kThreads, 0, st, part_lo, part_hi, nparts, (int)cols, bits, qp);
    QBP_LAUNCH_OK("chan_range_finalize_kernel");
    return QBP_OK;
}

// Whether a tensor takes the vector path.
static bool quant_vec(const float *x, int64_t cols, int perch, const QuantOut &o)
{
    return aligned16(x) && (!perch || cols % 4 == 0) && (!o.q8 || ((uintptr_t)o.q8 & 3) == 0) && (!o.q16 || ((uintptr_t)o.q16 & 7) == 0) &&
           (!o.hi || ((uintptr_t)o.hi & 3) == 0) && (!o.lo || ((uintptr_t)o.lo & 3) == 0);
}

static int launch_quantize(const float *x, int64_t n, int64_t cols, int perch, int rounding, const RangeSrc &r, uint32_t id8,
                           uint32_t id16, uint64_t seed, const QuantOut &o, cudaStream_t st, uint64_t index_base = 0)
{
    if (n == 0) return QBP_OK;
    const bool vec = quant_vec(x, cols, perch, o);
    if (o.rowsum8 && !vec) return fail(QBP_ERR_INVALID_ARG, "quantize: fused row sums need the vector path");
    const int64_t per_block = (int64_t)kThreads * (vec ? 4 * kUnroll : 1);
    const bool sr = rounding == QBP_ROUND_STOCHASTIC;
    const PhiloxKeys key = philox_keys_host(seed);
    // per-channel parameter table: 2 x cols x 8 bytes of dynamic shared memory when that stays within 32 KB
    const int smem_cols = (perch && vec && cols <= 2048) ? (int)cols : 0;
    const bool totals = o.chansum8 || o.chansum16;
    // (fewer than 2^22 rows: with a grid of at least one block per SM, or one block per 1024 vectors, a block sees
    // fewer than 65536 of them, and its int32 totals of 16-bit codes cannot overflow)
    if (totals && !(vec && !perch && quantizer_totals_supported(cols) && n / cols < (1ll << 22)))
        return fail(QBP_ERR_INVALID_ARG, "quantize: per-channel totals need the vector path and cols / 4 a power of two <= %d", kThreads);
    const size_t smem = !vec ? 0 : totals ? (size_t)cols * 2 * sizeof(int) : (size_t)smem_cols * 2 * sizeof(float2);
    const int64_t groups = (n + per_block - 1) / per_block;
    const QuantJob J{x, n, (int)cols, r, id8, id16, o, smem_cols, index_base};
    const bool j32 = (((uint64_t)n + index_base) >> 2) < (1ull << 32) - 1;
#define QBP_QUANT3(SR_, VEC_, PC_, TOT_, J32_)                                                                          \
    do {                                                                                                                \
        const int grid = grid_for(blocks_per_sm<quantize_kernel<SR_, VEC_, PC_, TOT_, J32_>>(kThreads), groups);        \
        QBP_TRACE_BEGIN(st);                                                                                            \
        launch(quantize_kernel<SR_, VEC_, PC_, TOT_, J32_>, grid, kThreads, smem, st, J, key);                          \
    } while (0)
#define QBP_QUANT(PC_, TOT_)                                                                                            \
    do {                                                                                                                \
        if (sr) { if (j32) QBP_QUANT3(true, 4, PC_, TOT_, true); else QBP_QUANT3(true, 4, PC_, TOT_, false); }          \
        else QBP_QUANT3(false, 4, PC_, TOT_, false);                                                                    \
    } while (0)
    if (sr && vec && !perch && !totals && j32 && o.q8 && o.hi && o.lo && !o.q16 && !o.rowsum8) {
        QBP_TRACE_BEGIN(st);
        if (id8 == id16) launch(bifurcate_kernel<true>, grid_for(blocks_per_sm<bifurcate_kernel<true>>(kThreads), groups), kThreads, 0, st, J, key);
        else             launch(bifurcate_kernel<false>, grid_for(blocks_per_sm<bifurcate_kernel<false>>(kThreads), groups), kThreads, 0, st, J, key);
        QBP_LAUNCH_OK("bifurcate_kernel");
        return QBP_OK;
    }
    if (totals) QBP_QUANT(false, true);           // (vector path, per tensor: checked above)
    else if (vec && perch) QBP_QUANT(true, false);
    else if (vec) QBP_QUANT(false, false);
    else if (sr) { if (perch) QBP_QUANT3(true, 1, true, false, false); else QBP_QUANT3(true, 1, false, false, false); }
    else         { if (perch) QBP_QUANT3(false, 1, true, false, false); else QBP_QUANT3(false, 1, false, false, false); }
#undef QBP_QUANT3
#undef QBP_QUANT
    QBP_LAUNCH_OK("quantize_kernel");
    return QBP_OK;
}

// Whether the quantising kernel itself can emit the row sums of its 8-bit codes: per-tensor, 16-byte aligned tensors whose rows are
// 4, 8, ..., 128 elements (a row is then a power-of-two group of lanes of one warp) or, where the sums are cleared beforehand
// (`add`), a multiple of 16 (added in pieces).  Fills the record in.
static bool fuse_rowsums(const float *x, int64_t n, int64_t cols, bool add, int32_t *row_sums, QuantOut &o)
{
    const int64_t v = cols / 4, group = std::min<int64_t>(v & -v, 32);
    const bool whole = group == v;
    if (cols % 4 || v < 1 || (!whole && !(add && cols % 16 == 0 && n / 4 < (1ll << 31) - 2048)) || !aligned16(x) || ((uintptr_t)o.q8 & 3) ||
        (o.q16 && ((uintptr_t)o.q16 & 7)) || (o.hi && ((uintptr_t)o.hi & 3)) || (o.lo && ((uintptr_t)o.lo & 3)))
        return false;
    o.rowsum8 = row_sums; o.rs_group = !whole && v >= 32 && group < 32 ? 0 : (int)group;
    o.rs_shift = -1; o.rs_div = FastDiv{};
    if (whole) o.rs_shift = 31 - __builtin_clz((unsigned)v); else o.rs_div = make_fastdiv((int)v);
    return true;
}

// Row / column sums of stored codes, complete.
int launch_rowsum(const void *q, bool is_signed, int64_t rows, int64_t cols, int32_t *sums, cudaStream_t st)
{
    const SumJob job{q, rows, cols, kSumRows, is_signed ? 1 : 0, sums};
    return rows == 0 ? QBP_OK : launch_code_sums(&job, 1, st);
}
int launch_colsum(const void *q, bool is_signed, int64_t rows, int64_t cols, int64_t *sums, cudaStream_t st, bool cleared)
{
    if (cols % 16 || !aligned16(q)) return fail(QBP_ERR_INVALID_ARG, "column sums need cols %% 16 == 0 and 16-byte aligned codes");
    const SumJob job{q, rows, cols, kSumCols, is_signed ? 1 : 0, nullptr, 0, 0, sums};
    if (!cleared)
        if (int rc = launch_clear(sums, 2 * cols, st)) return rc;
    return rows == 0 ? QBP_OK : launch_code_sums(&job, 1, st);
}

static int check_common(const float *x, int64_t rows, int64_t cols, int granularity, int rounding,
                        const qbp_qparams *qp_out)
{
    if (rows < 0 || cols <= 0) return fail(QBP_ERR_INVALID_ARG, "quantize: rows must be >= 0 and cols > 0");
    if (granularity != QBP_PER_TENSOR && granularity != QBP_PER_CHANNEL)
        return fail(QBP_ERR_INVALID_ARG, "quantize: granularity must be QBP_PER_TENSOR or QBP_PER_CHANNEL");
    if (rounding != QBP_ROUND_NEAREST && rounding != QBP_ROUND_STOCHASTIC)
        return fail(QBP_ERR_INVALID_ARG, "quantize: rounding must be QBP_ROUND_NEAREST or QBP_ROUND_STOCHASTIC");
    if (!qp_out) return fail(QBP_ERR_INVALID_ARG, "quantize: qp_out is NULL");
    if (!x && rows * cols > 0) return fail(QBP_ERR_INVALID_ARG, "quantize: x is NULL");
    if (((uintptr_t)x & 3) != 0) return fail(QBP_ERR_INVALID_ARG, "quantize: x is not 4-byte aligned");
    return QBP_OK;
}

static size_t quant_ws_bytes(int64_t cols, int granularity)
{
    if (granularity == QBP_PER_CHANNEL) return 2 * align_up(sizeof(float) * kScanMaxStrips * (size_t)cols, 256) + 256;
    return align_up(sizeof(float2) * kMaxParts, 256) + 256;
}

// Shared body of the 8- and 16-bit entry points.
static int quantize_any(int bits, const float *x, int64_t rows, int64_t cols, int granularity, int rounding,
                        uint64_t seed, uint32_t tensor_id, const qbp_qparams *range_in, const QuantOut &o,
                        qbp_qparams *qp_out, void *ws, size_t ws_bytes, cudaStream_t st)
{
    int rc = check_common(x, rows, cols, granularity, rounding, qp_out);
    if (rc) return rc;
    const int perch = granularity == QBP_PER_CHANNEL;
    const int64_t n = rows * cols;
    qbp_qparams *qp8 = bits == 8 ? qp_out : nullptr, *qp16 = bits == 16 ? qp_out : nullptr;
    RangeSrc r{nullptr, 0, nullptr, qp8, qp16};
    if (range_in && (perch || n == 0)) {
        const int count = perch ? (int)cols : 1;
        QBP_TRACE_BEGIN(st);
        launch(qparams_from_range_kernel, (count + 255) / 256, 256, 0, st, range_in, count, bits, qp_out);
        QBP_LAUNCH_OK("qparams_from_range_kernel");
    } else if (range_in) {
        r.given = range_in;
    } else {
        if (!ws || ws_bytes < quant_ws_bytes(cols, granularity))
            return fail(QBP_ERR_WORKSPACE, "quantize: workspace of %zu bytes needed, %zu given",
                        quant_ws_bytes(cols, granularity), ws_bytes);
        WsCarver w(ws, ws_bytes);
        if (perch) {
            float *plo = w.take<float>((size_t)kScanMaxStrips * cols);
            float *phi = w.take<float>((size_t)kScanMaxStrips * cols);
            rc = launch_chan_range(x, rows, cols, bits, plo, phi, qp_out, st);
        } else if (n == 0) {
            rc = launch_empty_qparams(qp8, qp16, st);
        } else {
            float2 *parts = w.take<float2>(kMaxParts);
            rc = launch_range(x, n, parts, &r.nparts, st, ZeroJobs{}, rounding == QBP_ROUND_NEAREST);
            r.parts = parts;
        }
        if (rc) return rc;
    }
    return launch_quantize(x, n, cols, perch, rounding, r, tensor_id, tensor_id, seed, o, st);
}

// ------------------------------------------------- built-in scratch (no allocation)
// Scratch of qbp_quantize_s8_static: lives in the library's device image, so every GPU that loads the
// library holds these bytes until the process exits.  Sized for the per-channel range scan of
// QBP_STATIC_MAX_CHANNELS channels (two float partial tables of kScanMaxStrips rows), which also covers the
// per-tensor scan.  Host code must not pass this name to a kernel: it is resolved per device below.
constexpr size_t kStaticScratchBytes = 2 * sizeof(float) * (size_t)kScanMaxStrips * QBP_STATIC_MAX_CHANNELS + 256;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

static std::mutex g_static_mu;
static void *g_static_ptr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device, looked up once per device.
static int static_scratch_address(void **out)
{
    int dev = -1;
    QBP_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(QBP_ERR_CUDA, "quantize_s8_static: device ordinal %d not supported", dev);
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void *p = nullptr;
        QBP_CUDA_OK(cudaGetSymbolAddress(&p, g_static_scratch));
        if (!p) return fail(QBP_ERR_CUDA, "quantize_s8_static: the built-in scratch has no device address");
        g_static_ptr[dev] = p;
    }
    *out = g_static_ptr[dev];
    return QBP_OK;
}

// The quantising half of the bifurcation.
static int bifurcate_tail(const float *g, int64_t rows, int64_t cols, uint64_t seed, uint32_t tensor_id8,
                          uint32_t tensor_id16, int8_t *q8, const RangeSrc &r, int32_t *row_sums8, int8_t *hi, uint8_t *lo,
                          cudaStream_t st, uint64_t index_base = 0, int64_t *tot16 = nullptr, bool lo_signed = false)
{
    QuantOut o = quant_out(q8, nullptr, hi, lo, lo_signed ? 0x80808080u : 0u);
    if (tot16 && rows * cols > 0)                         // (cleared by the caller, who asked quantizer_totals_supported(cols) first)
        o.chansum16 = reinterpret_cast<unsigned long long *>(tot16);
    const bool fused = row_sums8 && rows * cols > 0 && fuse_rowsums(g, rows * cols, cols, false, row_sums8, o);
    int rc = launch_quantize(g, rows * cols, cols, 0, QBP_ROUND_STOCHASTIC, r, tensor_id8, tensor_id16, seed, o, st, index_base);
    if (rc) return rc;
    if (row_sums8 && !fused) return launch_rowsum(q8, true, rows, cols, row_sums8, st);
    return QBP_OK;
}

// Bifurcation of a gradient whose range partials (min, max per block) were left by the kernel that wrote it.
int bifurcate_with_range_partials(const float *g, int64_t rows, int64_t cols, uint64_t seed, uint32_t tensor_id8,
                                  uint32_t tensor_id16, int8_t *q8, qbp_qparams *qp8, int32_t *row_sums8, int8_t *hi,
                                  uint8_t *lo, qbp_qparams *qp16, const float2 *partials, int nparts, cudaStream_t st,
                                  int64_t *tot16, bool lo_signed)
{
    return bifurcate_tail(g, rows, cols, seed, tensor_id8, tensor_id16, q8, RangeSrc{partials, nparts, nullptr, qp8, qp16}, row_sums8,
                          hi, lo, st, 0, tot16, lo_signed);
}

bool quantizer_totals_supported(int64_t cols)
{
    return cols % 4 == 0 && cols / 4 <= kThreads && ((cols / 4) & (cols / 4 - 1)) == 0;
}

size_t quantize_operands_ws_bytes() { return 2 * align_up(sizeof(float2) * kMaxParts, 256); }
int quantize_operands(QuantOperand *x, QuantOperand *w, int *status, void *ws, size_t ws_bytes, cudaStream_t st, bool add_rows, void *clear, int64_t clear_words)
{
    if (!ws || ws_bytes < quantize_operands_ws_bytes()) return fail(QBP_ERR_WORKSPACE, "quantize: workspace too small");
    WsCarver c(ws, ws_bytes);
    QuantOperand *ops[2] = {x, w};
    QuantOut o[2];
    float2 *parts[2];
    bool vec[2] = {true, true};
    // (the status word, the caller's, the activation's or the weights' totals, either operand's row sums in pieces)
    ZeroJobs zero{};
    int rc = status ? zero.add(status, 1) : QBP_OK;
    if (rc || (rc = zero.add(clear, clear_words))) return rc;
    // small tensors: everything in one launch
    {
        SmallJob J{};
        J.zero = zero;
        bool small = x != nullptr;
        int count = 0, cols = 0;
        for (int i = 0; i < 2 && small; ++i) {
            if (!ops[i]) continue;
            QuantOperand &op = *ops[i];
            if ((rc = check_common(op.v, op.rows, op.cols, QBP_PER_TENSOR, QBP_ROUND_NEAREST, op.qp))) return rc;
            SmallOperand &s = J.op[count++];
            const int64_t n = op.rows * op.cols;
            s = SmallOperand{op.v, (int)(n / 4), (int)op.cols, quant_out(op.q, nullptr, nullptr, nullptr), op.qp, op.col_sums, 0};
            small = n > 0 && n <= kSmallElems && op.cols % 4 == 0 && op.cols <= kSmallMaxCols && quant_vec(op.v, op.cols, 0, s.o) &&
                    (!op.row_sums || fuse_rowsums(op.v, n, op.cols, true, op.row_sums, s.o));
            if (op.col_sums) s.pieces = sum_pieces(op.rows, op.cols);
            if (op.tot && i == 0) s.o.chansum8 = reinterpret_cast<unsigned long long *>(op.tot);
            else if (op.tot && (rc = J.zero.add(op.tot, 2 * op.cols))) return rc;
            if (s.colsum || s.o.chansum8) cols = std::max(cols, s.cols);
        }
        if (small) {
            for (int i = 0; i < 2; ++i)
                if (ops[i]) { ops[i]->row_sums_left = ops[i]->row_sums != nullptr; ops[i]->tot_left = ops[i]->tot && i == 0; ops[i]->col_sums_left = ops[i]->col_sums != nullptr; }
            QBP_TRACE_BEGIN(st);
            launch(operands_prep_kernel, count * kSmallCtas, kSmallThreads, (size_t)cols * sizeof(int), st, J);
            QBP_LAUNCH_OK("operands_prep_kernel");
            return QBP_OK;
        }
    }
    // The weights' column sums beside their codes: of at most 3 M elements, in blocks of at most 64 K (a launch and its reading of the
    // codes less: 3 us; 64 x 4080 -> 4080, whose 16.6 M the strips read at two thirds of the bandwidth, 158 -> 165 us).  Where they are
    // not taken, a launch for code sums follows anyway, and takes the activation's rows as well.
    StripJob S{w->rows, sum_pieces(w->rows, w->cols), nullptr};
    const int64_t strip_blocks = (w->cols + 63) / 64 * S.pieces;
    if (w->col_sums) {
        if (x && w->cols % 4 == 0 && w->rows * w->cols <= std::min<int64_t>(strip_blocks * 65536, 3ll << 20) && aligned16(w->v) &&
            ((uintptr_t)w->q & 3) == 0 && aligned16(x->v) && ((uintptr_t)x->q & 3) == 0 && !x->tot) S.col_sums = w->col_sums;
        w->col_sums_left = S.col_sums != nullptr;
        add_rows = add_rows && w->col_sums_left;
    }
    for (int i = 0; i < 2; ++i) {
        parts[i] = c.take<float2>(kMaxParts);
        if (!ops[i]) continue;
        QuantOperand &op = *ops[i];
        if ((rc = check_common(op.v, op.rows, op.cols, QBP_PER_TENSOR, QBP_ROUND_NEAREST, op.qp))) return rc;
        o[i] = quant_out(op.q, nullptr, nullptr, nullptr);
        op.row_sums_left = op.row_sums && fuse_rowsums(op.v, op.rows * op.cols, op.cols, add_rows, op.row_sums, o[i]);
        if (op.row_sums_left && o[i].rs_shift < 0 && (rc = zero.add(op.row_sums, op.rows))) return rc;
        vec[i] = quant_vec(op.v, op.cols, 0, o[i]);
        if (op.tot) {
            if ((rc = zero.add(op.tot, 2 * op.cols))) return rc;
            if (i == 0 && vec[i] && quantizer_totals_supported(op.cols)) { o[i].chansum8 = reinterpret_cast<unsigned long long *>(op.tot); op.tot_left = true; }
        }
    }
    // the scans (and what they clear on the way), then the codes; the weights ride along with the activation
    if (x && vec[0] && vec[1]) {
        const int64_t nx = x->rows * x->cols, nw = w->rows * w->cols;
        ScanJob a{x->v, nx, parts[0], scan_blocks(nx, true), 1}, b{w->v, nw, parts[1], scan_blocks(nw, true), 0};
        // one wave in all: each tensor its share
        const int wave = std::min(kMaxParts, sm_count() * blocks_per_sm<range_partial_kernel<4>>(kThreads));
        if (a.blocks + b.blocks > wave) {
            b.blocks = std::max(1, std::min(b.blocks, (int)(wave * nw / (nx + nw))));
            a.blocks = std::min(a.blocks, wave - b.blocks);
        }
        QBP_TRACE_BEGIN(st);
        launch(range_partial_kernel<4>, a.blocks + b.blocks, kThreads, 0, st, a, b, zero);
        QBP_LAUNCH_OK("range_partial_kernel");
        const QuantJob ja{x->v, nx, (int)x->cols, RangeSrc{parts[0], a.blocks, nullptr, x->qp, nullptr}, 0, 0, o[0], 0, 0};
        const QuantJob jb{w->v, nw, (int)w->cols, RangeSrc{parts[1], b.blocks, nullptr, w->qp, nullptr}, 0, 0, o[1], 0, 0};
        const int64_t per_block = (int64_t)kThreads * 4 * kUnroll;
        const bool totals = o[0].chansum8 != nullptr;
        const int qwave = sm_count() * (totals ? blocks_per_sm<quantize_pair_kernel<true>>(kThreads) : blocks_per_sm<quantize_pair_kernel<false>>(kThreads));
        int64_t ga = (nx + per_block - 1) / per_block, gb = (nw + per_block - 1) / per_block;
        if (S.col_sums) {
            gb = strip_blocks;
            ga = std::max<int64_t>(1, std::min<int64_t>(ga, qwave));
        } else if (ga + gb > qwave) { gb = std::max<int64_t>(1, std::min(gb, qwave * nw / (nx + nw))); ga = std::min(ga, qwave - gb); }
        QBP_TRACE_BEGIN(st);
        if (totals) launch(quantize_pair_kernel<true>, (int)(ga + gb), kThreads, (size_t)x->cols * 2 * sizeof(int), st, ja, jb, (int)gb, S);
        else        launch(quantize_pair_kernel<false>, (int)(ga + gb), kThreads, 0, st, ja, jb, (int)gb, S);
        QBP_LAUNCH_OK("quantize_pair_kernel");
        return QBP_OK;
    }
    for (int i = 0; i < 2; ++i) {
        if (!ops[i]) continue;
        QuantOperand &op = *ops[i];
        RangeSrc r{parts[i], 0, nullptr, op.qp, nullptr};
        if ((rc = launch_range(op.v, op.rows * op.cols, parts[i], &r.nparts, st, zero))) return rc;
        zero = ZeroJobs{};
        if ((rc = launch_quantize(op.v, op.rows * op.cols, op.cols, 0, QBP_ROUND_NEAREST, r, 0, 0, 0, o[i], st))) return rc;
    }
    return QBP_OK;
}

}  // namespace qbp

using namespace qbp;

extern "C" __attribute__((visibility("default"))) const char *qbp_last_error(void) { return g_err; }

extern "C" __attribute__((visibility("default"))) int qbp_trace_enable(int on)
{
    for (TraceRec &r : g_trace) { g_event_pool.push_back(r.a); g_event_pool.push_back(r.b); }
    g_trace.clear();
    g_trace_on = on != 0;
    return QBP_OK;
}

extern "C" __attribute__((visibility("default"))) int qbp_trace_count(void) { return (int)g_trace.size(); }

extern "C" __attribute__((visibility("default"))) int qbp_trace_read(int index, char *name, int name_cap, float *ms)
{
    if (index < 0 || index >= (int)g_trace.size() || !name || name_cap <= 0 || !ms)
        return fail(QBP_ERR_INVALID_ARG, "trace_read: bad index or NULL output");
    const TraceRec &r = g_trace[index];
    if (!r.name) return fail(QBP_ERR_INVALID_ARG, "trace_read: record %d was never closed", index);
    snprintf(name, (size_t)name_cap, "%s", r.name);
    QBP_CUDA_OK(cudaEventElapsedTime(ms, r.a, r.b));
    return QBP_OK;
}

extern "C" __attribute__((visibility("default"))) size_t qbp_range_chunked_workspace_bytes(void)
{
    return 2 * align_up(sizeof(float2) * kMaxParts, 256) + 256;
}

extern "C" __attribute__((visibility("default"))) int qbp_range_chunked(const float *x, int64_t rows, int64_t cols, int64_t chunks,
                                                                       qbp_qparams *range_out, void *ws, size_t ws_bytes,
                                                                       void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (!x || !range_out) return fail(QBP_ERR_INVALID_ARG, "range_chunked: NULL argument");
    if (rows <= 0 || cols <= 0) return fail(QBP_ERR_INVALID_ARG, "range_chunked: empty tensor");
    if (chunks < 1 || chunks > kMaxParts || rows % chunks)
        return fail(QBP_ERR_INVALID_ARG, "range_chunked: rows (%lld) must be a multiple of chunks (%lld), at most %d chunks",
                    (long long)rows, (long long)chunks, kMaxParts);
    if (!ws || ws_bytes < qbp_range_chunked_workspace_bytes())
        return fail(QBP_ERR_WORKSPACE, "range_chunked: workspace of %zu bytes needed, %zu given",
                    qbp_range_chunked_workspace_bytes(), ws_bytes);
    WsCarver w(ws, ws_bytes);
    float2 *parts = w.take<float2>(kMaxParts);
    float2 *per_chunk = w.take<float2>(kMaxParts);
    const int64_t n_chunk = rows / chunks * cols;
    const bool vec = aligned16(x) && n_chunk % 4 == 0;
    // about one wave of blocks in all, at least one per chunk
    const int64_t per_block = (int64_t)kThreads * kRangeUnroll * (vec ? 4 : 1);
    const int wave = grid_for(vec ? blocks_per_sm<chunk_range_partial_kernel<4>>(kThreads) : blocks_per_sm<chunk_range_partial_kernel<1>>(kThreads),
                              (rows * cols + per_block - 1) / per_block);
    int bpc = (int)std::max<int64_t>(1, std::min<int64_t>((n_chunk + per_block - 1) / per_block, wave / chunks));
    bpc = (int)std::min<int64_t>(bpc, kMaxParts / chunks);
    QBP_TRACE_BEGIN(st);
    if (vec) launch(chunk_range_partial_kernel<4>, dim3(bpc, (unsigned)chunks), kThreads, 0, st, x, n_chunk, parts);
    else     launch(chunk_range_partial_kernel<1>, dim3(bpc, (unsigned)chunks), kThreads, 0, st, x, n_chunk, parts);
    QBP_LAUNCH_OK("chunk_range_partial_kernel");
    QBP_TRACE_BEGIN(st);
    launch(chunk_range_finalize_kernel, 1, kThreads, 0, st, parts, (int)chunks, bpc, per_chunk, range_out);
    QBP_LAUNCH_OK("chunk_range_finalize_kernel");
    return QBP_OK;
}

extern "C" __attribute__((visibility("default"))) size_t qbp_quantize_workspace_bytes(int64_t rows, int64_t cols, int granularity)
{
    (void)rows;
    return quant_ws_bytes(cols > 0 ? cols : 1, granularity);
}

extern "C" __attribute__((visibility("default"))) int qbp_quantize_s8(const float *x, int64_t rows, int64_t cols, int granularity, int rounding,
                               uint64_t seed, uint32_t tensor_id, const qbp_qparams *range_in, int8_t *q,
                               qbp_qparams *qp_out, int32_t *row_sums, int64_t *col_sums, void *ws, size_t ws_bytes,
                               void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (!q && rows * cols > 0) return fail(QBP_ERR_INVALID_ARG, "quantize_s8: q is NULL");
    if ((row_sums || col_sums) && granularity != QBP_PER_TENSOR)
        return fail(QBP_ERR_INVALID_ARG, "quantize_s8: row/column sums are per-tensor only");
    QuantOut o = quant_out(q, nullptr, nullptr, nullptr);
    const bool fused = row_sums && rows * cols > 0 && fuse_rowsums(x, rows * cols, cols, false, row_sums, o);
    int rc = quantize_any(8, x, rows, cols, granularity, rounding, seed, tensor_id, range_in, o, qp_out, ws, ws_bytes, st);
    if (rc) return rc;
    if (row_sums && !fused) { rc = launch_rowsum(q, true, rows, cols, row_sums, st); if (rc) return rc; }
    if (col_sums) { rc = launch_colsum(q, true, rows, cols, col_sums, st); if (rc) return rc; }
    return QBP_OK;
}

extern "C" __attribute__((visibility("default"))) int qbp_quantize_s16(const float *x, int64_t rows, int64_t cols, int granularity, int rounding,
                                uint64_t seed, uint32_t tensor_id, const qbp_qparams *range_in, int16_t *q,
                                int8_t *hi, uint8_t *lo, qbp_qparams *qp_out, void *ws, size_t ws_bytes, void *stream)
{
    if (!q && !hi && !lo) return fail(QBP_ERR_INVALID_ARG, "quantize_s16: q, hi and lo are all NULL");
    QuantOut o = quant_out(nullptr, q, hi, lo);
    return quantize_any(16, x, rows, cols, granularity, rounding, seed, tensor_id, range_in, o, qp_out, ws, ws_bytes,
                        (cudaStream_t)stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_bifurcate(const float *g, int64_t rows, int64_t cols, uint64_t seed, uint32_t tensor_id8,
                             uint32_t tensor_id16, int8_t *q8, qbp_qparams *qp8, int32_t *row_sums8, int8_t *hi,
                             uint8_t *lo, qbp_qparams *qp16, void *ws, size_t ws_bytes, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (rows < 0 || cols <= 0) return fail(QBP_ERR_INVALID_ARG, "bifurcate: rows must be >= 0 and cols > 0");
    if (!qp8 || !qp16) return fail(QBP_ERR_INVALID_ARG, "bifurcate: qp8 / qp16 is NULL");
    if (rows * cols > 0 && (!g || !q8 || !hi || !lo)) return fail(QBP_ERR_INVALID_ARG, "bifurcate: NULL tensor");
    if (((uintptr_t)g & 3) != 0) return fail(QBP_ERR_INVALID_ARG, "bifurcate: g is not 4-byte aligned");
    if (!ws || ws_bytes < quant_ws_bytes(cols, QBP_PER_TENSOR))
        return fail(QBP_ERR_WORKSPACE, "bifurcate: workspace of %zu bytes needed, %zu given",
                    quant_ws_bytes(cols, QBP_PER_TENSOR), ws_bytes);
    WsCarver w(ws, ws_bytes);
    float2 *parts = w.take<float2>(kMaxParts);
    RangeSrc r{parts, 0, nullptr, qp8, qp16};
    int rc = rows * cols > 0 ? launch_range(g, rows * cols, parts, &r.nparts, st) : launch_empty_qparams(qp8, qp16, st);
    if (rc) return rc;
    return bifurcate_tail(g, rows, cols, seed, tensor_id8, tensor_id16, q8, r, row_sums8, hi, lo, st);
}

// Both parameter records from clamping values the caller supplies.
__global__ void qparams_pair_from_range_kernel(const qbp_qparams *__restrict__ in, qbp_qparams *__restrict__ qp8,
                                               qbp_qparams *__restrict__ qp16)
{
    pdl_wait();
    *qp8 = make_qparams(in->vmin, in->vmax, 8);
    *qp16 = make_qparams(in->vmin, in->vmax, 16);
}

extern "C" __attribute__((visibility("default"))) int qbp_bifurcate_shard(const float *g, int64_t rows, int64_t cols, uint64_t seed,
                                   uint32_t tensor_id8, uint32_t tensor_id16, uint64_t index_base, const qbp_qparams *range_in,
                                   int8_t *q8, qbp_qparams *qp8, int32_t *row_sums8, int8_t *hi, uint8_t *lo,
                                   qbp_qparams *qp16, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (rows < 0 || cols <= 0) return fail(QBP_ERR_INVALID_ARG, "bifurcate_shard: rows must be >= 0 and cols > 0");
    if (!qp8 || !qp16 || !range_in) return fail(QBP_ERR_INVALID_ARG, "bifurcate_shard: qp8 / qp16 / range_in is NULL");
    if (rows * cols > 0 && (!g || !q8 || !hi || !lo)) return fail(QBP_ERR_INVALID_ARG, "bifurcate_shard: NULL tensor");
    if (((uintptr_t)g & 3) != 0) return fail(QBP_ERR_INVALID_ARG, "bifurcate_shard: g is not 4-byte aligned");
    if (index_base % 4) return fail(QBP_ERR_INVALID_ARG, "bifurcate_shard: index_base must be a multiple of 4");
    if (rows * cols == 0) {
        QBP_TRACE_BEGIN(st);
        launch(qparams_pair_from_range_kernel, 1, 1, 0, st, range_in, qp8, qp16);
        QBP_LAUNCH_OK("qparams_pair_from_range_kernel");
        return QBP_OK;
    }
    return bifurcate_tail(g, rows, cols, seed, tensor_id8, tensor_id16, q8, RangeSrc{nullptr, 0, range_in, qp8, qp16}, row_sums8, hi, lo, st, index_base);
}

// out = (float)acc * (sa * sb): the dequantisation of a weight gradient whose int64 accumulators were added up
// over several GPUs first (integer addition is exact, so the sum does not depend on the order of the GPUs).
__global__ void dequant_s64_kernel(const long long *__restrict__ acc, int64_t n, const qbp_qparams *qa,
                                   const qbp_qparams *qb, float *__restrict__ out)
{
    pdl_wait();
    const float s = __fmul_rn(qa->scale, qb->scale);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __fmul_rn((float)acc[i], s);
}

extern "C" __attribute__((visibility("default"))) int qbp_dequant_s64(const int64_t *acc, int64_t count, const qbp_qparams *qa,
                               const qbp_qparams *qb, float *out, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (count < 0 || (count > 0 && (!acc || !out)) || !qa || !qb) return fail(QBP_ERR_INVALID_ARG, "dequant_s64: NULL argument");
    if (count == 0) return QBP_OK;
    const int grid = (int)std::min<int64_t>((count + 255) / 256, (int64_t)sm_count() * 8);
    QBP_TRACE_BEGIN(st);
    launch(dequant_s64_kernel, grid, 256, 0, st, (const long long *)acc, count, qa, qb, out);
    QBP_LAUNCH_OK("dequant_s64_kernel");
    return QBP_OK;
}

// fp32 master-weight update (Section 6 "Putting it all together": the updates stay in float32 and run once per
// minibatch): g = dw + wd * w;  v = mu * v + g (with a momentum buffer);  w = w - lr * v.  Every operation is
// rounded on its own, in this order.
// A launch takes up to kSgdTensors tensors, each with its share of the blocks (the nine tensors of three layers: 2 us each as
// launches of their own, which is all they take).
constexpr int kSgdTensors = 32;
struct SgdTensor { float *w; const float *dw; float *v; int64_t n; float wd; int first_block; };
struct SgdTensors { SgdTensor t[kSgdTensors]; int count; };
__global__ void __launch_bounds__(256) sgd_update_kernel(const __grid_constant__ SgdTensors J, float lr, float mu)
{
    pdl_wait();
    int k = 0;
    while (k + 1 < J.count && (int)blockIdx.x >= J.t[k + 1].first_block) ++k;
    const SgdTensor &T = J.t[k];
    const int last = k + 1 < J.count ? J.t[k + 1].first_block : (int)gridDim.x;
    float *const w = T.w, *const v = T.v;
    const float *const dw = T.dw;
    const int64_t n = T.n, step = (int64_t)(last - T.first_block) * 256;
    const float wd = T.wd;
    for (int64_t i = (int64_t)((int)blockIdx.x - T.first_block) * 256 + threadIdx.x; i < n; i += step) {
        const float wi = w[i];
        float g = __fadd_rn(dw[i], __fmul_rn(wd, wi));
        if (v) { g = __fadd_rn(__fmul_rn(mu, v[i]), g); v[i] = g; }
        w[i] = __fsub_rn(wi, __fmul_rn(lr, g));
    }
}

extern "C" __attribute__((visibility("default"))) int qbp_sgd_update(float *w, const float *dw, float *momentum_buf, int64_t count,
                              float lr, float momentum, float weight_decay, void *stream)
{
    if (count < 0 || (count > 0 && (!w || !dw))) return fail(QBP_ERR_INVALID_ARG, "sgd_update: NULL tensor");
    if (count == 0) return QBP_OK;
    const qbp_sgd_tensor t{w, dw, momentum_buf, count, weight_decay, 0};
    return qbp_sgd_update_many(&t, 1, lr, momentum, stream);
}

extern "C" __attribute__((visibility("default"))) int qbp_sgd_update_many(const qbp_sgd_tensor *tensors, int n_tensors, float lr, float momentum,
                                                                          void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (n_tensors < 0 || (n_tensors > 0 && !tensors)) return fail(QBP_ERR_INVALID_ARG, "sgd_update_many: NULL tensors or a negative count");
    for (int i = 0; i < n_tensors; ++i)
        if (tensors[i].count < 0 || (tensors[i].count > 0 && (!tensors[i].w || !tensors[i].dw)))
            return fail(QBP_ERR_INVALID_ARG, "sgd_update_many: tensor %d is NULL or of negative size", i);
    for (int i = 0; i < n_tensors;) {
        SgdTensors J{};
        int blocks = 0;
        for (; i < n_tensors && J.count < kSgdTensors; ++i) {
            const qbp_sgd_tensor &t = tensors[i];
            if (t.count == 0) continue;
            J.t[J.count++] = SgdTensor{t.w, t.dw, t.momentum_buf, t.count, t.weight_decay, blocks};
            blocks += (int)std::min<int64_t>((t.count + 255) / 256, (int64_t)sm_count() * 8);
        }
        if (!J.count) break;
        QBP_TRACE_BEGIN(st);
        launch(sgd_update_kernel, blocks, 256, 0, st, J, lr, momentum);
        QBP_LAUNCH_OK("sgd_update_kernel");
    }
    return QBP_OK;
}

extern "C" __attribute__((visibility("default"))) int qbp_quantize_s8_static(const float *x, int64_t rows, int64_t cols, int granularity,
                                      int rounding, uint64_t seed, uint32_t tensor_id, int8_t *q,
                                      qbp_qparams *qp_out, void *stream)
{
    if (!q && rows * cols > 0) return fail(QBP_ERR_INVALID_ARG, "quantize_s8_static: q is NULL");
    int rc = check_common(x, rows, cols, granularity, rounding, qp_out);
    if (rc) return rc;
    if (granularity == QBP_PER_CHANNEL && cols > QBP_STATIC_MAX_CHANNELS)
        return fail(QBP_ERR_UNSUPPORTED_SHAPE,
                    "quantize_s8_static: %lld channels exceed the built-in scratch (at most %d per-channel ranges); "
                    "use qbp_quantize_s8 with a caller workspace",
                    (long long)cols, QBP_STATIC_MAX_CHANNELS);
    if (quant_ws_bytes(cols, granularity) > kStaticScratchBytes)
        return fail(QBP_ERR_UNSUPPORTED_SHAPE, "quantize_s8_static: the scan needs %zu scratch bytes, %zu are built in",
                    quant_ws_bytes(cols, granularity), kStaticScratchBytes);
    void *scratch = nullptr;
    rc = static_scratch_address(&scratch);
    if (rc) return rc;
    // every partial the finalising kernel reads was written by this call's scan: nothing has to start at zero
    QuantOut o = quant_out(q, nullptr, nullptr, nullptr);
    return quantize_any(8, x, rows, cols, granularity, rounding, seed, tensor_id, nullptr, o, qp_out, scratch,
                        kStaticScratchBytes, (cudaStream_t)stream);
}
