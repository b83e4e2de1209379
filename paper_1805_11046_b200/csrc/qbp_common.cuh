// Shared host/device helpers of libqbp: error reporting, launch checks, small
// numeric helpers with a pinned IEEE operation order, Philox4x32-10, and thin
// wrappers over the sm_100a PTX used by the tensor-core kernels (mbarrier,
// TMA, tcgen05).  No kernel lives here.
#pragma once

#include <cuda_runtime.h>
#include <cstdarg>
#include <cstdint>
#include <cstdio>

#include "../../include/qbp.h"

namespace qbp {

// ---------------------------------------------------------------- host side
void set_error(const char *fmt, ...);          // defined in qbp_quant.cu
int fail(int status, const char *fmt, ...);    // sets the message, returns status

#define QBP_CUDA_OK(expr)                                                         \
    do {                                                                          \
        cudaError_t e_ = (expr);                                                  \
        if (e_ != cudaSuccess)                                                    \
            return ::qbp::fail(QBP_ERR_CUDA, "%s: %s", #expr, cudaGetErrorString(e_)); \
    } while (0)

// Optional per-kernel timing (qbp_trace_enable): an event pair around every launch.
void trace_begin(cudaStream_t st);
void trace_end(const char *name, cudaStream_t st);
#define QBP_TRACE_BEGIN(st) ::qbp::trace_begin(st)

// Placed after every kernel launch; expects the stream in a variable named `st`.
#define QBP_LAUNCH_OK(name)                                                       \
    do {                                                                          \
        ::qbp::trace_end(name, st);                                               \
        cudaError_t e_ = cudaGetLastError();                                      \
        if (e_ != cudaSuccess)                                                    \
            return ::qbp::fail(QBP_ERR_CUDA, "launch of %s: %s", name, cudaGetErrorString(e_)); \
    } while (0)

// Kernels of one stream run one after another, but a kernel's launch need not wait until the one before has been retired:
// launch() marks every kernel as a programmatic dependent of its predecessor, whose blocks let it go as they exit, and each kernel
// waits, before it touches the predecessor's results, until those are visible (pdl_wait).  A chain of dependent small kernels then
// costs about 2 us each instead of 4 to 5.  Only the short kernels whose successor is a product (code sums and zero-point terms) let
// it go while they run (pdl_trigger): elsewhere blocks that wait on an SM beside the running kernel made that kernel slower (per-channel
// statistics of 51 MB 14.5 -> 20 us, the layer of 56 x 56 x 64 543 -> 577 us, three layers' inference at batch 8 106 -> 117 us).
// There are two forms of it.
//   - Terms always, and code sums whose launch was asked for it (SumJobs::beside, sums of 1 to 32 MB), let the product go behind their
//     own wait: all that was launched before them is complete then, the product's operands and parameters among it.  The product is
//     told so (`beside`) and starts on its operands at once; only its epilogue, which reads the sums or terms and writes the output,
//     waits for their end, and so does whoever raises its status word, which they may clear.
//   - Other code sums let it go at their start, ahead of their wait: the kernels before them may still run, so the product is not told
//     and waits in every role before its first access; it has only set itself up by then (barriers, tensor memory, parameters).
// Any other successor of either form waits like the second.  (Layer gradient of 16 x 7 x 7, 512 -> 512 channels, with its terms:
// 27.6 -> 21.6 us; the layer of 20 x 19 x 19, 96 -> 160, 92.8 -> 91.2; the low-bit layer 196.5 -> 194.4.)
// While launches are timed one by one the dependency is the ordinary one.
bool trace_is_on();
template <typename... P, typename... A>
inline void launch(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = trace_is_on() ? 0 : 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);     // (an error is found by QBP_LAUNCH_OK)
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
int sm_count();                                // cached multiprocessor count of the current device

// Function attributes (the opt-in to more than 48 KB of dynamic shared memory) belong to a device: set them once
// per device ordinal, whichever host thread gets there first.
constexpr int kMaxDevices = 64;
struct PerDeviceOnce {
    bool done[kMaxDevices] = {};
    // true when the caller still has to do the set-up for the current device (and then calls mark())
    bool pending(int *dev_out)
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); *dev_out = -1; return true; }
        *dev_out = dev;
        return !__atomic_load_n(&done[dev], __ATOMIC_ACQUIRE);
    }
    void mark(int dev) { if (dev >= 0) __atomic_store_n(&done[dev], true, __ATOMIC_RELEASE); }
};
#define QBP_SMEM_OPT_IN(once, kernel, bytes)                                                                       \
    do {                                                                                                           \
        int dev_ = -1;                                                                                             \
        if ((once).pending(&dev_)) {                                                                               \
            QBP_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(bytes)));  \
            (once).mark(dev_);                                                                                     \
        }                                                                                                          \
    } while (0)

// Carves 256-byte aligned pieces out of the caller's workspace.
struct WsCarver {
    char *base; size_t off; size_t cap;
    WsCarver(void *ws, size_t bytes) : base(static_cast<char *>(ws)), off(0), cap(bytes) {}
    template <typename T> T *take(size_t count) {
        size_t bytes = align_up(count * sizeof(T), 256);
        T *p = reinterpret_cast<T *>(base + off);
        off += bytes;
        return p;
    }
    bool ok() const { return base != nullptr && off <= cap; }
};

// Where a kernel that quantises per tensor takes its range from: the (min, max) pairs that the kernel before left (per block or
// per channel; `parts`), clamping values the caller gave (`given`), or -- both NULL -- finished records at qp8 / qp16.  In the
// first two cases every block works out the parameters itself (about a microsecond, most of it behind its first loads;
// a launch of its own for it costs two and more) and the first block leaves the records at qp8 / qp16 (each nullable).
struct RangeSrc { const float2 *parts; int nparts; const qbp_qparams *given; qbp_qparams *qp8, *qp16; };
// Regions of 32-bit words that a kernel clears on the way (a status word, sums that a later kernel adds to); one too many is an error.
constexpr int kMaxZeroJobs = 5;
struct ZeroJobs {
    int count;
    uint32_t *p[kMaxZeroJobs]; int64_t words[kMaxZeroJobs];
    [[nodiscard]] int add(void *at, int64_t n)
    {
        if (n <= 0) return QBP_OK;
        if (count == kMaxZeroJobs) return fail(QBP_ERR_INVALID_ARG, "more than %d regions to clear in one launch", kMaxZeroJobs);
        p[count] = static_cast<uint32_t *>(at); words[count++] = n;
        return QBP_OK;
    }
};

// -------------------------------------------------------------- device side
#ifdef __CUDACC__

// The two halves of a programmatic launch (see launch()).  Only code_sums_kernel and conv_terms_kernel trigger: the terms behind their
// wait, the sums behind or ahead of it.  A kernel that allocates tensor memory never does: its successor could take that memory first
// and then wait for a kernel that cannot go on.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A load of what a kernel that let this one go while it ran writes (code sums, zero-point terms): an ordinary global load that
// stays behind pdl_wait().  __ldg would take the non-coherent path, which is for memory that nothing writes while the reading
// kernel is resident; everything else that a kernel reads was written by blocks that had ended before it started.
__device__ __forceinline__ int32_t load_after_wait(const int32_t *p)
{
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies
// (one wide multiply each); the round keys are key + r * (0x9E3779B9, 0xBB67AE85).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c.x;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c.z;
        const uint32_t k0 = k.x + (uint32_t)r * 0x9E3779B9u, k1 = k.y + (uint32_t)r * 0xBB67AE85u;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k0, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k1, (uint32_t)p0);
    }
    return c;
}

// Scale and zero-point from clamping values (Appendix B), fp32, fixed order.
__device__ __forceinline__ qbp_qparams make_qparams(float vmin, float vmax, int bits)
{
    const int L = (1 << bits) - 1;
    vmin = fminf(vmin, 0.0f);
    vmax = fmaxf(vmax, 0.0f);
    float range = __fsub_rn(vmax, vmin);
    float s = (range == 0.0f) ? 1.0f : __fdiv_rn(range, (float)L);
    float z = rintf(__fdiv_rn(-vmin, s));
    z = fminf(fmaxf(z, 0.0f), (float)L);
    qbp_qparams q;
    q.scale = s;
    q.zero_point = (int)z - (1 << (bits - 1));
    q.vmin = vmin;
    q.vmax = vmax;
    return q;
}

// One element to its unsigned code in [0, L].  rnd is the element's Philox word; stochastic rounding takes a
// 16-bit draw from it: the high half-word for an 8-bit code, the low half-word for a 16-bit code (the two copies
// of one gradient then round independently from one word).
template <bool STOCHASTIC>
__device__ __forceinline__ int quantize_code(float x, float inv_scale, float zp_u, float Lf, uint32_t rnd)
{
    float t = __fmaf_rn(x, inv_scale, zp_u);
    float c;
    if (!STOCHASTIC) {
        c = rintf(t);
    } else {
        float f = floorf(t);
        float frac = __fsub_rn(t, f);
        const uint32_t draw = (Lf == 255.0f) ? (rnd >> 16) : (rnd & 0xFFFFu);
        float u = __fmul_rn((float)draw, 0x1p-16f);
        c = (u < frac) ? __fadd_rn(f, 1.0f) : f;
    }
    // c is integral: the saturating conversion is the clamp to [0, 2^bits - 1] (Lf selects the width)
    uint32_t code;
    if (Lf == 255.0f) asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(code) : "f"(c));
    else              asm("cvt.rni.sat.u16.f32 %0, %1;" : "=r"(code) : "f"(c));
    return (int)code;
}

// The stochastic codes of one element in fixed point: the same results as quantize_code<true> with fewer
// instructions.  With t = fma(x, inv, zp), f = floor(t), frac = t - f and a 16-bit draw d, the code is
// f + [d * 2^-16 < frac] = f + [d < ceil(frac * 2^16)] (d is an integer).  t * 2^16 is exact in fp32 and
// ceil(t * 2^16) = f * 2^16 + ceil(frac * 2^16), so adding 0xFFFF - d carries into bit 16 exactly when the code
// rounds up.  The conversion saturates negative t to 0 (code 0, as the clamp gives) and the minimum with
// L * 2^16 is the clamp at the top (then nothing can carry).
// The caller passes inv_scale and zp_u already multiplied by 2^16: scaling by a power of two commutes with the
// rounding of the fused multiply-add, so fma(x, inv * 2^16, zp * 2^16) is exactly 2^16 * fma(x, inv, zp).
// What is stored is the code with its top bit flipped (code - 2^(M-1)); that bit is flipped by the same addition.
// 8 bits: the stored code is byte 2 of the result (byte 3 is not to be used); the draw is the high half of rnd.
__device__ __forceinline__ uint32_t quantize_sr8_byte2(float x, float inv_scale_2p16, float zp_u_2p16, uint32_t rnd)
{
    uint32_t tc;
    asm("cvt.rpi.sat.u32.f32 %0, %1;" : "=r"(tc) : "f"(__fmaf_rn(x, inv_scale_2p16, zp_u_2p16)));
    return min(tc, 0x00FF0000u) + 0x0080FFFFu - (rnd >> 16);
}
// 16 bits: the stored code is the upper half of the result (high byte = byte 3, low byte = byte 2); the draw is the low half of rnd.
__device__ __forceinline__ uint32_t quantize_sr16_top_half(float x, float inv_scale_2p16, float zp_u_2p16, uint32_t rnd)
{
    uint32_t tc;
    asm("cvt.rpi.sat.u32.f32 %0, %1;" : "=r"(tc) : "f"(__fmaf_rn(x, inv_scale_2p16, zp_u_2p16)));
    return min(tc, 0xFFFF0000u) + 0x80000000u + ((~rnd) & 0xFFFFu);
}

// Philox4x32-10 with the ten round keys precomputed (they depend on the key only); passed to a kernel by value,
// they sit in its constant parameter space and cost no registers.
struct PhiloxKeys { uint32_t k0[10], k1[10]; };
inline PhiloxKeys philox_keys_host(uint64_t seed)
{
    PhiloxKeys r;
    for (int i = 0; i < 10; ++i) {
        r.k0[i] = (uint32_t)seed + (uint32_t)i * 0x9E3779B9u;
        r.k1[i] = (uint32_t)(seed >> 32) + (uint32_t)i * 0xBB67AE85u;
    }
    return r;
}
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const PhiloxKeys &k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c.x;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k.k0[r], (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k.k1[r], (uint32_t)p0);
    }
    return c;
}

// Four consecutive elements of a gradient bifurcated (Section 6): the four stored 8-bit codes, and the high and low limbs of the
// four stored 16-bit codes (the low one XORed with lo_flip).  r8, r16: their Philox words (the same for equal tensor ids: the 8-bit
// draw is a word's high half, the 16-bit draw its low half).  c16: the 16-bit codes, each in the upper half of its word.
struct BifWords { uint32_t q8, hi, lo; };
__device__ __forceinline__ BifWords bifurcate4(const float (&v)[4], float inv8, float zp8, float inv16, float zp16, const uint4 &r8,
                                               const uint4 &r16, uint32_t lo_flip, uint32_t (&c16)[4])
{
    const uint32_t w8[4] = {r8.x, r8.y, r8.z, r8.w}, w16[4] = {r16.x, r16.y, r16.z, r16.w};
    uint32_t c8[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        c8[e] = quantize_sr8_byte2(v[e], inv8, zp8, w8[e]);
        c16[e] = quantize_sr16_top_half(v[e], inv16, zp16, w16[e]);
    }
    // (low, low, high, high) bytes of two 16-bit codes each, then the two words: four permutes for both limbs
    const uint32_t t01 = __byte_perm(c16[0], c16[1], 0x7362), t23 = __byte_perm(c16[2], c16[3], 0x7362);
    return {__byte_perm(__byte_perm(c8[0], c8[1], 0x0062), __byte_perm(c8[2], c8[3], 0x0062), 0x5410), __byte_perm(t01, t23, 0x7632),
            __byte_perm(t01, t23, 0x5410) ^ lo_flip};
}

// Range BN (Section 3, Eq. (range)): xhat and y of one element and the per-channel scale 1 / (C(n) (max - min)).
// The order of operations is part of the contract: every kernel that normalises (the apply passes, the fused
// epilogue of a product) must produce the same bits, so that forward, backward and requantisation agree.
__device__ __forceinline__ float bn_xhat(float x, float mu, float s) { return __fmul_rn(__fsub_rn(x, mu), s); }
__device__ __forceinline__ float bn_y(float xh, float g, float b) { return __fadd_rn(__fmul_rn(g, xh), b); }
// One element of the Range BN backward (the derivative stated with Eq. (rangebn) in Section 3, ties as in the forward):
// dx = s * (gamma * dy - m1 - k2 * ind), ind = [x == max] - [x == min].  Every operation is rounded on its own and
// none is contracted, so the value is a monotone function of dy for fixed (s >= 0, gamma, m1, k2, ind): the extremes of
// dx over a set of positions are this function of the extremes of dy (which is how the gradient's range is known
// before the gradient is written).  t = k2 * ind.
__device__ __forceinline__ float bn_dx(float d, float t, float s, float g, float m1)
{
    return __fmul_rn(s, __fsub_rn(__fsub_rn(__fmul_rn(g, d), m1), t));
}
// k2 * ind of a value (in a constant channel, max == min, s is 0 and t does not count)
__device__ __forceinline__ float bn_k2_ind(float x, float lo, float hi, float k2) { return x == hi ? k2 : x == lo ? -k2 : 0.0f; }
// Floats as integers that compare the same way (and back): for atomic minima and maxima of floats.
__device__ __forceinline__ int float_order(float f) { const int b = __float_as_int(f); return b ^ ((b >> 31) & 0x7fffffff); }
__device__ __forceinline__ float order_float(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }
__device__ __forceinline__ float bn_scale(float lo, float hi, float Cn);
// The rectifier's mask of a Range BN output as a threshold on the input.  y(x) = bn_y(bn_xhat(x, mu, s), g, b) is a
// monotone function of x (every operation is rounded on its own and monotone, s >= 0): rising for g >= 0, falling for
// g < 0, so {x : y(x) > 0} is a ray, and its end is found by a search over the floats in their order.  Returns (t, sgn) with  y(x) > 0  <=>  sgn * x >= t  for finite x (sgn = +-1; t = +-inf: none / all).
__device__ inline float2 relu_threshold(float mu, float s, float g, float b)
{
    const bool rising = !(g < 0.0f);
    const float sgn = rising ? 1.0f : -1.0f;
    // (the keys of x, or of -x when the output falls: the output then rises with the key; the key of -x is -1 - key)
    auto on = [&](long long k) { return bn_y(bn_xhat(order_float(rising ? (int)k : -1 - (int)k), mu, s), g, b) > 0.0f; };
    long long lo = float_order(-3.402823466e38f), hi = float_order(3.402823466e38f);
    if (!on(hi)) return make_float2(INFINITY, sgn);
    if (on(lo)) return make_float2(-INFINITY, sgn);
    // Outwards from where the output is zero in real numbers, in growing steps, then between the last two: with the two ends four
    // evaluations for beta = 0, 4.7 on average otherwise, where halving the whole range takes 34, 3 us at the end of every backward
    // statistics' pass.
    const float x0 = sgn * __fsub_rn(mu, __fdiv_rn(b, __fmul_rn(g, s)));
    if (fabsf(x0) < 3.0e38f) {
        const long long k0 = float_order(x0);
        if (on(k0)) {
            hi = k0;
            for (long long step = 1; hi - step > lo; step *= 8) { if (on(hi - step)) hi -= step; else { lo = hi - step; break; } }
        } else {
            lo = k0;
            for (long long step = 1; lo + step < hi; step *= 8) { if (on(lo + step)) { hi = lo + step; break; } lo += step; }
        }
    }
    while (hi - lo > 1) { const long long mid = lo + (hi - lo) / 2; if (on(mid)) hi = mid; else lo = mid; }       // smallest key that is on
    return make_float2(order_float((int)hi), sgn);
}
__device__ __forceinline__ float bn_scale(float lo, float hi, float Cn)
{
    float r = __fsub_rn(hi, lo);
    return r > 0.0f ? __fdiv_rn(1.0f, __fmul_rn(Cn, r)) : 0.0f;
}

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The whole block's (min, max) of per-thread values (threads a multiple of 32, at most 1024; once per kernel).
__device__ __forceinline__ float2 block_min_max(float lo, float hi)
{
    __shared__ float2 s_red[32];
    lo = warp_min(lo); hi = warp_max(hi);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = make_float2(lo, hi);
    __syncthreads();
    float2 r = s_red[0];
    for (unsigned w = 1; w < blockDim.x / 32; ++w) { const float2 t = s_red[w]; r.x = fminf(r.x, t.x); r.y = fmaxf(r.y, t.y); }
    return r;
}
// ... of (min, max) pairs in memory.
__device__ __forceinline__ float2 block_range(const float2 *__restrict__ parts, int nparts)
{
    float lo = INFINITY, hi = -INFINITY;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) { const float2 t = __ldg(parts + i); lo = fminf(lo, t.x); hi = fmaxf(hi, t.y); }
    return block_min_max(lo, hi);
}
// A thread's share of the clearing, `threads` threads taking part.
__device__ __forceinline__ void run_zero_jobs(const ZeroJobs &z, int64_t thread, int64_t threads)
{
#pragma unroll
    for (int k = 0; k < kMaxZeroJobs && k < z.count; ++k)        // (unrolled: an index into a parameter would copy it to local memory)
        for (int64_t i = thread; i < z.words[k]; i += threads) z.p[k][i] = 0u;
}
struct QParamsReg { float inv, zp_u; };       // 1 / scale and the unsigned zero-point
__device__ __forceinline__ QParamsReg qparams_reg(const qbp_qparams &qp, int bits)
{
    QParamsReg r;
    r.inv = __fdiv_rn(1.0f, qp.scale);
    r.zp_u = (float)(qp.zero_point + (1 << (bits - 1)));
    return r;
}
// The parameters of the copies that are wanted, by a whole block; `first`: the block that leaves the records.
__device__ __forceinline__ void resolve_range(const RangeSrc &R, bool want8, bool want16, bool first, QParamsReg &p8, QParamsReg &p16)
{
    if (!R.parts && !R.given) {
        if (want8) p8 = qparams_reg(*R.qp8, 8);
        if (want16) p16 = qparams_reg(*R.qp16, 16);
        return;
    }
    const float2 r = R.given ? make_float2(R.given->vmin, R.given->vmax) : block_range(R.parts, R.nparts);
    if (want8) {
        const qbp_qparams q = make_qparams(r.x, r.y, 8);
        if (first && threadIdx.x == 0 && R.qp8) *R.qp8 = q;
        p8 = qparams_reg(q, 8);
    }
    if (want16) {
        const qbp_qparams q = make_qparams(r.x, r.y, 16);
        if (first && threadIdx.x == 0 && R.qp16) *R.qp16 = q;
        p16 = qparams_reg(q, 16);
    }
}

// ---- sm_100a PTX wrappers ---------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` SM clock cycles (by default about a second) and reports false; the
// caller then raises the kernel's status word and leaves through its normal exit.
constexpr long long kWaitLimitCycles = 2000000000ll;
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit = kWaitLimitCycles)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}

// The same wait by every lane of a converged warp; the answer is the same in all of them.
__device__ __forceinline__ bool mbar_wait_uniform(uint64_t *bar, uint32_t parity, long long limit = kWaitLimitCycles)
{
    const bool ok = mbar_wait(bar, parity, limit);
    return __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
}

// The same wait for a whole warp: one lane polls (with a short sleep between polls, so that waiting warps
// leave the shared-memory pipe to the warps that feed the tensor core), the result is shared by shuffle.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, long long limit = kWaitLimitCycles)
{
    int ok = 1;
    if ((threadIdx.x & 31) == 0 && !mbar_try_wait(bar, parity)) {
        const long long t0 = clock64();
        while (!mbar_try_wait(bar, parity)) {
            if (clock64() - t0 > limit) { ok = 0; break; }
            __nanosleep(40);
        }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    return ok != 0;
}

// A kernel whose bounded wait ran out records it here; the word only ever goes from 0 to QBP_ERR_TIMEOUT.
__device__ __forceinline__ void raise_timeout(int *status) { atomicExch(status, (int)QBP_ERR_TIMEOUT); }

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// TMA tiled loads, completion reported on an mbarrier as transferred bytes.
__device__ __forceinline__ void tma_load_2d(void *dst, const void *map, uint64_t *bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const void *map, uint64_t *bar, int x, int y, int z, int w)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
// TMA tiled stores (shared -> global) as bulk groups of the issuing thread; elements of the box that fall
// outside the tensor are not written.  The x coordinate times the element size must be a multiple of 16.
__device__ __forceinline__ void tma_store_2d(const void *map, const void *src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(smem_u32(src)), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void tma_store_4d(const void *map, const void *src, int x, int y, int z, int w)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(map), "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z), "r"(w)
                 : "memory");
}
// Per-thread asynchronous 16-byte copies global -> shared (L2 only), in groups a thread commits and waits for itself:
// what a thread copies and reads back itself needs no barrier.
__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// ... until at most N of this thread's groups are still in flight
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Until every store group of this thread has finished reading its shared-memory source.
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Until all but the latest store group of this thread have finished reading their sources.
__device__ __forceinline__ void tma_store_wait_read_but_one() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
// Until every store group of this thread is complete.
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Named barrier over `count` threads (a multiple of 32) of the CTA.
__device__ __forceinline__ void named_barrier(int id, int count)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void tma_prefetch_desc(const void *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// Tensor memory (TMEM) management; executed by one full warp.
__device__ __forceinline__ void tmem_alloc(uint32_t *slot_in_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot_in_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Three-input minimum / maximum (one instruction on sm_100).
__device__ __forceinline__ float fmin3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// True in exactly one lane of a converged warp.  The MMA warps run whole and put this around each tcgen05.mma and
// commit, rather than branching on the lane index once around the loop: the instruction takes its operands from
// warp-uniform registers, and only in code the compiler knows to be convergent are descriptors that change from
// one MMA to the next kept there (measured: 63 against 110 cycles per 128 x 64 x 32 MMA).
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}

// D[tmem] (+)= A[smem] * B[smem], 8-bit integer operands, int32 accumulator.  Volatile keeps it in order with
// the barrier waits and commits around it; there is no memory clobber, so that the issuing thread's loads of
// the next descriptors can be scheduled across it (that thread is bound by its own instruction latency).
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}
// Arrive on an mbarrier once every MMA issued so far by this thread has finished.
__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns of the accumulator into registers.
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// ... 16 columns
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait()
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

#endif  // __CUDACC__
}  // namespace qbp
