// Sums of stored codes for the products' zero-point corrections: per row, per column, per image edge, several tensors at once.
// The body runs in a launch of its own (code_sums_kernel) or in extra blocks of a kernel that has the machine to itself for
// too short a time to fill it (bn_bwd_finalize_kernel, conv_terms_kernel).
#pragma once

#include "qbp_mma.cuh"

namespace qbp {

constexpr int kSumThreads = 256;
struct SumJobDev { const uint8_t *q; int64_t rows; int cols, kind, first, blocks, G, pieces, corner_pieces, H, W, lg_log2; uint32_t flip; int32_t *out; int64_t *out64; };
struct SumJobs { SumJobDev j[kMaxSumJobs]; int count; ZeroJobs zero; };
// The device form of `count` jobs; *blocks: the blocks they take.  (qbp_quant.cu)
int fill_sum_jobs(const SumJob *jobs, int count, SumJobs &J, int *blocks);

#ifdef __CUDACC__
// Block `blk` of the jobs.  Unsigned codes are summed as codes - 128 (top bit flipped) and 128 per code is added at the end, so
// that one form of the dot product serves both.
// Per row: a group of G lanes per row, four 16-byte loads in flight.  Per column and per edge: a block takes a strip of up to
// 128 columns (eight 16-byte groups across, 32 rows high) over one piece of the rows, four rows in flight per thread; its
// rows meet by shuffle and in 4 KB of shared memory.
// Bound by the read of the codes where there are many, by latency otherwise (the operands of an 8192^3 product, 134 MB: 33 us with the launch, 4 TB/s).
__device__ __forceinline__ void code_sums_block(const SumJobs &J, int blk)
{
    int k = 0;
    while (k + 1 < J.count && blk >= J.j[k + 1].first) ++k;
    const SumJobDev &j = J.j[k];
    const int bid = blk - j.first, cv = j.cols >> 4, lane = threadIdx.x & 31;
    const uint32_t flip = j.flip;
    if (j.kind == kSumRows) {
        const int G = j.G, gl = lane % G;
        const int groups_per_block = kSumThreads / G;
        // (the loop bound is the block's, so that the shuffles see whole warps)
        for (int64_t rb = (int64_t)bid * groups_per_block; rb < j.rows; rb += (int64_t)j.blocks * groups_per_block) {
            const int64_t r = rb + threadIdx.x / G;
            const bool in = r < j.rows;
            const uint4 *row = reinterpret_cast<const uint4 *>(j.q + (in ? r : 0) * j.cols);
            int acc = 0;
            auto add = [&](const uint4 &v) {
                acc = __dp4a((int)(v.x ^ flip), 0x01010101, acc); acc = __dp4a((int)(v.y ^ flip), 0x01010101, acc);
                acc = __dp4a((int)(v.z ^ flip), 0x01010101, acc); acc = __dp4a((int)(v.w ^ flip), 0x01010101, acc);
            };
            int c = in ? gl : cv;
            for (; c + 3 * G < cv; c += 4 * G) {
                uint4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = __ldg(row + c + u * G);
#pragma unroll
                for (int u = 0; u < 4; ++u) add(v[u]);
            }
            for (; c < cv; c += G) add(__ldg(row + c));
            for (int o = G >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (in && gl == 0) j.out[r] = acc + (flip ? 128 * j.cols : 0);
        }
        return;
    }
    // a strip is 16 * lg columns wide (lg = 8, or the channels' groups when they are fewer: no lane idles) and 256 / lg rows high
    __shared__ int s_acc[kSumThreads / 32][128];
    const int lg = 1 << j.lg_log2, strips = (cv + lg - 1) >> j.lg_log2, strip = bid % strips;
    // (edges: the pieces of the four long ones, then those of the corners)
    const int unit = bid / strips, long_units = 4 * j.pieces;
    const bool corner = j.kind == kSumEdges && unit >= long_units;
    const int nth = corner ? unit - long_units : unit;
    const int edge = j.kind != kSumEdges ? 0 : (corner ? 4 : 0) + nth % 4;
    const int piece = j.kind != kSumEdges ? unit : nth / 4, pieces = corner ? j.corner_pieces : j.pieces;
    // an edge: `len` positions of every image, `step` apart, from `off`
    const int HW = j.H * j.W;
    const int len = edge < 2 ? j.W : edge < 4 ? j.H : 1, step = edge < 2 ? 1 : j.W;
    const int off = ((edge == 1 || edge >= 6) ? (j.H - 1) * j.W : 0) + ((edge == 3 || edge == 5 || edge == 7) ? j.W - 1 : 0);
    const int64_t rows = j.kind == kSumEdges ? j.rows / HW * len : j.rows;
    auto row_of = [&](int64_t r) -> int64_t {
        if (j.kind != kSumEdges) return r;
        const unsigned img = (unsigned)r / (unsigned)len;
        return (int64_t)img * HW + off + (int64_t)((unsigned)r - img * (unsigned)len) * step;
    };
    const int64_t r_begin = rows * piece / pieces, r_end = rows * (piece + 1) / pieces;
    const int g = (strip << j.lg_log2) + (lane & (lg - 1)), ty = (int)threadIdx.x >> j.lg_log2, rpb = kSumThreads >> j.lg_log2;
    int acc[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) acc[e] = 0;
    if (g < cv) {
        constexpr int U = 4;
        const uint8_t *base = j.q + (int64_t)g * 16;
        for (int64_t r = r_begin + ty; r < r_end; r += rpb * U) {
            uint4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r + rpb * u < r_end) v[u] = __ldg(reinterpret_cast<const uint4 *>(base + row_of(r + rpb * u) * j.cols));
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (r + rpb * u >= r_end) break;
                const uint32_t w[4] = {v[u].x ^ flip, v[u].y ^ flip, v[u].z ^ flip, v[u].w ^ flip};
#pragma unroll
                for (int e = 0; e < 16; ++e) acc[e] = __dp4a((int)w[e >> 2], 1 << (8 * (e & 3)), acc[e]);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 16; ++e)
        for (int o = lg; o < 32; o <<= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if (lane < lg) {
#pragma unroll
        for (int e = 0; e < 16; ++e) s_acc[threadIdx.x >> 5][lane * 16 + e] = acc[e];
    }
    named_barrier(1, kSumThreads);       // (the block may have more threads than take part)
    const int c = (strip << (j.lg_log2 + 4)) + (int)threadIdx.x;
    if ((int)threadIdx.x < 16 * lg && c < j.cols) {
        int sum = 0;
#pragma unroll
        for (int w = 0; w < kSumThreads / 32; ++w) sum += s_acc[w][threadIdx.x];
        const int whole = sum + (flip ? 128 * (int)(r_end - r_begin) : 0);
        const int64_t at = (int64_t)(j.kind == kSumEdges ? edge : j.out64 ? 0 : piece) * j.cols + c;
        if (j.out64) { if (whole) atomicAdd(reinterpret_cast<unsigned long long *>(j.out64 + at), (unsigned long long)(long long)whole); }
        else j.out[at] = whole;
    }
}

#endif  // __CUDACC__
}  // namespace qbp
