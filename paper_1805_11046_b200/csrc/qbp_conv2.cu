// The 3 x 3 convolution products y = W x and g_{l-1} = g_l W^T (Section 1, Eq. (grad_layer)) on CTA pairs:
// tcgen05.mma.cta_group::2, for layers with many channels, where the products are bound by the tensor pipe.
//
// Two CTAs of a cluster compute one tile of 256 output positions x bn channels (bn = 256 or 128): CTA r holds its box of 128
// positions (the A operand, loaded per tap and channel chunk as a shifted box, zeros outside the image) and half of the filter
// tile's columns, and the accumulator of its positions.  One thread of the leader issues every MMA.  With 256 channels the
// single-CTA kernel (128 x 256 tiles, the filter re-read per tile) fetched 48 KB per 512 MMA cycles and SM, 26 TB/s over the
// chip at full rate, and ran at a third of it (56 us forward, 48 us layer gradient for 50176 positions, 256 -> 256
// channels); a pair fetches 32 KB per SM for the same cycles and overlaps the epilogue with the next tile's MMAs.
//
// Roles per CTA, barriers and bounded waits as in the dense product on CTA pairs; no TMA load uses cluster multicast.
#include "qbp_mma.cuh"
#include "qbp_pair.cuh"

#include <algorithm>

namespace qbp {

constexpr int kC2Threads = 320;
constexpr int kC2EpiWarps = 8;
constexpr int kC2MaxStages = 8;
constexpr uint32_t kC2Slab = 32 * 128;
constexpr uint32_t kC2Smem = 225u * 1024u;

struct C2Stat { double sum; float lo, hi; };

struct Conv2Params {
    CUtensorMap mapA, mapB, mapC;
    uint32_t a_desc_lo, b_desc_lo, idesc;
    uint32_t b_bytes;                // this CTA's half of a filter tile
    int dgrad, bn, nbuf;
    int stages, cg;                  // ring stages of one (tap, chunk); stages released per commit
    int k_iters, cchunks;            // 9 taps x channel chunks of 128 (a ragged last one is zero-filled on the activation side)
    int tiles_m, tiles_n, tiles_total, pairs;      // pairs is a multiple of tiles_n: a pair meets one column tile only
    FastDiv d_tiles_n, d_tiles_w, d_tiles_h;
    int Nimg, H, W, C, N;            // C: channels of the filter's innermost extent; N: channels produced
    int bw_log2, bh_log2;            // the position box of a CTA: bw x bh x images = 128
    int32_t *acc_out; float *out;
    const int32_t *rowterm, *colterm;              // [positions], [16 border classes][N]
    const qbp_qparams *qa, *qb;
    float *st_lo, *st_hi; double *st_sum;          // per-channel statistics of the output, a row per CTA (NULL: not wanted)
    int beside;                      // the launch before writes the terms and neither operands nor parameters: only the epilogue waits for it
    int *status;
};

// The four MMAs of a stage (128 reduction channels of one tap).  BK: the filter operand's step per 32 of them in 16-byte units
// (2 inside a K-major row; 32 rows of an M/N-major tile of RB bytes a row: 2 * RB).
template <uint32_t BK, uint32_t RB, bool FIRST>
__device__ __forceinline__ void conv2_issue_stage(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc)
{
    constexpr uint32_t a_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t b_hi = ((8u * RB) >> 4) | (1u << 14) | ((RB == 128 ? 2u : 4u) << 29);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
        if (elect_one())
            mma_i8_pair(d_tmem, ((uint64_t)a_hi << 32) | (uint64_t)(a_lo + (uint32_t)kk * 2u),
                        ((uint64_t)b_hi << 32) | (uint64_t)(b_lo + (uint32_t)kk * BK), idesc, (FIRST && kk == 0) ? 0u : 1u);
}

struct Conv2MmaArgs {
    uint64_t *full_bar, *empty_bar, *acc_full, *acc_empty;
    uint32_t ring, stage_bytes, tmem, a_desc_lo, b_desc_lo, idesc, bn;
    int k_iters;
    uint32_t stages, cg, nbuf;
    int tile0, tiles_total, tile_step;
};
// False when a wait ran out.
template <uint32_t BK, uint32_t RB>
__device__ __forceinline__ bool conv2_mma_loop(const Conv2MmaArgs &A)
{
    uint32_t s = 0, ph = 0, buf = 0, bph = 1, in_group = 0, group = 0, a_addr = A.ring;
    for (int tile = A.tile0; tile < A.tiles_total; tile += A.tile_step) {
        if (!mbar_wait_uniform(&A.acc_empty[buf], bph)) return false;
        tc_fence_after();
        const uint32_t d_tmem = A.tmem + buf * A.bn;
        for (int it = 0; it < A.k_iters; ++it) {
            if (!mbar_wait_uniform(&A.full_bar[s], ph)) return false;
            tc_fence_after();
            const uint32_t a_lo = ((a_addr >> 4) & 0x3FFFu) | A.a_desc_lo;
            const uint32_t b_lo = (((a_addr + 16384u) >> 4) & 0x3FFFu) | A.b_desc_lo;
            if (it == 0) conv2_issue_stage<BK, RB, true>(d_tmem, a_lo, b_lo, A.idesc);
            else         conv2_issue_stage<BK, RB, false>(d_tmem, a_lo, b_lo, A.idesc);
            if (++in_group == A.cg) {
                if (elect_one()) mma_commit_pair(&A.empty_bar[group]);
                in_group = 0; ++group;
            }
            a_addr += A.stage_bytes;
            if (++s == A.stages) { s = 0; ph ^= 1u; group = 0; a_addr = A.ring; }
        }
        if (elect_one()) mma_commit_pair(&A.acc_full[buf]);
        if (++buf == A.nbuf) { buf = 0; bph ^= 1u; }
    }
    return true;
}

// Where this CTA's box of a tile starts.
struct Conv2Box { int w0, h0, img0; };
__device__ __forceinline__ Conv2Box conv2_box(const Conv2Params &P, int tile, uint32_t rank)
{
    int tile_m, t1, tw, tn, th;
    tile_m = P.d_tiles_n.div(tile);
    P.d_tiles_w.divmod(tile_m * 2 + (int)rank, t1, tw);
    P.d_tiles_h.divmod(t1, tn, th);
    Conv2Box b;
    b.w0 = tw << P.bw_log2; b.h0 = th << P.bh_log2; b.img0 = tn << (7 - P.bw_log2 - P.bh_log2);
    return b;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kC2Threads, 1) qbp_conv2_kernel(const __grid_constant__ Conv2Params P)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kC2MaxStages], empty_bar[kC2MaxStages], acc_full[4], acc_empty[4];
    __shared__ uint32_t tmem_slot;

    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);
    const uint32_t stage_bytes = 16384u + P.b_bytes;
    uint8_t *staging = smem + (size_t)P.stages * stage_bytes;
    int32_t *s_cterm = reinterpret_cast<int32_t *>(staging + kC2EpiWarps * kC2Slab);                  // [16][bn]
    C2Stat *s_stat = reinterpret_cast<C2Stat *>(s_cterm + 16 * P.bn);                                 // [warp][bn / 2]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1;
    const int n0 = (pair % P.tiles_n) * P.bn;                                                         // this pair's column tile

    if (threadIdx.x == 0) {
        for (int s = 0; s < P.stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int b = 0; b < 4; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * kC2EpiWarps); }
        mbar_fence_init();
        tma_prefetch_desc(&P.mapA);
        tma_prefetch_desc(&P.mapB);
        if (P.out) tma_prefetch_desc(&P.mapC);
    }
    if (warp == 1) { tmem_alloc_pair(&tmem_slot, 512); tmem_relinquish_pair(); }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                  // both CTAs' barriers are initialised before either signals the other
    tc_fence_after();
    // (each role waits for the kernels before at its first use of their results: what it needs of the launch's parameters, and the
    // code up to there, has then been fetched)
    const uint32_t tmem_base = tmem_slot;
    bool timed_out = false;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------------------------------------------- TMA producer (both CTAs)
            const uint32_t cg = (uint32_t)P.cg;
            const int n_mine = n0 + (P.bn >> 1) * (int)rank;
            bool waited = false;
            uint32_t s = 0, gph = 1, in_group = 0, group = 0;
            for (int tile = pair; tile < P.tiles_total && !timed_out; tile += P.pairs) {
                const Conv2Box o = conv2_box(P, tile, rank);
                for (int cc = 0; cc < P.cchunks && !timed_out; ++cc)
                    for (int tap = 0; tap < 9; ++tap) {
                        if (in_group == 0 && !mbar_wait(&empty_bar[group], gph)) { timed_out = true; break; }
                        if (++in_group == cg) { in_group = 0; ++group; }
                        uint8_t *sa = smem + (size_t)s * stage_bytes;
                        const uint32_t bar = map_to_cta(&full_bar[s], 0);
                        if (rank == 0) mbar_expect_tx(&full_bar[s], 2u * stage_bytes);
                        const int c0 = cc * 128, r = tap / 3, t = tap - 3 * r;
                        if (!waited) { if (!P.beside) pdl_wait(); waited = true; }
                        // forward: input row p - 1 + r feeds output row p; layer gradient: gradient row h + 1 - r feeds input row h
                        if (!P.dgrad) {
                            tma_load_4d_pair(sa, &P.mapA, bar, c0, o.w0 + t - 1, o.h0 + r - 1, o.img0);
                            tma_load_2d_pair(sa + 16384, &P.mapB, bar, tap * P.C + c0, n_mine);
                        } else {
                            tma_load_4d_pair(sa, &P.mapA, bar, c0, o.w0 + 1 - t, o.h0 + 1 - r, o.img0);
                            tma_load_2d_pair(sa + 16384, &P.mapB, bar, tap * P.C + n_mine, c0);
                        }
                        if (++s == (uint32_t)P.stages) { s = 0; gph ^= 1u; group = 0; }
                    }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------------------------------------------- MMA issuer (leader CTA only): the whole warp in step
            Conv2MmaArgs A;
            A.full_bar = full_bar; A.empty_bar = empty_bar; A.acc_full = acc_full; A.acc_empty = acc_empty;
            A.ring = smem_u32(smem); A.stage_bytes = stage_bytes; A.tmem = tmem_base;
            A.a_desc_lo = P.a_desc_lo; A.b_desc_lo = P.b_desc_lo; A.idesc = P.idesc; A.bn = (uint32_t)P.bn;
            A.k_iters = P.k_iters; A.stages = (uint32_t)P.stages; A.cg = (uint32_t)P.cg; A.nbuf = (uint32_t)P.nbuf;
            A.tile0 = pair; A.tiles_total = P.tiles_total; A.tile_step = P.pairs;
            // (a barrier's wait is bounded: its clock starts once the producer's copies can)
            if (!P.beside) pdl_wait();
            timed_out = !(!P.dgrad ? conv2_mma_loop<2, 128>(A) : P.bn == 256 ? conv2_mma_loop<256, 128>(A) : conv2_mma_loop<128, 64>(A));
        }
    } else {
        // ------------------------------------------------------- epilogue (each CTA drains its own 128 positions; the two groups
        // of four warps split the column chunks)
        const int ew = warp - 2, quad = warp & 3, half = ew >> 2, et = threadIdx.x - 64;
        const int row = quad * 32 + lane, hcols = P.bn >> 1;
        uint8_t *slab = staging + (size_t)ew * kC2Slab;
        pdl_wait();
        const float scale = __fmul_rn(P.qa->scale, P.qb->scale);
        C2Stat *my_stat = s_stat + (size_t)ew * hcols;
        for (int i = et; i < 16 * P.bn; i += 32 * kC2EpiWarps) {
            const int cls = i / P.bn, n = n0 + i - cls * P.bn;
            s_cterm[i] = n < P.N ? load_after_wait(P.colterm + (int64_t)cls * P.N + n) : 0;
        }
        if (P.st_sum)
            for (int i = lane; i < hcols; i += 32) { my_stat[i].sum = 0.0; my_stat[i].lo = INFINITY; my_stat[i].hi = -INFINITY; }
        named_barrier(1, 32 * kC2EpiWarps);
        const uint32_t leader_empty = map_to_cta(&acc_empty[0], 0);          // (8 bytes a barrier)

        // where this thread's accumulator row goes: its position, its border class, its warp's sub-box
        struct RowInfo { int64_t m; bool valid, slab_in; int cls, sx, sy, sz; };
        auto row_info = [&](int tile) {
            const Conv2Box o = conv2_box(P, tile, rank);
            RowInfo ri;
            const int q = o.w0 + (row & ((1 << P.bw_log2) - 1)), p = o.h0 + ((row >> P.bw_log2) & ((1 << P.bh_log2) - 1));
            const int n = o.img0 + (row >> (P.bw_log2 + P.bh_log2));
            ri.valid = n < P.Nimg && p < P.H && q < P.W;
            ri.m = ((int64_t)n * P.H + p) * P.W + q;
            ri.cls = (p == 0 ? 1 : 0) | (p == P.H - 1 ? 2 : 0) | (q == 0 ? 4 : 0) | (q == P.W - 1 ? 8 : 0);
            const int r0 = quad * 32;
            ri.sx = o.w0 + (r0 & ((1 << P.bw_log2) - 1));
            ri.sy = o.h0 + ((r0 >> P.bw_log2) & ((1 << P.bh_log2) - 1));
            ri.sz = o.img0 + (r0 >> (P.bw_log2 + P.bh_log2));
            ri.slab_in = ri.sx < P.W && ri.sy < P.H && ri.sz < P.Nimg;
            return ri;
        };
        const int ncol = P.N - n0 < P.bn ? P.N - n0 : P.bn;                        // columns of this tile inside the matrix
        const int c_begin = half * (hcols >> 5), c_end = min((ncol + 31) >> 5, (half + 1) * (hcols >> 5));
        uint32_t buf = 0, fph = 0;
        RowInfo ri = row_info(pair < P.tiles_total ? pair : 0);
        int rterm = (pair < P.tiles_total && ri.valid) ? load_after_wait(P.rowterm + ri.m) : 0;
        for (int tile = pair; tile < P.tiles_total; tile += P.pairs) {
            // the next tile's row term is fetched now, so that its latency hides behind this tile
            const int tile_next = tile + P.pairs;
            const RowInfo ri_next = row_info(tile_next < P.tiles_total ? tile_next : 0);
            const int rterm_next = (tile_next < P.tiles_total && ri_next.valid) ? load_after_wait(P.rowterm + ri_next.m) : 0;
            const int32_t *cterm = s_cterm + ri.cls * P.bn;
            if (!timed_out && !mbar_wait_warp(&acc_full[buf], fph)) timed_out = true;
            if (!timed_out) {
                tc_fence_after();
                const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + buf * (uint32_t)P.bn;
                if (c_begin >= c_end) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_empty + 8u * buf);
                }
                for (int c = c_begin; c < c_end; ++c) {
                    const int c0 = c * 32;
                    uint32_t r[32];
                    tmem_ld_32x32(t_addr + (uint32_t)c0, r);
                    tmem_ld_wait();
                    if (c == c_end - 1) {
                        // this warp has read its part of the accumulator: tell the leader's MMA thread
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(leader_empty + 8u * buf);
                    }
                    const int lim = ncol - c0 < 32 ? ncol - c0 : 32;
                    int acc[32];
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const int4 ct = *reinterpret_cast<const int4 *>(cterm + c0 + j);
                        acc[j] = (int)r[j] + rterm + ct.x; acc[j + 1] = (int)r[j + 1] + rterm + ct.y;
                        acc[j + 2] = (int)r[j + 2] + rterm + ct.z; acc[j + 3] = (int)r[j + 3] + rterm + ct.w;
                    }
                    if (P.acc_out && ri.valid) {
                        int32_t *dst = P.acc_out + ri.m * P.N + n0 + c0;
                        if (lim == 32) {
#pragma unroll
                            for (int j = 0; j < 32; j += 4)
                                *reinterpret_cast<int4 *>(dst + j) = make_int4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j < lim) dst[j] = acc[j];
                        }
                    }
                    if (!P.out && !P.st_sum) continue;
                    // the store that last used the slab must have read it before it is overwritten
                    if (lane == 0) tma_store_wait_read();
                    __syncwarp();
                    uint8_t *rowp = slab + lane * 128;
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        *reinterpret_cast<float4 *>(rowp + (((j >> 2) ^ (lane & 7)) << 4)) =
                            make_float4(__fmul_rn((float)acc[j], scale), __fmul_rn((float)acc[j + 1], scale),
                                        __fmul_rn((float)acc[j + 2], scale), __fmul_rn((float)acc[j + 3], scale));
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0 && P.out && ri.slab_in) {
                        tma_store_4d(&P.mapC, slab, n0 + c0, ri.sx, ri.sy, ri.sz);
                        tma_store_commit();
                    }
                    if (P.st_sum) {
                        // lane = column of the slab: its 32 rows (the valid ones) read back from shared memory
                        const unsigned vmask = __ballot_sync(0xffffffffu, ri.valid);
                        float cs = 0.0f, clo = INFINITY, chi = -INFINITY;
                        if (vmask == 0xffffffffu) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const uint8_t *colp = slab + k * 128 + ((((lane >> 2) ^ k) << 4) | ((lane & 3) << 2));
#pragma unroll
                                for (int r8 = 0; r8 < 4; r8 += 2) {
                                    const float v0 = *reinterpret_cast<const float *>(colp + r8 * 1024);
                                    const float v1 = *reinterpret_cast<const float *>(colp + (r8 + 1) * 1024);
                                    cs += v0; cs += v1; clo = fmin3(clo, v0, v1); chi = fmax3(chi, v0, v1);
                                }
                            }
                        } else {
#pragma unroll 8
                            for (int k = 0; k < 32; ++k) {
                                if (!((vmask >> k) & 1u)) continue;
                                const float v = *reinterpret_cast<const float *>(slab + k * 128 + ((((lane >> 2) ^ (k & 7)) << 4) | ((lane & 3) << 2)));
                                cs += v; clo = fminf(clo, v); chi = fmaxf(chi, v);
                            }
                        }
                        if (lane < lim && vmask) {
                            C2Stat &a = my_stat[c0 - half * hcols + lane];
                            a.sum += (double)cs; a.lo = fminf(a.lo, clo); a.hi = fmaxf(a.hi, chi);
                        }
                        __syncwarp();                    // (every lane has read the slab before it is filled again)
                    }
                }
            }
            ri = ri_next; rterm = rterm_next;
            if (++buf == (uint32_t)P.nbuf) { buf = 0; fph ^= 1u; }
        }
        if (lane == 0) tma_store_wait_all();
        __syncwarp();
        if (P.st_sum) {
            // the CTA's warps together: one partial row per CTA, the neutral element outside its column tile
            named_barrier(1, 32 * kC2EpiWarps);
            const int64_t prow = (int64_t)blockIdx.x * P.N;
            for (int i = et; i < P.N; i += 32 * kC2EpiWarps) {
                double sum = 0.0; float lo = INFINITY, hi = -INFINITY;
                const int li = i - n0;
                if (li >= 0 && li < P.bn) {
                    const int h = li >= hcols ? 1 : 0;
                    for (int w = 0; w < 4; ++w) {
                        const C2Stat &a = s_stat[(size_t)(4 * h + w) * hcols + li - h * hcols];
                        sum += a.sum; lo = fminf(lo, a.lo); hi = fmaxf(hi, a.hi);
                    }
                }
                P.st_sum[prow + i] = sum; P.st_lo[prow + i] = lo; P.st_hi[prow + i] = hi;
            }
        }
    }

    if (timed_out) {
        pdl_wait();                      // (a launch before may clear the word)
        raise_timeout(P.status);
        __nanosleep(1000000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                  // neither CTA retires while the other may still read its memory or signal it
    if (warp == 1) { __syncwarp(); tmem_dealloc_pair(tmem_base, 512); }
}

// Column tile: 256 channels where that wastes no more columns than 128 and the tiles fill the machine, else 128.
static int conv2_bn(int64_t boxes, int Nout)
{
    const int64_t tiles_m = (boxes + 1) / 2;
    const int t256 = (Nout + 255) / 256, t128 = (Nout + 127) / 128;
    return 2 * t256 <= t128 && tiles_m * t256 >= sm_count() / 2 ? 256 : 128;
}

// Whether the pair kernel takes this product (of a supported convolution).
bool conv2_eligible(const qbp_conv_desc *d, bool dgrad)
{
    const int Cred = dgrad ? d->K : d->C, Nout = dgrad ? d->C : d->K;
    return d->R == 3 && Cred >= 96 && Nout >= 96 && (Nout + 127) / 128 <= sm_count() / 2;
}

int launch_conv2(bool dgrad, const qbp_conv_desc *d, const int8_t *in, const qbp_qparams *q_in, const int8_t *wgt,
                 const qbp_qparams *q_w, int32_t *acc_out, float *out, const int32_t *rowterm, const int32_t *colterm,
                 ColStatParts *stats, int *status, int bwl, int bhl, bool beside, cudaStream_t st)
{
    Conv2Params P{};
    const int Cred = dgrad ? d->K : d->C, Nout = dgrad ? d->C : d->K;
    const int bw = 1 << bwl, bh = 1 << bhl, bimg = 128 >> (bwl + bhl);
    const int tiles_w = (d->W + bw - 1) / bw, tiles_h = (d->H + bh - 1) / bh;
    const int64_t boxes = (int64_t)tiles_w * tiles_h * ((d->N + bimg - 1) / bimg);
    P.dgrad = dgrad ? 1 : 0; P.beside = beside ? 1 : 0;
    P.bn = conv2_bn(boxes, Nout);
    P.nbuf = 512 / P.bn;
    int rc;
    if ((rc = make_map_nhwc(&P.mapA, in, d->N, d->H, d->W, Cred, bimg, bh, bw, 128))) return rc;
    const OperandLayout a = layout_kmajor(128, 128);
    OperandLayout b;
    const uint32_t half = (uint32_t)P.bn / 2;
    if (!dgrad) { b = layout_kmajor(half, 128);         rc = make_map_2d(&P.mapB, wgt, d->K, 9ull * d->C, half, 128); }
    else        { b = layout_mnmajor(128, half, 1, 0);  rc = make_map_2d(&P.mapB, wgt, d->K, 9ull * d->C, 128, half); }
    if (rc) return rc;
    if (out) {
        const uint32_t sw = (uint32_t)std::min(bw, 32), sh = (uint32_t)std::min(bh, 32 / (int)sw), sn = 32 / (sw * sh);
        if ((rc = make_map_out_nhwc(&P.mapC, out, d->N, d->H, d->W, Nout, sn, sh, sw))) return rc;
    }
    P.a_desc_lo = a.desc_lo; P.b_desc_lo = b.desc_lo; P.b_bytes = b.tile_bytes;
    P.idesc = make_idesc(true, true, a.major, b.major, 256, (uint32_t)P.bn);
    P.cchunks = (Cred + 127) / 128; P.k_iters = 9 * P.cchunks;
    P.tiles_m = (int)((boxes + 1) / 2); P.tiles_n = (Nout + P.bn - 1) / P.bn;
    P.tiles_total = P.tiles_m * P.tiles_n;
    P.pairs = std::min(P.tiles_total, sm_count() / 2);
    P.pairs -= P.pairs % P.tiles_n;
    P.d_tiles_n = make_fastdiv(P.tiles_n); P.d_tiles_w = make_fastdiv(tiles_w); P.d_tiles_h = make_fastdiv(tiles_h);
    P.Nimg = d->N; P.H = d->H; P.W = d->W; P.C = d->C; P.N = Nout; P.bw_log2 = bwl; P.bh_log2 = bhl;
    P.acc_out = acc_out; P.out = out; P.rowterm = rowterm; P.colterm = colterm; P.qa = q_in; P.qb = q_w; P.status = status;
    if (stats) { P.st_lo = stats->lo; P.st_hi = stats->hi; P.st_sum = stats->sum; stats->rows = 2 * P.pairs; }
    const uint32_t stage_bytes = 16384u + P.b_bytes;
    const uint32_t fixed = 1024u + kC2EpiWarps * kC2Slab + 16u * (uint32_t)P.bn * 4u + (stats ? kC2EpiWarps * half * (uint32_t)sizeof(C2Stat) : 0u);
    P.cg = P.bn == 256 ? 1 : 2;          // (a commit every 512 cycles of MMAs)
    P.stages = std::min<int>(kC2MaxStages, (int)((kC2Smem - fixed) / stage_bytes));
    P.stages -= P.stages % P.cg;
    const size_t smem = fixed + (size_t)P.stages * stage_bytes;
    static PerDeviceOnce configured;
    QBP_SMEM_OPT_IN(configured, qbp_conv2_kernel, kC2Smem);
    QBP_TRACE_BEGIN(st);
    launch(qbp_conv2_kernel, 2 * P.pairs, kC2Threads, smem, st, P);
    QBP_LAUNCH_OK("qbp_conv2_kernel");
    return QBP_OK;
}

// ============================================== without statistics: channels as the accumulator's rows
// The same products where nobody wants the statistics of their output (layer gradients, the low-bit layer, plain calls).
//
// The accumulator's rows (tensor-memory lanes) are output channels, its columns output positions: the filter is the A operand and
// the activation the B operand.  A tile is 128 channels x npos positions, npos at most 256, on a CTA of its own.  (Pairs of CTAs with
// 256 channels, half of the positions' window each, were hardly faster where the products are long, 60 x 40 x 40, 512 -> 512 channels
// 168 against 170 us, and slower nearly everywhere else, in the mean of 980 shapes by 8 %: 2 x 17 x 17, 256 -> 256 14.9 against 13.1.)
// An epilogue thread then owns a channel: the channel's zero-point term is a register, a position's a broadcast, and a position's 32
// channels of a warp go out as one 128-byte line, where positions as rows stage every value in shared memory beside the operand
// reads and copies that want its port.  (Statistics would stay in registers too, but in sums of other 32 values: the mean's last
// bit changes with their grouping, and chained layers amplify that through their stochastic codes.  They keep the kernel above.)
//
// The positions of all images lie in one row of numbers: an image row takes W + 1 of them and an image H + 1 rows, the last
// column and the last row being padding that the neighbours share, so that the input position of a tap is the output position
// plus a constant.  A CTA's consecutive numbers and their neighbours (its window) are copied once per channel chunk, in boxes of 8,
// 4, 2 and 1 image rows, and a tap's operand is the window read from a shifted start: the shared-memory swizzle is a function of the
// address, so a start at any whole position reads what TMA wrote there.  The padding is then filled with the input's zero-point
// code, so that it adds zero to every corrected sum and one term per channel serves all positions.
// What bounds it: the operand bytes that all SMs together draw from the L2 (some 10 TB/s; 128 filter rows and a ninth of the window
// per tap against 128 + bn / 2 rows above), then the epilogue's instructions; the MMAs of a tile run at the pipe's rate.  Measured
// with the terms' kernel, before and after: 256 x 28 x 28, 128 -> 128 channels 55.7 -> 44.6 us, 8 x 40 x 40, 288 -> 288 37.9 -> 26.2,
// 20 x 19 x 19, 160 -> 96 16.2 -> 12.8, 16 x 7 x 7, 512 -> 512 21.8 -> 17.2, 30 x 17 x 17, 512 -> 512 38.7 -> 29.7.
//
// Roles per CTA: warp 0 copies filter tiles, warp 18 windows, warp 19 fills their padding, warp 1 issues the MMAs, warps 2..17 are
// the epilogue.  Every wait is bounded; no TMA load uses cluster multicast.
constexpr int kCtEpiWarps = 16;                 // (their chains of conversions, stores and comparisons are bound by latency: four warps a scheduler)
constexpr int kCtThreads = 32 * (kCtEpiWarps + 4);
constexpr int kCtMaxStages = 8;
constexpr int kCtMaxWindows = 3;
constexpr int kCtPanelWidth = 96;               // columns of an image taken together at most (two windows must fit)
constexpr int kCtChunks = 4;                    // of 16 positions per epilogue warp and tile, at most
constexpr int kCtBoxHeights = 4;                // windows are copied in boxes of 8, 4, 2 and 1 image rows
constexpr uint32_t kCtTapBytes = 128u * 128u;   // a filter tile of one tap: 128 output x 128 reduction channels
constexpr uint32_t kCtSmem = 225u * 1024u;

// Where a number lies: panels of at most kCtPanelWidth columns of an image follow one another, hp rows of s numbers each.
// One panel: number j of a row is column j, the last one padding.  Several: column first - 1 + j, a neighbour on either side.
struct ConvTGrid {
    int s, hp, np, wp, off;          // numbers per row, rows per panel, panels per image, columns per panel, its first column's j
    int pr, pc;                      // rows / columns on either side that the taps reach (0: one row / column, one tap row / column)
    FastDiv d_s, d_hp, d_np;
    int64_t total;                   // numbers in all
};
struct CtRun { unsigned vmask; int second; int64_t m1, m2; };         // a chunk's positions: see the epilogue
struct CtEpiShared { int32_t term[kCtEpiWarps][kCtChunks][16]; CtRun run[kCtEpiWarps][kCtChunks]; };

struct ConvTParams {
    CUtensorMap mapF, mapX[kCtBoxHeights];     // filter, activation
    uint32_t f_desc_lo, x_desc_lo, idesc;
    uint32_t window_bytes, window_start;       // room of a window; where its first number lies (the row it is in starts up to s - 1 before)
    int dgrad;
    int npos;                        // positions of a tile
    int stages, windows;             // ring stages of a tap row's filter tiles; windows in flight
    int cchunks;                     // channel chunks of 128 (of a ragged last one the rest is zero on the activation side)
    int tiles_n, tiles_total, units; // units (CTAs): a multiple of tiles_n, so that a unit meets one channel tile only
    FastDiv d_tiles_n;
    ConvTGrid g;
    int Nimg, H, W, C, N, Cred;      // C: channels of the filter's innermost extent; N: channels produced
    int32_t *acc_out; float *out;
    const int32_t *rowterm, *colterm;          // [positions], [16 border classes][N]
    const qbp_qparams *qa, *qb;
    int beside;                      // the launch before writes the terms and neither operands nor parameters: only the epilogue waits for it
    int *status;
};

// ---- MMA issue ------------------------------------------------------------------
// The MMA takes its operands from the warp's few uniform registers: what the direction and the operand layouts fix is spelled as
// constants and a tap's MMAs are unrolled.  With a tap's place in the window and in the filter's ring worked out per tap from
// the parameters, four MMAs of 64 cycles took the warp 750.
// The MMAs of one tap, in column T of COLS: 128 reduction channels.
template <bool DGRAD, int T, int COLS, bool FIRST>
__device__ __forceinline__ void convt_issue_tap(uint32_t d_tmem, uint32_t f_lo, uint32_t x_lo, uint32_t idesc)
{
    constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);           // 128-byte swizzle, groups of eight rows 1024 bytes apart
    constexpr uint32_t f_kstep = DGRAD ? 256u : 2u;                           // 32 reduction channels, in 16-byte units: rows of the tile, or inside one
    constexpr uint32_t col = DGRAD ? COLS - 1 - T : T;
#pragma unroll
    for (uint32_t kk = 0; kk < 4; ++kk) {
        const uint64_t f = ((uint64_t)hi << 32) | (uint64_t)(f_lo + T * (kCtTapBytes >> 4) + kk * f_kstep);
        const uint64_t x = ((uint64_t)hi << 32) | (uint64_t)(x_lo + col * 8u + kk * 2u);
        if (elect_one()) mma_i8(d_tmem, f, x, idesc, (FIRST && kk == 0) ? 0u : 1u);
    }
}

struct ConvTMmaArgs {
    uint64_t *full_bar, *empty_bar, *win_full, *win_empty, *acc_full, *acc_empty;
    uint32_t windows_at, window_bytes, window_start, ring, tmem, f_desc_lo, x_desc_lo, idesc;
    int cchunks, tap_rows;
    int tap0, row_step;              // the first tap row's start in the window, from tap row to tap row, in 16-byte units
    uint32_t stages, windows;
    int tile0, tiles_total, tile_step;
};
// False when a wait ran out.
template <bool DGRAD, int COLS>
__device__ __forceinline__ bool convt_mma_loop(const ConvTMmaArgs &A)
{
    constexpr uint32_t stage_bytes = kCtTapBytes * COLS;
    uint32_t s = 0, ph = 0, buf = 0, bph = 1, f_addr = A.ring, win = 0, wph = 0, w_addr = A.windows_at;
    for (int tile = A.tile0; tile < A.tiles_total; tile += A.tile_step) {
        if (!mbar_wait_uniform(&A.acc_empty[buf], bph)) return false;
        tc_fence_after();
        const uint32_t d_tmem = A.tmem + buf * 256u;
        bool first = true;
        for (int cc = 0; cc < A.cchunks; ++cc) {
            if (!mbar_wait_uniform(&A.win_full[win], wph)) return false;
            uint32_t x_lo = ((((w_addr + A.window_start) >> 4) + (uint32_t)A.tap0) & 0x3FFFu) | A.x_desc_lo;
            for (int r = 0; r < A.tap_rows; ++r, x_lo += (uint32_t)A.row_step) {
                const uint32_t f_lo = ((f_addr >> 4) & 0x3FFFu) | A.f_desc_lo;
                if (!mbar_wait_uniform(&A.full_bar[3 * s], ph)) return false;
                tc_fence_after();
                if (first) convt_issue_tap<DGRAD, 0, COLS, true>(d_tmem, f_lo, x_lo, A.idesc);
                else       convt_issue_tap<DGRAD, 0, COLS, false>(d_tmem, f_lo, x_lo, A.idesc);
                first = false;
                if (COLS == 3) {
                    if (!mbar_wait_uniform(&A.full_bar[3 * s + 1], ph)) return false;
                    tc_fence_after();
                    convt_issue_tap<DGRAD, COLS == 3 ? 1 : 0, COLS, false>(d_tmem, f_lo, x_lo, A.idesc);
                    if (!mbar_wait_uniform(&A.full_bar[3 * s + 2], ph)) return false;
                    tc_fence_after();
                    convt_issue_tap<DGRAD, COLS == 3 ? 2 : 0, COLS, false>(d_tmem, f_lo, x_lo, A.idesc);
                }
                if (elect_one()) mma_commit(&A.empty_bar[s]);
                f_addr += stage_bytes;
                if (++s == A.stages) { s = 0; ph ^= 1u; f_addr = A.ring; }
            }
            if (elect_one()) mma_commit(&A.win_empty[win]);
            w_addr += A.window_bytes;
            if (++win == A.windows) { win = 0; wph ^= 1u; w_addr = A.windows_at; }
        }
        if (elect_one()) mma_commit(&A.acc_full[buf]);
        buf ^= 1u;
        if (buf == 0) bph ^= 1u;
    }
    return true;
}

// A position's value under a predicate: stored, and the pointer moved on.
__device__ __forceinline__ void put_if(unsigned cond, uint32_t bits, char *&p, int64_t stride)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p st.global.b32 [%0], %2;\n\t@p add.s64 %0, %0, %3;\n\t}"
                 : "+l"(p) : "r"(cond), "r"(bits), "l"(stride) : "memory");
}

// The image rows (of s numbers, counted through all panels, -1 the one before the first) that a CTA's window of a tile touches.
struct ConvTRows { int first, count, start; };       // start: the window's first number
__device__ __forceinline__ ConvTRows convt_rows(const ConvTParams &P, int tile_m)
{
    ConvTRows w;
    const int reach = P.g.pr * P.g.s + P.g.pc;
    w.start = tile_m * P.npos - reach;
    w.first = P.g.d_s.div(w.start + 2 * P.g.s) - 2;                      // (reach <= 2 s)
    w.count = P.g.d_s.div(w.start + P.npos - 1 + 2 * reach + 2 * P.g.s) - 2 - w.first + 1;
    return w;
}

__global__ void __launch_bounds__(kCtThreads, 1) qbp_conv2t_kernel(const __grid_constant__ ConvTParams P)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[3 * kCtMaxStages], empty_bar[kCtMaxStages], win_landed[kCtMaxWindows], win_full[kCtMaxWindows],
        win_empty[kCtMaxWindows], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;

    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t *windows = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);
    uint8_t *ring = windows + (size_t)P.windows * P.window_bytes;
    const uint32_t stage_bytes = kCtTapBytes * (P.g.pc ? 3u : 1u);
    CtEpiShared &E = *reinterpret_cast<CtEpiShared *>(ring + (size_t)P.stages * stage_bytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int unit = (int)blockIdx.x, n_mine = (unit % P.tiles_n) * 128;                              // this CTA's first channel

    if (threadIdx.x == 0) {
        for (int s = 0; s < P.stages; ++s) { for (int t = 0; t < 3; ++t) mbar_init(&full_bar[3 * s + t], 1); mbar_init(&empty_bar[s], 1); }
        for (int w = 0; w < P.windows; ++w) { mbar_init(&win_landed[w], 1); mbar_init(&win_full[w], 1); mbar_init(&win_empty[w], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], kCtEpiWarps); }
        mbar_fence_init();
        tma_prefetch_desc(&P.mapF);
        for (int b = 0; b < kCtBoxHeights; ++b)
            if ((8 >> b) <= P.H) tma_prefetch_desc(&P.mapX[b]);
    }
    if (warp == 1) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (each role waits for the kernels before at its first use of their results: what it needs of the launch's parameters, and the
    // code up to there, has then been fetched)
    const uint32_t tmem_base = tmem_slot;
    bool timed_out = false;
    // the taps that reach a position: all nine, or of an image of one row or column the middle ones
    const int r0 = P.g.pr ? 0 : 1, r1 = P.g.pr ? 3 : 2, t0 = P.g.pc ? 0 : 1, t1 = P.g.pc ? 3 : 2;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------------------------------------------- TMA producer of the filter tiles
            bool waited = false;
            uint32_t s = 0, ph = 1;
            for (int tile = unit; tile < P.tiles_total && !timed_out; tile += P.units)
                for (int cc = 0; cc < P.cchunks && !timed_out; ++cc)
                    for (int r = r0; r < r1; ++r) {
                        if (!mbar_wait(&empty_bar[s], ph)) { timed_out = true; break; }
                        const int c0 = cc * 128;
                        if (!waited) { if (!P.beside) pdl_wait(); waited = true; }
                        for (int t = t0; t < t1; ++t) {
                            uint8_t *dst = ring + (size_t)s * stage_bytes + (uint32_t)(t - t0) * kCtTapBytes;
                            uint64_t *bar = &full_bar[3 * s + (uint32_t)(t - t0)];
                            mbar_expect_tx(bar, kCtTapBytes);
                            const int at = (3 * r + t) * P.C;
                            const int x = P.dgrad ? at + n_mine : at + c0, y = P.dgrad ? c0 : n_mine;
                            tma_load_2d(dst, &P.mapF, bar, x, y);
                        }
                        if (++s == (uint32_t)P.stages) { s = 0; ph ^= 1u; }
                    }
        }
    } else if (warp == 2 + kCtEpiWarps) {
        // -------------------------------------------------------- windows: a lane copies the rows of a panel
        uint32_t win = 0, ph = 1;
        bool waited = P.beside != 0;
        const int s = P.g.s;
        for (int tile = unit; tile < P.tiles_total && !timed_out; tile += P.units) {
            const ConvTRows w = convt_rows(P, P.d_tiles_n.div(tile));
            const int v0 = P.g.d_hp.div(w.first + P.g.hp) - 1, v1 = P.g.d_hp.div(w.first + w.count - 1 + P.g.hp) - 1;    // panels, -1 the one before the first
            // (the rows behind the panels v0 .. that the window touches are not copied)
            const int padding = P.g.pr ? P.g.d_hp.div(w.first + w.count + P.g.hp) - 1 - v0 : 0;
            const uint32_t bytes = (uint32_t)((w.count - padding) * s) * 128u;
            int img0, panel0;
            P.g.d_np.divmod(v0 + lane + P.g.np, img0, panel0);
            for (int cc = 0; cc < P.cchunks; ++cc) {
                if (!mbar_wait_uniform(&win_empty[win], ph)) { timed_out = true; break; }
                if (!waited) { pdl_wait(); waited = true; }
                uint8_t *base = windows + (size_t)win * P.window_bytes + P.window_start;
                if (lane == 0) mbar_expect_tx(&win_landed[win], bytes);
                __syncwarp();
                for (int v = v0 + lane, img = img0, panel = panel0; v <= v1; v += 32) {
                    if (v != v0 + lane) P.g.d_np.divmod(v + P.g.np, img, panel);
                    int row = max(w.first, v * P.g.hp);
                    const int end = min(w.first + w.count, v * P.g.hp + P.H);
                    for (int b = 0; row < end;) {
                        const int high = 8 >> b;
                        if (row + high > end) { ++b; continue; }
                        tma_load_4d(base + (row * s - w.start) * 128, &P.mapX[b], &win_landed[win], cc * 128, panel * P.g.wp - P.g.off, row - v * P.g.hp, img - 1);
                        row += high;
                    }
                }
                __syncwarp();
                if (++win == (uint32_t)P.windows) { win = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 3 + kCtEpiWarps) {
        // -------------------------------------------------------- the windows' padding, once their copies have landed
        uint32_t win = 0, ph = 0, zz = 0;
        const int s = P.g.s;
        if (!P.beside) pdl_wait();
        zz = ((uint32_t)P.qa->zero_point & 0xFFu) * 0x01010101u;
        for (int tile = unit; tile < P.tiles_total && !timed_out; tile += P.units) {
            const ConvTRows w = convt_rows(P, P.d_tiles_n.div(tile));
            int h0 = 0;
            if (P.g.pr) { int v; P.g.d_hp.divmod(w.first + P.g.hp, v, h0); }
            for (int cc = 0; cc < P.cchunks; ++cc) {
                const uint32_t base = smem_u32(windows) + win * P.window_bytes + P.window_start + (uint32_t)((w.first * s - w.start) * 128);   // of the first row
                const bool ragged = cc * 128 + 128 > P.Cred;
                // 16 bytes of padding (channels beyond the last stay zero): group g of a position's 128 bytes lies at g ^ (its line & 7)
                auto pad = [&](uint32_t line, int group) {
                    uint32_t z = zz;
                    if (ragged && cc * 128 + (group ^ (int)((line >> 7) & 7u)) * 16 >= P.Cred) z = 0u;
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(line + (uint32_t)group * 16u), "r"(z) : "memory");
                };
                if (!mbar_wait_uniform(&win_landed[win], ph)) { timed_out = true; break; }
                // a column of it in every row (of several panels: of the image's first and last) ...
                if (P.g.pc) {
                    uint32_t line = base + (uint32_t)((lane >> 3) * s) * 128u;
                    for (int i = lane >> 3; i < w.count; i += 4, line += 512u * (uint32_t)s) {
                        if (P.g.np == 1) { pad(line + (uint32_t)P.W * 128u, lane & 7); continue; }
                        int v, h, img, panel;
                        P.g.d_hp.divmod(w.first + i + P.g.hp, v, h);
                        P.g.d_np.divmod(v - 1 + P.g.np, img, panel);
                        if (panel == P.g.np - 1) pad(line + (uint32_t)(P.W - panel * P.g.wp + P.g.off) * 128u, lane & 7);
                        if (panel == 0) pad(line, lane & 7);
                    }
                }
                // ... and the row behind every panel
                if (P.g.pr)
                    for (int i = P.H - h0; i < w.count; i += P.g.hp)
                        for (int u = lane; u < 8 * s; u += 32) pad(base + (uint32_t)(i * s + (u >> 3)) * 128u, u & 7);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&win_full[win]);
                if (++win == (uint32_t)P.windows) { win = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------ MMA issuer: the whole warp in step
        ConvTMmaArgs A;
        A.full_bar = full_bar; A.empty_bar = empty_bar; A.win_full = win_full; A.win_empty = win_empty; A.acc_full = acc_full; A.acc_empty = acc_empty;
        A.windows_at = smem_u32(windows); A.window_bytes = P.window_bytes; A.window_start = P.window_start;
        A.ring = smem_u32(ring); A.tmem = tmem_base; A.f_desc_lo = P.f_desc_lo; A.x_desc_lo = P.x_desc_lo; A.idesc = P.idesc;
        A.cchunks = P.cchunks; A.stages = (uint32_t)P.stages; A.windows = (uint32_t)P.windows;
        // forward: input (p - 1 + r, q - 1 + t) feeds output (p, q); layer gradient: gradient (h + 1 - r, w + 1 - t) feeds input (h, w)
        A.tap_rows = r1 - r0;
        A.tap0 = P.dgrad ? 16 * P.g.pr * P.g.s : 0;
        A.row_step = P.dgrad ? -8 * P.g.s : 8 * P.g.s;
        A.tile0 = unit; A.tiles_total = P.tiles_total; A.tile_step = P.units;
        // (a barrier's wait is bounded: its clock starts once the producers' copies can)
        if (!P.beside) pdl_wait();
        const bool ok = t1 - t0 == 1 ? (P.dgrad ? convt_mma_loop<true, 1>(A) : convt_mma_loop<false, 1>(A))
                                     : (P.dgrad ? convt_mma_loop<true, 3>(A) : convt_mma_loop<false, 3>(A));
        timed_out = !ok;
    } else {
        // ------------------------------------------------------- epilogue (each CTA drains its own 128 channels; the four groups
        // of four warps split the chunks of 16 positions)
        const int ew = warp - 2, quad = warp & 3, group = ew >> 2;
        const int ch = n_mine + quad * 32 + lane;
        const bool ch_in = ch < P.N;
        const int chunks = P.npos >> 4, c_begin = chunks * group >> 2, c_end = chunks * (group + 1) >> 2;
        pdl_wait();
        const float scale = __fmul_rn(P.qa->scale, P.qb->scale);
        // (the taps that are left out of an image of one row or column: the border class without them)
        const int cterm = ch_in ? load_after_wait(P.colterm + (int64_t)((P.g.pr ? 0 : 3) | (P.g.pc ? 0 : 12)) * P.N + ch) : 0;
        auto hand_back = [&](uint32_t buf) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        };

        // The positions of this warp's chunks of a tile, two a lane: where they lie in the output (padding: nowhere), their terms.
        // A chunk's positions follow one another in the output, but for a step where a panel's row ends.
        bool valid[2]; int64_t m[2]; int term[2];
        auto look_up = [&](int tile) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                int rem, j, v, h, img, panel;
                const int at = c_begin * 16 + k * 32 + lane;
                P.g.d_s.divmod(P.d_tiles_n.div(tile) * P.npos + at, rem, j);
                P.g.d_hp.divmod(rem, v, h);
                P.g.d_np.divmod(v, img, panel);
                const int q = panel * P.g.wp - P.g.off + j;
                valid[k] = at < c_end * 16 && img < P.Nimg && h < P.H && j >= P.g.off && j < P.g.off + P.g.wp && q < P.W;
                m[k] = ((int64_t)img * P.H + h) * P.W + q;
                term[k] = valid[k] ? load_after_wait(P.rowterm + m[k]) : 0;
            }
        };
        auto put_down = [&]() {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                // (a lane's own chunk is half of the 32 positions)
                const unsigned sixteen = lane & 16 ? 0xffff0000u : 0xffffu;
                const unsigned vmask = __ballot_sync(0xffffffffu, valid[k]) & sixteen;
                const int64_t m1 = __shfl_sync(0xffffffffu, m[k], vmask ? __ffs(vmask) - 1 : lane);
                const unsigned step = __ballot_sync(0xffffffffu, valid[k] && m[k] != m1 + __popc(vmask & ((1u << lane) - 1u))) & sixteen;
                const int second = step ? __ffs(step) - 1 : lane;
                const int64_t m2 = __shfl_sync(0xffffffffu, m[k], second);
                E.term[ew][2 * k + (lane >> 4)][lane & 15] = term[k];
                if ((lane & 15) == 0) E.run[ew][2 * k + (lane >> 4)] = CtRun{lane & 16 ? vmask >> 16 : vmask, step ? second & 15 : 16, m1, m2};
            }
            __syncwarp();
        };
        if (unit < P.tiles_total) { look_up(unit); put_down(); }
        uint32_t buf = 0, fph = 0;
        for (int tile = unit; tile < P.tiles_total; tile += P.units) {
            // (the next tile's terms are fetched now, so that their latency hides behind this tile)
            const int tile_next = tile + P.units;
            if (tile_next < P.tiles_total) look_up(tile_next);
            if (!timed_out && !mbar_wait_warp(&acc_full[buf], fph)) timed_out = true;
            if (!timed_out) {
                tc_fence_after();
                const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + buf * 256u;
                if (c_begin >= c_end) hand_back(buf);
                for (int c = c_begin; c < c_end; ++c) {
                    uint32_t r[16];
                    tmem_ld_32x16(t_addr + (uint32_t)(c * 16), r);
                    const CtRun run = E.run[ew][c - c_begin];
                    const int4 *terms = reinterpret_cast<const int4 *>(E.term[ew][c - c_begin]);
                    tmem_ld_wait();
                    if (c == c_end - 1) hand_back(buf);              // this warp has read its part of the accumulator
                    int acc[16];
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const int4 t = terms[j >> 2];
                        acc[j] = (int)r[j] + t.x + cterm; acc[j + 1] = (int)r[j + 1] + t.y + cterm;
                        acc[j + 2] = (int)r[j + 2] + t.z + cterm; acc[j + 3] = (int)r[j + 3] + t.w + cterm;
                    }
                    // Position by position, under predicates (a branch each took twice the time); a chunk that a panel's row ends in is
                    // gone through twice.
                    const unsigned below = (1u << run.second) - 1u;
                    if (ch_in) {
#pragma unroll 1
                        for (int pass = 0; pass < (run.second < 16 ? 2 : 1); ++pass) {
                            const unsigned mask = pass ? run.vmask & ~below : run.vmask & below;
                            const int64_t at = ((pass ? run.m2 : run.m1) * P.N + ch) * 4, stride = (int64_t)P.N * 4;
                            if (P.acc_out) {
                                char *to = reinterpret_cast<char *>(P.acc_out) + at;
#pragma unroll
                                for (int j = 0; j < 16; ++j) put_if(mask & (1u << j), (uint32_t)acc[j], to, stride);
                            }
                            if (P.out) {
                                char *to = reinterpret_cast<char *>(P.out) + at;
#pragma unroll
                                for (int j = 0; j < 16; ++j) put_if(mask & (1u << j), __float_as_uint(__fmul_rn((float)acc[j], scale)), to, stride);
                            }
                        }
                    }
                }
            }
            __syncwarp();                                            // (every lane has read the terms before they are replaced)
            if (tile_next < P.tiles_total) put_down();
            buf ^= 1u;
            if (buf == 0) fph ^= 1u;
        }
    }

    if (timed_out) {
        pdl_wait();                      // (a launch before may clear the word)
        raise_timeout(P.status);
        __nanosleep(1000000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) { __syncwarp(); tmem_dealloc(tmem_base, 512); }
}

static ConvTGrid convt_grid(const qbp_conv_desc *d)
{
    ConvTGrid g{};
    g.pr = d->H > 1 ? 1 : 0; g.pc = d->W > 1 ? 1 : 0;
    g.np = (d->W + kCtPanelWidth - 1) / kCtPanelWidth; g.wp = (d->W + g.np - 1) / g.np; g.off = g.np > 1 ? 1 : 0;
    g.s = g.np > 1 ? g.wp + 2 : d->W + g.pc; g.hp = d->H + g.pr;
    g.d_s = make_fastdiv(g.s); g.d_hp = make_fastdiv(g.hp); g.d_np = make_fastdiv(g.np);
    g.total = (int64_t)d->N * g.np * g.hp * g.s;
    return g;
}

// The tile's positions.  A model of the launch in cycles per SM, the cheapest wins: rounds of tiles x (taps x chunks x the longest of
// the MMAs (2 cycles per position and tap), the copies (3 per operand row) and shared memory's port (128 bytes a cycle for operand
// reads and copies) + a tile's overhead) + the last tile's epilogue.
static ConvTPlan convt_plan(const qbp_conv_desc *d, const ConvTGrid &g, bool dgrad)
{
    const int Cred = dgrad ? d->K : d->C, Nout = dgrad ? d->C : d->K, cchunks = (Cred + 127) / 128;
    const int cols = g.pc ? 3 : 1, taps = (g.pr ? 3 : 1) * cols, reach = g.pr * g.s + g.pc;
    ConvTPlan best{};
    for (int npos = 256; npos >= 64; npos -= 32) {
        ConvTPlan p{};
        p.npos = npos;
        p.tiles_n = (Nout + 127) / 128;
        if (p.tiles_n > sm_count()) continue;
        const int64_t tiles = (g.total + npos - 1) / npos * p.tiles_n;
        p.units = (int)std::min<int64_t>(tiles, sm_count());
        p.units -= p.units % p.tiles_n;
        p.window_bytes = (uint32_t)align_up(128u * (size_t)(2 * g.s + npos + 2 * reach), 1024);
        const int room = (int)(kCtSmem - 1024u - (uint32_t)align_up(sizeof(CtEpiShared), 256));
        // two windows, or three where they leave the filter's ring three tap rows
        const int stage_bytes = cols * (int)kCtTapBytes;
        p.windows = room - 3 * (int)p.window_bytes >= 3 * stage_bytes ? 3 : 2;
        p.stages = std::min(kCtMaxStages, (room - p.windows * (int)p.window_bytes) / stage_bytes);
        if (p.stages < 2) continue;
        const double rows = 128.0 + (double)(4 * g.s + npos) / taps;
        const double port = (4.0 * (4096.0 + 32.0 * npos) + 128.0 * rows) / 128.0;
        const double stage = std::max({2.0 * npos, 3.0 * rows, port});
        p.cost = (double)((tiles + p.units - 1) / p.units) * (taps * cchunks * stage + 300.0) + 10.0 * npos;
        if (best.cost == 0.0 || p.cost < best.cost) best = p;
    }
    return best;
}

// Whether this kernel takes the product (of a supported convolution; bwl, bhl: log2 of the position box of the kernel above).
// Where that one takes it too, by both models, whose constants were fitted to 1400 shapes of 96 to 512 channels: the rule leaves the
// mean at 0.855 of the kernel above, and 5 shapes of one tile a CTA more than 4 % (at most 11 %) slower than it.  (Cycles by the models,
// here and above, then us: 238 x 17 x 17, 128 -> 160 channels 26.8 K / 24.7 K, 30.1 / 26.9, stays above; 256 x 14 x 14, 256 -> 256
// 40.3 K / 45.6 K, 38.3 / 36.9, stays; 512 x 14 x 14 68.8 K / 91.2 K, 63.3 / 65.1, comes here; 96 x 14 x 14 21.8 / 23.7, comes; 68 x 23 x
// 23, 512 -> 512 96.5 K / 152 K, 70.7 / 83.1, comes.)
bool conv2t_eligible(const qbp_conv_desc *d, bool dgrad, int bwl, int bhl, ConvTPlan &p)
{
    const int Cred = dgrad ? d->K : d->C, Nout = dgrad ? d->C : d->K;
    if (d->R != 3 || Cred < 96 || Nout < 96) return false;
    const ConvTGrid g = convt_grid(d);
    if (g.total >= (1ll << 31) - 4096) return false;
    p = convt_plan(d, g, dgrad);
    if (p.cost <= 0.0 || !conv2_eligible(d, dgrad)) return p.cost > 0.0;
    const int64_t boxes = (int64_t)((d->W + (1 << bwl) - 1) >> bwl) * ((d->H + (1 << bhl) - 1) >> bhl) * ((d->N + (128 >> (bwl + bhl)) - 1) / (128 >> (bwl + bhl)));
    const int bn = conv2_bn(boxes, Nout), tiles_n = (Nout + bn - 1) / bn;
    const int64_t tiles = (boxes + 1) / 2 * tiles_n;
    int64_t pairs = std::min<int64_t>(tiles, sm_count() / 2);
    pairs -= pairs % tiles_n;
    // (forward, columns beyond the last are not fetched; the layer gradient's filter tiles run into the next tap there)
    const double cols = dgrad ? bn : (double)Nout / tiles_n;
    const double above = (double)((tiles + pairs - 1) / pairs) * 9 * ((Cred + 127) / 128) * std::max(2.0 * bn, 3.3 * (128.0 + cols / 2));
    return p.cost < 0.8 * above + 2000.0;
}

int launch_conv2t(bool dgrad, const qbp_conv_desc *d, const int8_t *in, const qbp_qparams *q_in, const int8_t *wgt,
                 const qbp_qparams *q_w, int32_t *acc_out, float *out, const int32_t *rowterm, const int32_t *colterm,
                 const ConvTPlan &p, int *status, bool beside, cudaStream_t st)
{
    ConvTParams P{};
    const int Cred = dgrad ? d->K : d->C, Nout = dgrad ? d->C : d->K;
    P.g = convt_grid(d);
    P.cchunks = (Cred + 127) / 128;
    P.dgrad = dgrad ? 1 : 0; P.beside = beside ? 1 : 0;
    P.npos = p.npos;
    int rc;
    // filter: forward [K x 9 C], rows = output channels (K-major); layer gradient: rows = the reduction, columns = output channels
    if ((rc = make_map_2d(&P.mapF, wgt, d->K, 9ull * d->C, 128, 128))) return rc;
    for (int b = 0; b < kCtBoxHeights; ++b)
        if ((8 >> b) <= d->H && (rc = make_map_nhwc(&P.mapX[b], in, d->N, d->H, d->W, Cred, 1, 8u >> b, (uint32_t)P.g.s, 128))) return rc;
    const OperandLayout f = dgrad ? layout_mnmajor(128, 128, 1, 0) : layout_kmajor(128, 128), x = layout_kmajor(128, 128);
    P.f_desc_lo = f.desc_lo; P.x_desc_lo = x.desc_lo;
    P.idesc = make_idesc(true, true, f.major, x.major, 128, (uint32_t)p.npos);
    P.window_start = 128u * (uint32_t)P.g.s; P.window_bytes = p.window_bytes;
    P.windows = p.windows; P.stages = p.stages;
    P.tiles_n = p.tiles_n; P.units = p.units;
    P.tiles_total = (int)((P.g.total + p.npos - 1) / p.npos) * p.tiles_n;
    P.d_tiles_n = make_fastdiv(P.tiles_n);
    P.Nimg = d->N; P.H = d->H; P.W = d->W; P.C = d->C; P.N = Nout; P.Cred = Cred;
    P.acc_out = acc_out; P.out = out; P.rowterm = rowterm; P.colterm = colterm; P.qa = q_in; P.qb = q_w; P.status = status;
    const size_t smem = 1024u + (size_t)p.windows * p.window_bytes + (size_t)p.stages * (P.g.pc ? 3 : 1) * kCtTapBytes + sizeof(CtEpiShared);
    static PerDeviceOnce configured;
    QBP_SMEM_OPT_IN(configured, qbp_conv2t_kernel, kCtSmem);
    QBP_TRACE_BEGIN(st);
    launch(qbp_conv2t_kernel, p.units, kCtThreads, smem, st, P);
    QBP_LAUNCH_OK("qbp_conv2t_kernel");
    return QBP_OK;
}

}  // namespace qbp
