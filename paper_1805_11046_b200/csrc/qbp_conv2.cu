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

}  // namespace qbp
