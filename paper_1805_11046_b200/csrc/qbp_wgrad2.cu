// The dense weight gradient g_W = g_l I_{l-1}^T (Eq. (grad_weight)) on CTA pairs: tcgen05.mma.cta_group::2.
//
// dW [K x N] = X [M x K]^T G16 [M x N] with the 16-bit gradient as two byte limbs (G16 = 256 * hi + lo): two
// products per pair tile, X^T hi (s8 x s8) and X^T lo (s8 x u8), each into its own int32 accumulator, combined
// exactly in int64 in the epilogue.  The reduction runs over the M rows, so both operands are M/N-major in shared
// memory (TMA boxes [reduction rows x columns]).
//
// Two CTAs of a cluster compute one 256 x 256 output tile (or a narrower one, see launch_wgrad2): CTA r holds columns [128 r, 128 r + 128) of the X block
// (= output rows) and columns [128 r, 128 r + 128) of both limb blocks, and the accumulators of its 128 output rows
// (256 columns of the high product, 256 of the low one: all 512 columns of its tensor memory).  One thread of the
// leader issues every MMA; against the single-CTA kernel (256 x 128 tiles) each SM fetches a third fewer operand
// bytes per multiply-add and issues half the instructions.  A pair reduces all M rows of its tile, M <= 65536
// (the low limb's int32 bound, 128 * 255 * rows < 2^31), so nothing is split and no second kernel is needed:
// the epilogue applies the zero-point terms, the scale and stores.
//
// Roles per CTA: warp 0 loads this CTA's operand parts by TMA and reports them to the leader's "full" barrier;
// warp 1 allocates tensor memory (both CTAs) and, in the leader, issues the MMAs and releases stages with a commit
// that arrives in both CTAs; warps 2..9 drain this CTA's accumulator rows.  Every wait is bounded; on expiry the
// CTA raises the status word and leaves through the normal exit.  No TMA load here uses cluster multicast.
#include "qbp_mma.cuh"
#include "qbp_pair.cuh"

#include <algorithm>
#include <type_traits>

namespace qbp {

constexpr int kW2Threads = 320;
constexpr int kW2EpiWarps = 8;
constexpr int kW2MaxStages = 8;                 // of 24, 32 or 48 KB: 128 reduction rows x (128 X + bn / 2 hi + bn / 2 lo columns)
constexpr uint32_t kW2Ring = 192u * 1024u;
constexpr int kW2Cg = 2;                        // stages released per commit
constexpr int kW2GroupM = 8;
constexpr uint32_t kW2Slab = 32 * 128;
constexpr uint32_t kW2XBytes = 128u * 128u;
constexpr uint32_t kW2Smem = 1024u + kW2Ring + kW2EpiWarps * kW2Slab;

struct Wgrad2Params {
    CUtensorMap mapX, mapHi, mapLo, mapC;
    uint32_t x_desc_lo, g_desc_lo;   // descriptor bits 16..31 of the M/N-major tiles of 128 and of bn / 2 columns
    uint32_t idesc_hi;               // s8 x s8, M = 256, N = bn, both operands M/N-major
    uint32_t lo_flip;                // the low limb's descriptor = idesc_hi ^ lo_flip: the B sign bit for unsigned low bytes, 0 for lo - 128
    int bn, stages;                  // columns of a pair tile (256, 128 or 64); ring stages
    uint32_t stage_bytes;
    int k_iters;                     // reduction steps of 128 rows
    int tiles_m, tiles_n, tiles_total, pairs;
    FastDiv d_group;
    int64_t M, N, K;                 // reduction rows; output columns; output rows
    long long *acc_out; float *dW;
    CodeSums sx, shi, slo;           // code sums over the M rows: rowterm = -zg * sx[k] + M * zx * zg, colterm = -zx * (256 * shi[n] + slo[n])
    const long long *tot_g;          // [N]: totals of 256 * hi + (unsigned low byte) over the rows, in place of shi and slo (NULL: not there)
    int beside;                      // the launch before makes the code sums: only the epilogue waits for it
    int zg_shift;                    // 128 for signed low bytes (lo - 128 against zg - 128)
    const qbp_qparams *qx, *qg;
    int *status;
};

// The eight pair MMAs of a stage (128 reduction rows = four k steps per limb), the limb outermost: switching
// between the two instruction descriptors stalls the MMA pipe.  Offsets in 16-byte units: 256 per k step of an
// M/N-major 128-byte-row tile, 2 RB of one of RB columns (bn / 2) of a limb, 8 RB per limb tile; the upper descriptor word is the
// swizzle of that many bytes and groups of eight rows.
template <uint32_t RB, bool FIRST>
__device__ __forceinline__ void w2_issue_stage(uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc_hi, uint32_t lo_flip)
{
    constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t g_hi = ((8u * RB) >> 4) | (1u << 14) | ((RB == 128 ? 2u : RB == 64 ? 4u : 6u) << 29);
    const uint32_t idesc_lo = idesc_hi ^ lo_flip;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int limb = i >> 2, kk = i & 3;
        if (elect_one())
            mma_i8_pair(tmem + 256u * (uint32_t)limb, ((uint64_t)hi << 32) | (uint64_t)(a_lo + (uint32_t)kk * 256u),
                   ((uint64_t)g_hi << 32) | (uint64_t)(b_lo + (uint32_t)limb * (8u * RB) + (uint32_t)kk * (2u * RB)),
                   limb ? idesc_lo : idesc_hi, (FIRST && kk == 0) ? 0u : 1u);
    }
}

struct W2Tile { int k0, n0; };
__device__ __forceinline__ W2Tile w2_tile(const Wgrad2Params &P, int tile)
{
    int g, r, tile_m, tile_n;
    P.d_group.divmod(tile, g, r);                        // by kW2GroupM * tiles_n
    const int rows_here = min(kW2GroupM, P.tiles_m - g * kW2GroupM);
    if (rows_here == kW2GroupM) { tile_n = r / kW2GroupM; tile_m = g * kW2GroupM + r % kW2GroupM; }
    else                        { tile_n = r / rows_here; tile_m = g * kW2GroupM + r % rows_here; }
    W2Tile t; t.k0 = tile_m * 256; t.n0 = tile_n * P.bn;
    return t;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kW2Threads, 1) qbp_wgrad2_kernel(const __grid_constant__ Wgrad2Params P)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kW2MaxStages], empty_bar[kW2MaxStages], acc_full, acc_empty;
    __shared__ uint32_t tmem_slot;

    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);
    uint8_t *staging = smem + kW2Ring;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        // "full": the leader's arrive + the bytes of both CTAs; "empty": one multicast commit per stage group;
        // "acc_full": one multicast commit per tile; "acc_empty" (the leader's is waited on): 8 warps of each CTA
        for (int s = 0; s < kW2MaxStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&acc_full, 1); mbar_init(&acc_empty, 2 * kW2EpiWarps);
        mbar_fence_init();
        tma_prefetch_desc(&P.mapX); tma_prefetch_desc(&P.mapHi); tma_prefetch_desc(&P.mapLo);
        if (P.dW) tma_prefetch_desc(&P.mapC);
    }
    if (warp == 1) { tmem_alloc_pair(&tmem_slot, 512); tmem_relinquish_pair(); }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                   // both CTAs' barriers are initialised before either signals the other
    tc_fence_after();
    // (each role waits for the kernels before at its first use of their results: what it needs of the launch's parameters, and the
    // code up to there, has then been fetched)
    const uint32_t tmem_base = tmem_slot;
    bool timed_out = false;

    if (warp == 0) {
        if (lane == 0) {
            // ---------------------------------------------------- TMA producer (both CTAs)
            bool waited = false;
            uint32_t s = 0, gph = 1, in_group = 0, group = 0;
            for (int tile = pair; tile < P.tiles_total && !timed_out; tile += P.pairs) {
                const W2Tile o = w2_tile(P, tile);
                const int k_mine = o.k0 + 128 * (int)rank, n_mine = o.n0 + (P.bn >> 1) * (int)rank;
                for (int it = 0; it < P.k_iters; ++it) {
                    if (in_group == 0 && !mbar_wait(&empty_bar[group], gph)) { timed_out = true; break; }
                    if (++in_group == (uint32_t)kW2Cg) { in_group = 0; ++group; }
                    uint8_t *sa = smem + (size_t)s * P.stage_bytes;
                    const uint32_t bar = map_to_cta(&full_bar[s], 0);
                    if (rank == 0) mbar_expect_tx(&full_bar[s], 2u * P.stage_bytes);
                    const int m0 = it * 128;
                    if (!waited) { if (!P.beside) pdl_wait(); waited = true; }
                    tma_load_2d_pair(sa, &P.mapX, bar, k_mine, m0);
                    tma_load_2d_pair(sa + kW2XBytes, &P.mapHi, bar, n_mine, m0);
                    tma_load_2d_pair(sa + kW2XBytes + 64 * P.bn, &P.mapLo, bar, n_mine, m0);
                    if (++s == (uint32_t)P.stages) { s = 0; gph ^= 1u; group = 0; }
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------------------------------------------- MMA issuer (leader CTA only): the whole warp in step
            // (a barrier's wait is bounded: its clock starts once the producer's copies can)
            if (!P.beside) pdl_wait();
            const auto issue = [&](auto columns) {
                constexpr uint32_t RB = decltype(columns)::value;
                uint32_t s = 0, ph = 0, in_group = 0, group = 0, eph = 1;
                const uint32_t ring = smem_u32(smem);
                uint32_t a_addr = ring;
                for (int tile = pair; tile < P.tiles_total; tile += P.pairs) {
                    if (!mbar_wait_uniform(&acc_empty, eph)) return false;
                    eph ^= 1u;
                    tc_fence_after();
                    for (int it = 0; it < P.k_iters; ++it) {
                        if (!mbar_wait_uniform(&full_bar[s], ph)) return false;
                        tc_fence_after();
                        const uint32_t a_lo = ((a_addr >> 4) & 0x3FFFu) | P.x_desc_lo;
                        const uint32_t b_lo = (((a_addr + kW2XBytes) >> 4) & 0x3FFFu) | P.g_desc_lo;
                        if (it == 0) w2_issue_stage<RB, true>(tmem_base, a_lo, b_lo, P.idesc_hi, P.lo_flip);
                        else         w2_issue_stage<RB, false>(tmem_base, a_lo, b_lo, P.idesc_hi, P.lo_flip);
                        if (++in_group == (uint32_t)kW2Cg) {
                            if (elect_one()) mma_commit_pair(&empty_bar[group]);
                            in_group = 0; ++group;
                        }
                        a_addr += P.stage_bytes;
                        if (++s == (uint32_t)P.stages) { s = 0; ph ^= 1u; group = 0; a_addr = ring; }
                    }
                    if (elect_one()) mma_commit_pair(&acc_full);
                }
                return true;
            };
            timed_out = !(P.bn == 256 ? issue(std::integral_constant<uint32_t, 128>{})
                          : P.bn == 128 ? issue(std::integral_constant<uint32_t, 64>{}) : issue(std::integral_constant<uint32_t, 32>{}));
        }
    } else {
        // ------------------------------------------------------- epilogue (each CTA drains its own 128 output rows)
        // the two groups of four warps split the column chunks of 32
        const int ew = warp - 2, quad = warp & 3, half = ew >> 2, per_group = P.bn >> 6;
        const int row = quad * 32 + lane;
        uint8_t *slab = staging + (size_t)ew * kW2Slab;
        pdl_wait();
        const float scale = __fmul_rn(P.qx->scale, P.qg->scale);
        const long long zx = P.qx->zero_point, zg = P.qg->zero_point - P.zg_shift;
        const uint32_t leader_empty = map_to_cta(&acc_empty, 0);
        uint32_t fph = 0;
        for (int tile = pair; tile < P.tiles_total; tile += P.pairs) {
            const W2Tile o = w2_tile(P, tile);
            const int64_t k = (int64_t)o.k0 + 128 * (int)rank + row;                  // output row
            const bool valid = k < P.K;
            const bool slab_in = (int64_t)o.k0 + 128 * (int)rank + quad * 32 < P.K;
            const long long rterm = valid ? -zg * P.sx.at(k) + P.M * zx * zg : 0;
            const int64_t ncol = P.N - o.n0;
            // lane l takes the column terms of column l of this warp's four chunks, while the MMAs run (the sums come in pieces:
            // two pieces of all eight sums are in flight at a time -- one sum after the other took up to 64 us a tile)
            long long ct[4] = {0, 0, 0, 0};
            const int32_t *ph = P.shi.p + o.n0 + half * per_group * 32 + lane, *pl = P.slo.p + o.n0 + half * per_group * 32 + lane;
            if (P.tot_g) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < per_group && (half * per_group + i) * 32 + lane < ncol) ct[i] = P.tot_g[o.n0 + (half * per_group + i) * 32 + lane] - P.zg_shift * P.M;
            } else
#pragma unroll 2
            for (int k = 0; k < P.shi.pieces; ++k) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < per_group && (half * per_group + i) * 32 + lane < ncol) ct[i] += 256 * (long long)load_after_wait(ph + 32 * i) + load_after_wait(pl + 32 * i);
                ph += P.shi.stride; pl += P.slo.stride;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) ct[i] *= -zx;
            const int nchunks = (int)((ncol < P.bn ? ncol : P.bn) + 31) / 32;
            if (!timed_out && !mbar_wait_warp(&acc_full, fph)) timed_out = true;
            fph ^= 1u;
            if (!timed_out) {
                tc_fence_after();
                const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
                const int c_begin = half * per_group, c_end = min(nchunks, (half + 1) * per_group);
                if (c_begin >= c_end) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_empty);
                }
                for (int c = c_begin; c < c_end; ++c) {
                    const int c0 = c * 32;
                    uint32_t rh[32], rl[32];
                    tmem_ld_32x32(t_addr + (uint32_t)c0, rh);
                    tmem_ld_32x32(t_addr + 256u + (uint32_t)c0, rl);
                    tmem_ld_wait();
                    if (c == c_end - 1) {
                        // this warp has read its part of the accumulators: tell the leader's MMA warp
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(leader_empty);
                    }
                    const int lim = (int)(ncol - c0 < 32 ? ncol - c0 : 32);
                    // (lane l holds the column term of column c0 + l; the row's 32 sums take them by shuffle)
                    const int ci = c - c_begin;
                    const long long my_cterm = ci == 0 ? ct[0] : ci == 1 ? ct[1] : ci == 2 ? ct[2] : ct[3];
                    if (P.dW) {
                        if (lane == 0) tma_store_wait_read();
                        __syncwarp();
                    }
                    uint8_t *rowp = slab + lane * 128;
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        long long a4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            a4[e] = 256ll * (long long)(int)rh[j + e] + (long long)(int)rl[j + e] + rterm +
                                    __shfl_sync(0xffffffffu, my_cterm, j + e);
                        if (P.acc_out && valid) {
                            long long *dst = P.acc_out + k * P.N + o.n0 + c0 + j;
                            if (j + 4 <= lim) {
                                *reinterpret_cast<longlong2 *>(dst) = make_longlong2(a4[0], a4[1]);
                                *reinterpret_cast<longlong2 *>(dst + 2) = make_longlong2(a4[2], a4[3]);
                            } else {
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    if (j + e < lim) dst[e] = a4[e];
                            }
                        }
                        if (P.dW)
                            *reinterpret_cast<float4 *>(rowp + (((j >> 2) ^ (lane & 7)) << 4)) =
                                make_float4(__fmul_rn((float)a4[0], scale), __fmul_rn((float)a4[1], scale),
                                            __fmul_rn((float)a4[2], scale), __fmul_rn((float)a4[3], scale));
                    }
                    if (P.dW) {
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0 && slab_in) {
                            tma_store_2d(&P.mapC, slab, o.n0 + c0, o.k0 + 128 * (int)rank + quad * 32);
                            tma_store_commit();
                        }
                    }
                }
            }
        }
        if (lane == 0) tma_store_wait_all();
        __syncwarp();
    }

    if (timed_out) {
        pdl_wait();                       // (the launch before may clear the word)
        raise_timeout(P.status);
        __nanosleep(1000000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                   // neither CTA retires while the other may still read its memory or signal it
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// Columns of a pair tile: where tiles of 256 fit the pairs once, half as many (64 at least) as long as they do: rings and epilogues get
// shorter, and SMs that had none take part.  Call with its sums, 256 columns -> by this rule: 1024 rows for 2048 x 1008 18.3 ->
// 15.6 us, 4096 for 1024 x 1024 31.7 -> 24.1, 16384 for 256 x 512 84.9 -> 57.0.  And never wider than the columns there are, also
// where the row tiles alone do not fit: 4096 rows for 20000 x 128 68.4 -> 54.7 (single-CTA kernel 52.3), 1024 for 65536 x 128
// 55.9 -> 44.3 (49.3), 8192 for 65536 x 64 264 -> 216 (200)
static int w2_columns(int64_t N, int64_t K)
{
    const int64_t tiles_m = (K + 255) / 256;
    int bn = 256;
    while (bn > 64 && (N <= bn / 2 || tiles_m * ((N + bn / 2 - 1) / (bn / 2)) <= sm_count() / 2)) bn /= 2;
    return bn;
}

// Whether the pair kernel takes this plain product: a reduction that one pair can hold in int32, and one of (call with its sums, first
// with the single-CTA kernel, then with this one)
//   - fewer than 512 rows (or 640): large outputs (64 rows for 2048 x 2048: 15.7 and 13.3 us; not 384 for 256 x 256: 9.2 and 9.6, nor
//     539 for 192 x 672: 9.7 and 10.4);
//   - more: where the longer walk of a pair over all rows, about 2.9 us per 1000, costs less than the single-CTA kernel's
//     partial sums, about 1 us per 10000 outputs (8192 rows for 4096 x 128: 68.9 and 39.6, 2048 for 1024 x 208: 35.2 and 16.3; not
//     512 for 128 x 128: 9.1 and 9.4, 8192 for 128 x 128: 20.5 and 31.9, 65536 for 256 x 256: 49.6 and 228).
//   - and not where its tiles stay 256 columns wide although 128 x 128 tiles of the other kernel fit the SMs once: those leave half as
//     much to read out per CTA, on nearly all SMs (558 rows for 1568 x 1328: 14.2 and 16.8, 16 for 1568 x 1296 11.2 and 13.2, 1162 for
//     832 x 2480 18.6 and 20.8).
bool wgrad2_eligible(int64_t M, int64_t N, int64_t K)
{
    if (M > 65536 || N < 64 || K < 64) return false;
    if (N * K < (M < 512 ? 1 << 20 : M < 640 ? 1 << 18 : 1 << 15) || (M >= 512 && 29 * M > 30000 + N * K)) return false;
    const bool once = (K + 255) / 256 * ((N + 255) / 256) <= sm_count() / 2;
    return !(once && w2_columns(N, K) == 256 && (K + 127) / 128 * ((N + 127) / 128) <= sm_count());
}

int launch_wgrad2(int64_t M, int64_t N, int64_t K, const int8_t *x, const qbp_qparams *qx, const int8_t *g_hi,
                  const uint8_t *g_lo, const qbp_qparams *qg16, int64_t *acc_out, float *dW, const CodeSums &sx,
                  const CodeSums &shi, const CodeSums &slo, const int64_t *tot_g, int *status, bool beside, cudaStream_t st, bool lo_signed)
{
    Wgrad2Params P{};
    int rc;
    P.bn = w2_columns(N, K);
    P.tiles_m = (int)((K + 255) / 256); P.tiles_n = (int)((N + P.bn - 1) / P.bn);
    P.tiles_total = P.tiles_m * P.tiles_n;
    // per-CTA operand parts: 128 reduction rows x 128 columns of X, x bn / 2 of each limb, M/N-major
    const uint32_t half = (uint32_t)P.bn / 2;
    if ((rc = make_map_2d(&P.mapX, x, M, K, 128, 128))) return rc;
    if ((rc = make_map_2d(&P.mapHi, g_hi, M, N, 128, half))) return rc;
    if ((rc = make_map_2d(&P.mapLo, g_lo, M, N, 128, half))) return rc;
    if (dW && (rc = make_map_out_2d(&P.mapC, dW, K, N))) return rc;
    P.x_desc_lo = layout_mnmajor(128, 128, 1, 0).desc_lo; P.g_desc_lo = layout_mnmajor(128, half, 1, 0).desc_lo;
    P.idesc_hi = make_idesc(true, true, 1, 1, 256, (uint32_t)P.bn);
    P.lo_flip = lo_signed ? 0u : (1u << 10);
    P.stage_bytes = kW2XBytes + 2u * 128u * half;
    P.stages = (int)(kW2Ring / P.stage_bytes);            // 4, 6 or 8: a multiple of kW2Cg
    P.k_iters = (int)((M + 127) / 128);
    P.pairs = std::min(P.tiles_total, sm_count() / 2);
    P.d_group = make_fastdiv(kW2GroupM * P.tiles_n);
    P.M = M; P.N = N; P.K = K;
    P.acc_out = (long long *)acc_out; P.dW = dW;
    P.beside = beside ? 1 : 0; P.tot_g = (const long long *)tot_g; P.sx = sx; P.shi = shi; P.slo = slo; P.zg_shift = lo_signed ? 128 : 0; P.qx = qx; P.qg = qg16; P.status = status;
    static PerDeviceOnce configured;
    QBP_SMEM_OPT_IN(configured, qbp_wgrad2_kernel, kW2Smem);
    QBP_TRACE_BEGIN(st);
    launch(qbp_wgrad2_kernel, 2 * P.pairs, kW2Threads, kW2Smem, st, P);
    QBP_LAUNCH_OK("qbp_wgrad2_kernel");
    return QBP_OK;
}

}  // namespace qbp
