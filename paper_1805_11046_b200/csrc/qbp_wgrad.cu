// Weight gradient g_W = g_l I_{l-1}^T (Eq. (grad_weight)) from the 16-bit copy
// of the layer gradient and the 8-bit layer input (Sections 6, 7), on the
// int8 tensor cores.
//
// The 16-bit code is split into a signed high byte and an unsigned low byte,
// g16 = 256*hi + lo, so that  sum x*g16 = 256 * sum x*hi + sum x*lo  with two
// tcgen05.mma kind::i8 products (s8 x s8 and s8 x u8) into two int32
// accumulators in tensor memory.  The reduction runs over the batch rows
// (batch x spatial positions for a convolution): both operands are therefore
// "M/N-major" in shared memory -- the TMA box is [reduction rows x channels].
// A CTA reduces at most 65536 rows (128*255*65536 < 2^31 bounds the low limb,
// 128*128*65536 the high one) and combines its two accumulators exactly in
// int64.  Integer addition is order-free, so the split of the reduction over
// CTAs does not change the result.
//
// Work split: an item is (group of up to `ma` accumulator tiles of 128 output
// rows, tile of bn output columns); the reduction of an item is cut into
// slices in proportion to the item's cost per reduction step, so that one
// wave of CTAs finishes together.  A CTA that owns a whole reduction applies
// the zero-points and the scale itself; otherwise the CTAs write int64
// partials and a second kernel adds them up.
//
// Convolution: the MMA's 128 rows hold `chunks` filter taps x the input
// channels of one tap (2 taps x 64 channels, or 1 tap x 128 channels); each
// tap is its own TMA load of the input, shifted by the tap offset, padding
// zero-filled.  Zero-points are applied afterwards from the operands' code sums
// and those of the images' edges (a tap near the border sees fewer positions).
//
// The TMA-issuing lanes run from a small table built once per CTA (one entry per load of a stage); the MMA warp
// runs whole with an elected issuer and the stage's MMAs fully unrolled for the operand layouts (see
// wg_issue_stage); stages are released in groups: a tcgen05.commit drains the MMA pipeline, which short MMAs
// cannot afford often.
#include "qbp_mma.cuh"

#include <algorithm>

namespace qbp {

constexpr int kWgThreads = 192;
constexpr int kWgFinalizeLanes = 4;   // lanes of the second kernel that share one output element's partials
constexpr int kWgRows = 128;         // reduction rows per pipeline stage: four k steps of 32 (what the MMA warp does
                                     // between stages is a fixed cost, so a stage should hold many MMAs)
constexpr int kWgMaxStages = 16;
constexpr int kWgMaxTiles = 4;       // A tiles (128 accumulator rows each) per CTA: 4 x 2 limbs x 64 columns fill tensor memory
constexpr int kWgMaxLoads = 32;      // TMA loads per stage: one lane each
constexpr uint32_t kWgSmem = 220u * 1024u;

struct WgradParams {
    CUtensorMap mapX, mapHi, mapLo;
    OperandLayout a, b;
    uint32_t idesc_hi, idesc_lo;
    // The low bytes stored as lo - 128 (signed): both limbs have one operand type, and a stage's MMAs take the high
    // and the low tile side by side as one B operand of 2 * bn columns (the x tile is then read from shared memory
    // once instead of once per limb).  g16 - zg = 256 * hi + (lo - 128) - (zg - 128): everything downstream works on
    // those limbs with the zero-point zg - 128.
    int lo_signed;
    uint32_t b2_desc_lo, idesc_fused;
    int tot_g_plain;                 // tot_g holds totals of 256 * hi + lo (left by a quantiser), not of the stored limbs
    // 3 x 3 convolution from halo tiles (with lo_signed): a stage holds the pixel box of x once, with its border of
    // one position (10 positions per box row), instead of one shifted copy per tap; a tap's operand is that tile read
    // from a shifted start (see wg_issue_stage_halo).  halo_bh: box rows per image in a stage (8 or 4; 0: not used).
    int halo_bh;
    uint32_t halo_bytes;             // the tile's room in a stage (1024-byte multiple)
    uint32_t halo_box_bytes;         // bytes one load of it brings
    uint32_t ones_off;               // offset (from the ring's start) of a region of halo_bytes filled with the code 1
    uint32_t a_chunk_bytes;          // bytes of one A chunk (kr rows x rb_a)
    int conv;                        // 0: x [M x K], g [M x N]; 1: NHWC tensors
    int stages, cg, bn, tmem_cols;   // cg: stages released by one commit
    int stages_last, cg_last;        // the ring of the CTAs of the last A group (fewer A tiles: smaller and more stages)
    int kr;                          // reduction rows per pipeline stage
    int a_chunks, rb_a;              // chunks per A tile, bytes (= channels / columns) per chunk row
    int ma;                          // A tiles per CTA (they share the g tiles of a stage)
    int a_tiles;                     // A tiles in all: plain K/128; conv tap groups x channel tiles
    int a_groups;                    // ceil(a_tiles / ma)
    int tiles_c;                     // conv: channel tiles per tap group
    int tiles_b;                     // output-channel (N) tiles of bn
    int iters_total;                 // reduction steps of kr rows each
    int s_full, s_last;              // slices of an item of a full A group / of the last (possibly smaller) group
    int ctas_full;                   // CTAs working on full groups: (a_groups - 1) * tiles_b * s_full
    int direct;                      // every item is one slice: the CTA finishes its outputs itself (plain only)
    // conv geometry
    int H, W, Nimg, pad, R, S, C, taps;
    int bw_log2, bh_log2, tiles_w, tiles_h;
    FastDiv d_tiles_w, d_tiles_h;
    // plain geometry
    int64_t M, N, K;
    long long *part;                 // int64 partials, one block of part_stride values per CTA
    int64_t part_stride;             // ma * 128 * bn, padded
    // plain product: code sums over the M rows, in pieces or (cx set) as for a convolution (acc = raw - zg * sx[k] - zx * (256 * shi[n] + slo[n]) + M * zx * zg)
    CodeSums sx, shi, slo;
    // over all positions ([C], [N], [N]); convolution: and over the edges of the images ([8][...], see kSumEdges)
    const long long *cx, *chi, *clo, *ex, *ehi, *elo;
    const qbp_qparams *qx, *qg;
    long long *acc_out; float *dW;
    int dW_vec;                      // dW starts on a 16-byte boundary
    int *status;
    // Convolution: per-channel totals of the stored codes over all positions (x: [C]; the 16-bit gradient codes
    // 256 * hi + lo: [N]) that the kernels which wrote the codes left; NULL: cx / chi / clo hold them.
    const long long *tot_x, *tot_g;
    // The gradient's per-channel totals from the product itself: when the taps do not fill the last A tile, its first
    // spare chunk is filled with the code 1 once (nothing else writes there), so that the first accumulator row of
    // that chunk is sum over all positions of 1 * g -- MMA rows that were computed and thrown away before.  The
    // epilogue adds that row into ones_tot [N] (zeroed beforehand).  NULL: not used.
    unsigned long long *ones_tot;
};

// A plain product: the sum of a gradient column's codes as the limbs are stored.
__device__ __forceinline__ long long wg_plain_sum_g(const WgradParams &P, int n)
{
    if (P.tot_g) return P.tot_g[n] - (P.lo_signed ? 128 * P.M : 0);
    return P.cx ? 256 * P.chi[n] + P.clo[n] : 256 * P.shi.at(n) + P.slo.at(n);
}

// Which item and slice a CTA works on.
struct WgItem { int ag, tb, slice, slices; };

__device__ __forceinline__ WgItem wg_item(const WgradParams &P, int bid)
{
    WgItem w;
    int item;
    if (bid < P.ctas_full) { item = bid / P.s_full; w.slice = bid % P.s_full; w.slices = P.s_full; }
    else {
        const int r = bid - P.ctas_full;
        item = P.ctas_full / P.s_full + r / P.s_last; w.slice = r % P.s_last; w.slices = P.s_last;
    }
    w.ag = item / P.tiles_b; w.tb = item % P.tiles_b;
    return w;
}

// ---- MMA issue ------------------------------------------------------------------
// The MMA takes its operands from the warp's few uniform registers.  What the operand layouts (row bytes RBA of the
// x chunks, RBB of the gradient tiles = output columns per tile) and the number NT of A tiles fix is therefore
// spelled as constants and the MMAs of a stage are fully unrolled: descriptors that were looked up per MMA, or
// built from many run-time values, cost 110 to 150 cycles per MMA against 40 to 50 this way.
struct WgMmaArgs {
    uint64_t *full_bar, *empty_bar, *acc_bar;
    uint32_t ring, stage_bytes, a_bytes, tmem;
    int k_iters;
    uint32_t stages, cg;
    uint32_t a_desc_lo, b_desc_lo, idesc_hi;
    // halo tiles: per A tile of the CTA, (start of its first tap in the halo tile) >> 4 | (distance to its second
    // tap) >> 4 << 16, and what multiplies the stage's address (>> 4) before that is added: 1, or 1 - 65536 for the
    // tile whose second chunk is the region of ones (its distance is then counted from the ring's start).
    uint32_t tile_desc[4], tile_mult[4];
};


__host__ __device__ constexpr uint32_t wg_swizzle_bits(uint32_t row_bytes) { return row_bytes == 128 ? 2u : row_bytes == 64 ? 4u : 6u; }

// The 2 * KK * NT MMAs of a stage of kWgRows reduction rows: the limb outermost (switching between the s8 x s8 and s8 x u8
// instruction descriptors stalls the MMA pipe), then the k step, then the A tile, so that consecutive MMAs write
// different accumulators.  FIRST: the stage starts the reduction (its first k step overwrites the accumulators).
// FUSED: both limbs are signed and one MMA takes them side by side (N = 2 * RBB; b_lo then carries the distance
// between the two tiles as its leading byte offset and idesc_hi that N): KK * NT MMAs.
template <int RBA, int RBB, int NT, bool FIRST, bool FUSED>
__device__ __forceinline__ void wg_issue_stage(uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc_hi)
{
    constexpr uint32_t a_hi = ((8u * RBA) >> 4) | (1u << 14) | (wg_swizzle_bits(RBA) << 29);
    constexpr uint32_t b_hi = ((8u * RBB) >> 4) | (1u << 14) | (wg_swizzle_bits(RBB) << 29);
    constexpr uint32_t a_kstep = 2u * RBA, b_kstep = 2u * RBB;     // 32 reduction rows, in 16-byte units
    constexpr int KK = kWgRows / 32;                               // k steps per stage
    constexpr uint32_t a_tile16 = (uint32_t)kWgRows * 128u / 16u;  // an A tile: kWgRows rows x 128 bytes
    constexpr uint32_t b_tile16 = (uint32_t)kWgRows * RBB / 16u;   // a limb's tile: kWgRows rows x RBB bytes
    if (FUSED) {
#pragma unroll
        for (int i = 0; i < KK * NT; ++i) {
            const int kk = i / NT, j = i % NT;
            const uint32_t ao = (uint32_t)j * a_tile16 + (uint32_t)kk * a_kstep;
            if (elect_one())
                mma_i8(tmem + (uint32_t)(j * 2 * RBB), ((uint64_t)a_hi << 32) | (uint64_t)(a_lo + ao),
                       ((uint64_t)b_hi << 32) | (uint64_t)(b_lo + (uint32_t)kk * b_kstep), idesc_hi, (FIRST && kk == 0) ? 0u : 1u);
        }
        return;
    }
    const uint32_t idesc_lo = idesc_hi ^ (1u << 10);               // the low limb is unsigned
#pragma unroll
    for (int i = 0; i < 2 * KK * NT; ++i) {
        const int limb = i / (KK * NT), kk = (i / NT) % KK, j = i % NT;
        const uint32_t ao = (uint32_t)j * a_tile16 + (uint32_t)kk * a_kstep;
        const uint32_t bo = (uint32_t)limb * b_tile16 + (uint32_t)kk * b_kstep;
        if (elect_one())
            mma_i8(tmem + (uint32_t)((j * 2 + limb) * RBB), ((uint64_t)a_hi << 32) | (uint64_t)(a_lo + ao),
                   ((uint64_t)b_hi << 32) | (uint64_t)(b_lo + bo), limb ? idesc_lo : idesc_hi, (FIRST && kk == 0) ? 0u : 1u);
    }
}

// The MMA warp's loop over its slice of the reduction.  False when a wait ran out.
template <int RBA, int RBB, int NT, bool FUSED>
__device__ __forceinline__ bool wg_mma_loop(const WgMmaArgs &A)
{
    uint32_t s = 0, ph = 0;
    uint32_t in_group = 0, group = 0;          // stages issued of the current release group, its index (no divisions here:
                                               // what this warp does between two stages leaves the MMA pipe idle)
    uint32_t a_addr = A.ring;
    for (int i = 0; i < A.k_iters; ++i) {
        if (!mbar_wait_uniform(&A.full_bar[s], ph)) return false;
        tc_fence_after();
        const uint32_t a_lo = ((a_addr >> 4) & 0x3FFFu) | A.a_desc_lo;
        const uint32_t b_lo = (((a_addr + A.a_bytes) >> 4) & 0x3FFFu) | A.b_desc_lo;
        if (i == 0) wg_issue_stage<RBA, RBB, NT, true, FUSED>(A.tmem, a_lo, b_lo, A.idesc_hi);
        else        wg_issue_stage<RBA, RBB, NT, false, FUSED>(A.tmem, a_lo, b_lo, A.idesc_hi);
        // release the group of stages this one completes (the commit covers every MMA issued so far)
        if (++in_group == A.cg) {
            if (elect_one()) mma_commit(&A.empty_bar[group]);
            in_group = 0; ++group;
        }
        a_addr += A.stage_bytes;
        if (++s == A.stages) { s = 0; ph ^= 1u; group = 0; a_addr = A.ring; }
    }
    if (elect_one()) mma_commit(A.acc_bar);
    return true;
}

template <int RBA, int RBB, bool FUSED>
__device__ __forceinline__ bool wg_mma_dispatch_nt(int nt, const WgMmaArgs &A)
{
    // (128 output columns per tile leave room for two A tiles in tensor memory)
    if (nt == 1) return wg_mma_loop<RBA, RBB, 1, FUSED>(A);
    if (nt == 2) return wg_mma_loop<RBA, RBB, 2, FUSED>(A);
    if (RBB == 128) return false;
    if (nt == 3) return wg_mma_loop<RBA, RBB, (RBB == 128 ? 1 : 3), FUSED>(A);
    return wg_mma_loop<RBA, RBB, (RBB == 128 ? 1 : 4), FUSED>(A);
}

// ---- the same from halo tiles ---------------------------------------------------
// The x tile of a stage is the pixel box (8 positions wide, BH rows, 16 / BH images) with a border of one position:
// rows of kWgHaloW positions.  The operand of tap (r, s) is the tile read from r * kWgHaloW + s positions in: the
// shared-memory swizzle is a function of the address, so a window that starts any whole number of positions into the
// tile reads what TMA wrote there.  A k step of 32 positions is four box rows: groups of eight positions a tile row
// apart (the stride byte offset), starting at the box row's place in the tile.
constexpr int kWgHaloW = 10;
template <int RBA, int BH>
__host__ __device__ constexpr uint32_t wg_halo_kstep16(int kk)
{
    return (uint32_t)((((kk * 4) / BH) * (BH + 2) * kWgHaloW + ((kk * 4) % BH) * kWgHaloW) * RBA / 16);
}

template <int RBA, int RBB, int NT, bool FIRST, int BH>
__device__ __forceinline__ void wg_issue_stage_halo(uint32_t tmem, const uint32_t (&a_lo)[NT], uint32_t b_lo, uint32_t idesc)
{
    constexpr uint32_t a_hi = (((uint32_t)kWgHaloW * RBA) >> 4) | (1u << 14) | (wg_swizzle_bits(RBA) << 29);
    constexpr uint32_t b_hi = ((8u * RBB) >> 4) | (1u << 14) | (wg_swizzle_bits(RBB) << 29);
    constexpr uint32_t b_kstep = 2u * RBB;
    constexpr int KK = kWgRows / 32;
#pragma unroll
    for (int i = 0; i < KK * NT; ++i) {
        const int kk = i / NT, j = i % NT;
        if (elect_one())
            mma_i8(tmem + (uint32_t)(j * 2 * RBB), ((uint64_t)a_hi << 32) | (uint64_t)(a_lo[j] + wg_halo_kstep16<RBA, BH>(kk)),
                   ((uint64_t)b_hi << 32) | (uint64_t)(b_lo + (uint32_t)kk * b_kstep), idesc, (FIRST && kk == 0) ? 0u : 1u);
    }
}

template <int RBA, int RBB, int NT, int BH>
__device__ __forceinline__ bool wg_mma_loop_halo(const WgMmaArgs &A)
{
    uint32_t s = 0, ph = 0, in_group = 0, group = 0;
    uint32_t a_addr = A.ring;
    for (int i = 0; i < A.k_iters; ++i) {
        if (!mbar_wait_uniform(&A.full_bar[s], ph)) return false;
        tc_fence_after();
        const uint32_t base = (a_addr >> 4) & 0x3FFFu;
        uint32_t a_lo[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) a_lo[j] = base * A.tile_mult[j] + A.tile_desc[j];
        const uint32_t b_lo = (((a_addr + A.a_bytes) >> 4) & 0x3FFFu) | A.b_desc_lo;
        if (i == 0) wg_issue_stage_halo<RBA, RBB, NT, true, BH>(A.tmem, a_lo, b_lo, A.idesc_hi);
        else        wg_issue_stage_halo<RBA, RBB, NT, false, BH>(A.tmem, a_lo, b_lo, A.idesc_hi);
        if (++in_group == A.cg) {
            if (elect_one()) mma_commit(&A.empty_bar[group]);
            in_group = 0; ++group;
        }
        a_addr += A.stage_bytes;
        if (++s == A.stages) { s = 0; ph ^= 1u; group = 0; a_addr = A.ring; }
    }
    if (elect_one()) mma_commit(A.acc_bar);
    return true;
}

template <int RBA, int RBB>
__device__ __forceinline__ bool wg_mma_dispatch_halo(int nt, int bh, const WgMmaArgs &A)
{
    if (RBA < 64 || nt < 1 || nt > 4 || (RBB == 128 && nt > 2)) return false;
    constexpr int R = RBA < 64 ? 64 : RBA;             // (instances for the layouts that can occur only)
    if (bh == 8) {
        if (nt == 1) return wg_mma_loop_halo<R, RBB, 1, 8>(A);
        if (nt == 2) return wg_mma_loop_halo<R, RBB, 2, 8>(A);
        if (nt == 3) return wg_mma_loop_halo<R, RBB, (RBB == 128 ? 1 : 3), 8>(A);
        return wg_mma_loop_halo<R, RBB, (RBB == 128 ? 1 : 4), 8>(A);
    }
    if (nt == 1) return wg_mma_loop_halo<R, RBB, 1, 4>(A);
    if (nt == 2) return wg_mma_loop_halo<R, RBB, 2, 4>(A);
    if (nt == 3) return wg_mma_loop_halo<R, RBB, (RBB == 128 ? 1 : 3), 4>(A);
    return wg_mma_loop_halo<R, RBB, (RBB == 128 ? 1 : 4), 4>(A);
}

// One instance per pair of operand layouts: RBA = row bytes of the x chunks, RBB = row bytes of the gradient tiles.
template <int RBA, int RBB>
__global__ void __launch_bounds__(kWgThreads, 1) qbp_wgrad_kernel(const __grid_constant__ WgradParams P)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kWgMaxStages], empty_bar[kWgMaxStages], acc_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int4 s_load[kWgMaxLoads];      // (destination offset in the stage, 0 x / 1 hi / 2 lo, channel offset, tap dw | dh << 16)
    __shared__ int s_counts[1];               // loads per stage
    __shared__ long long s_cterm[128];        // direct epilogue: the tile's column terms

    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);
    const uint32_t a_tile_bytes = P.a_chunk_bytes * (uint32_t)P.a_chunks;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const WgItem wi = wg_item(P, blockIdx.x);
    const int ag = wi.ag;
    const int n0 = wi.tb * P.bn;
    const int it_begin = (int)((int64_t)P.iters_total * wi.slice / wi.slices);
    const int it_end = (int)((int64_t)P.iters_total * (wi.slice + 1) / wi.slices);
    const int k_iters = it_end - it_begin;
    const int n_tiles = min(P.ma, P.a_tiles - ag * P.ma);        // A tiles this CTA owns
    const uint32_t a_bytes = P.halo_bh ? P.halo_bytes : a_tile_bytes * (uint32_t)n_tiles;
    const uint32_t stage_bytes = a_bytes + 2u * P.b.tile_bytes;
    const bool last_group = ag == P.a_groups - 1;
    const int stages = last_group ? P.stages_last : P.stages, cg = last_group ? P.cg_last : P.cg;

    // chunks present in A tile `at`: conv -- taps left in the tap group; plain -- column chunks left in K
    auto chunks_of = [&](int at) {
        if (P.conv) return min(P.a_chunks, P.taps - (at / P.tiles_c) * P.a_chunks);
        return min(P.a_chunks, (int)((P.K - (int64_t)at * 128 + P.rb_a - 1) / P.rb_a));
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&acc_bar, 1);
        mbar_fence_init();
        tma_prefetch_desc(&P.mapX); tma_prefetch_desc(&P.mapHi); tma_prefetch_desc(&P.mapLo);
        // the loads of one stage
        int nl = 0;
        s_load[nl++] = make_int4((int)a_bytes, 1, n0, 0);
        s_load[nl++] = make_int4((int)(a_bytes + P.b.tile_bytes), 2, n0, 0);
        if (P.halo_bh) s_load[nl++] = make_int4(0, 0, 0, ((-P.pad) & 0xFFFF) | ((-P.pad) << 16));     // the box with its border
        for (int j = 0; j < (P.halo_bh ? 0 : n_tiles); ++j) {
            const int at = ag * P.ma + j, nc = chunks_of(at);
            for (int c = 0; c < nc; ++c) {
                const int dst = (int)((uint32_t)j * a_tile_bytes + (uint32_t)c * P.a_chunk_bytes);
                if (!P.conv) s_load[nl++] = make_int4(dst, 0, at * 128 + c * P.rb_a, 0);
                else {
                    const int tap = (at / P.tiles_c) * P.a_chunks + c;
                    const int dh = tap / P.S - P.pad, dw = tap % P.S - P.pad;
                    s_load[nl++] = make_int4(dst, 0, (at % P.tiles_c) * P.rb_a, (dw & 0xFFFF) | (dh << 16));
                }
            }
        }
        s_counts[0] = nl;
    }
    if (warp == 1) { tmem_alloc(&tmem_slot, (uint32_t)P.tmem_cols); tmem_relinquish(); }
    if (P.ones_tot && last_group && P.halo_bh) {
        // halo tiles: the spare chunk of the last A tile is read from a region of its own, filled with the code 1
        uint4 *dst = reinterpret_cast<uint4 *>(smem + P.ones_off);
        for (uint32_t i = threadIdx.x; i < P.halo_bytes / 16; i += kWgThreads) dst[i] = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
        fence_proxy_async();
    } else if (P.ones_tot && last_group) {
        // the spare chunk of the last A tile, in every stage: the code 1 in every byte (whatever the swizzle)
        const int j_last = n_tiles - 1, c_spare = chunks_of(P.a_tiles - 1);
        for (int st_i = 0; st_i < stages; ++st_i) {
            uint4 *dst = reinterpret_cast<uint4 *>(smem + (size_t)st_i * stage_bytes + (size_t)j_last * a_tile_bytes + (size_t)c_spare * P.a_chunk_bytes);
            for (uint32_t i = threadIdx.x; i < P.a_chunk_bytes / 16; i += kWgThreads) dst[i] = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
        }
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // (each role waits for the kernels before at its first use of their results: what it needs of the launch's parameters, and the
    // code up to there, has then been fetched)
    const uint32_t tmem_base = tmem_slot;
    bool timed_out = false;

    if (warp == 0) {
        // ---------------------------------------------------- TMA producer (lane 0 owns the barriers)
        const int n_loads = s_counts[0];
        uint32_t tx_bytes = 2u * P.b.tile_bytes + (P.halo_bh ? P.halo_box_bytes : 0u);
        for (int j = 0; j < (P.halo_bh ? 0 : n_tiles); ++j) tx_bytes += (uint32_t)chunks_of(ag * P.ma + j) * P.a_chunk_bytes;
        const int4 ld = lane < n_loads ? s_load[lane] : make_int4(0, 0, 0, 0);
        const int dw = (int)(short)(ld.w & 0xFFFF), dh = ld.w >> 16;
        const void *map = ld.y == 0 ? (const void *)&P.mapX : ld.y == 1 ? (const void *)&P.mapHi : (const void *)&P.mapLo;
        uint32_t s = 0, gph = 1;                      // stage, parity of the stage group's "empty" barrier
        uint32_t in_group = 0, group = 0;             // position in the release group, the group's index
        for (int i = 0; i < k_iters; ++i) {
            int ok = 1;
            if (lane == 0) {
                if (in_group == 0) ok = mbar_wait(&empty_bar[group], gph) ? 1 : 0;
                if (ok) mbar_expect_tx(&full_bar[s], tx_bytes);
            }
            if (++in_group == (uint32_t)cg) { in_group = 0; ++group; }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) { timed_out = true; break; }
            if (i == 0) pdl_wait();
            if (lane < n_loads) {
                uint8_t *dst = smem + (size_t)s * stage_bytes + ld.x;
                const int it = it_begin + i;
                if (!P.conv) tma_load_2d(dst, map, &full_bar[s], ld.z, it * P.kr);
                else {
                    int t1, tw, tn, th;
                    P.d_tiles_w.divmod(it, t1, tw);
                    P.d_tiles_h.divmod(t1, tn, th);
                    const int w0 = tw << P.bw_log2, h0 = th << P.bh_log2;
                    const int img0 = tn * (P.kr >> (P.bw_log2 + P.bh_log2));
                    tma_load_4d(dst, map, &full_bar[s], ld.z, w0 + dw, h0 + dh, img0);
                }
            }
            __syncwarp();
            if (++s == (uint32_t)stages) { s = 0; gph ^= 1u; group = 0; }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------ MMA issuer (the whole warp in step, an elected lane issues)
        WgMmaArgs A;
        A.full_bar = full_bar; A.empty_bar = empty_bar; A.acc_bar = &acc_bar;
        A.ring = smem_u32(smem); A.stage_bytes = stage_bytes; A.a_bytes = a_bytes; A.tmem = tmem_base;
        A.k_iters = k_iters; A.stages = (uint32_t)stages; A.cg = (uint32_t)cg;
        A.a_desc_lo = P.a.desc_lo;
        // (a barrier's wait is bounded: its clock starts once the producer's copies can)
        pdl_wait();
        if (P.halo_bh) {
            // where each A tile's taps start in the halo tile (tap (r, s): r tile rows and s positions in)
            for (int j = 0; j < 4; ++j) {
                const int at = min(ag * P.ma + j, P.a_tiles - 1);
                const int tap0 = at * P.a_chunks, tap1 = tap0 + 1;
                const uint32_t off0 = (uint32_t)((tap0 / P.S) * kWgHaloW + tap0 % P.S) * (uint32_t)P.rb_a >> 4;
                uint32_t lbo = 0, mult = 1u;
                if (P.a_chunks == 2 && tap1 < P.taps)
                    lbo = ((uint32_t)((tap1 / P.S) * kWgHaloW + tap1 % P.S) * (uint32_t)P.rb_a >> 4) - off0;
                else if (P.a_chunks == 2 && P.ones_tot) {
                    // the region of ones, from wherever the stage is: (ones - (stage + off0)) << 16 = (ones - off0) << 16 - (stage << 16)
                    lbo = ((A.ring + P.ones_off) >> 4) - off0;
                    mult = 1u - 65536u;
                }
                A.tile_desc[j] = off0 + (lbo << 16);
                A.tile_mult[j] = mult;
            }
            A.b_desc_lo = P.b2_desc_lo; A.idesc_hi = P.idesc_fused;
            timed_out = !wg_mma_dispatch_halo<RBA, RBB>(n_tiles, P.halo_bh, A);
        } else if (P.lo_signed) {
            A.b_desc_lo = P.b2_desc_lo; A.idesc_hi = P.idesc_fused;
            timed_out = !wg_mma_dispatch_nt<RBA, RBB, true>(n_tiles, A);
        } else {
            A.b_desc_lo = P.b.desc_lo; A.idesc_hi = P.idesc_hi;
            timed_out = !wg_mma_dispatch_nt<RBA, RBB, false>(n_tiles, A);
        }
    } else {
        // ------------------------------------------------------- epilogue
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        pdl_wait();
        // what the epilogue needs of other kernels' results is fetched beside the products: the scale, the zero-points (signed
        // low bytes: the limbs hold g16 - 128, against the zero-point zg - 128) and, one tile of rows ahead, the row terms
        const float scale = P.direct ? __fmul_rn(P.qx->scale, P.qg->scale) : 0.0f;
        const long long zg_d = P.direct ? P.qg->zero_point - (P.lo_signed ? 128 : 0) : 0, zz_d = P.direct ? P.M * P.qx->zero_point * zg_d : 0;
        auto row_of = [&](int at, int64_t &k) {                     // whether this thread's row of A tile `at` is one of the result's
            const bool valid = row / P.rb_a < chunks_of(at);
            k = (int64_t)at * 128 + row;                            // plain: output row
            if (!P.conv) return valid && k < P.K;
            return valid && (at % P.tiles_c) * P.rb_a + row % P.rb_a < P.C;
        };
        auto row_term = [&](int at) {
            int64_t k;
            return P.direct && row_of(at, k) ? -zg_d * P.sx.at(k) + zz_d : 0ll;
        };
        long long rterm = n_tiles > 0 ? row_term(ag * P.ma) : 0;
        if (P.direct) {
            const int t = threadIdx.x - 64;
            const long long zx = P.qx->zero_point;
            if (t < P.bn) s_cterm[t] = (int64_t)n0 + t < P.N ? -zx * wg_plain_sum_g(P, n0 + t) : 0;
            named_barrier(3, 128);
        }
        if (k_iters > 0 && !mbar_wait_warp(&acc_bar, 0)) timed_out = true;
        tc_fence_after();
        if (!timed_out && k_iters > 0) {
            long long *part = P.part + (int64_t)blockIdx.x * P.part_stride;
            for (int j = 0; j < n_tiles; ++j) {
                const int at = ag * P.ma + j;
                int64_t k;
                const bool valid = row_of(at, k);
                const long long rterm_next = j + 1 < n_tiles ? row_term(at + 1) : 0;
                const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(j * 2 * P.bn);
                for (int c0 = 0; c0 < P.bn; c0 += 32) {
                    if ((int64_t)n0 + c0 >= P.N) break;                     // (a ragged last tile: nothing reads those)
                    uint32_t rh[32], rl[32];
                    tmem_ld_32x32(t_addr + (uint32_t)c0, rh);
                    tmem_ld_32x32(t_addr + (uint32_t)(P.bn + c0), rl);
                    tmem_ld_wait();
                    if (P.ones_tot && at == P.a_tiles - 1 && row == P.rb_a * chunks_of(at)) {
                        // the row of ones: this slice's sum of the 16-bit gradient codes, per output channel
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (n0 + c0 + e < P.N)
                                atomicAdd(P.ones_tot + n0 + c0 + e, (unsigned long long)(256ll * (long long)(int)rh[e] + (long long)(int)rl[e]));
                    }
                    if (!valid) continue;
                    if (P.direct) {
                        // the whole reduction is here: zero-points, scale, store (N is a multiple of 16: groups of four
                        // columns are whole; the column terms come from shared memory -- read per element from global
                        // memory, between stores they might alias, they cost a load latency each)
                        const int64_t at_out = k * P.N + n0 + c0;
#pragma unroll
                        for (int e = 0; e < 32; e += 4) {
                            if ((int64_t)n0 + c0 + e >= P.N) break;
                            long long a4[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) a4[q] = 256ll * (long long)(int)rh[e + q] + (long long)(int)rl[e + q] + rterm + s_cterm[c0 + e + q];
                            if (P.acc_out) {
                                long long *dst = P.acc_out + at_out + e;
#pragma unroll
                                for (int q = 0; q < 4; ++q) dst[q] = a4[q];
                            }
                            if (P.dW) {
                                const float4 v = make_float4(__fmul_rn((float)a4[0], scale), __fmul_rn((float)a4[1], scale),
                                                             __fmul_rn((float)a4[2], scale), __fmul_rn((float)a4[3], scale));
                                float *dst = P.dW + at_out + e;
                                if (P.dW_vec) *reinterpret_cast<float4 *>(dst) = v;
                                else { dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w; }
                            }
                        }
                    } else if (P.conv) {
                        // partial block [tile][column][row]: a warp's 32 rows are contiguous, and so are the
                        // channels the second kernel reads together
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            part[((int64_t)j * P.bn + c0 + e) * 128 + row] = 256ll * (long long)(int)rh[e] + (long long)(int)rl[e];
                    } else {
                        // partial block [tile][row][column]
                        long long *dst = part + ((int64_t)j * 128 + row) * P.bn + c0;
#pragma unroll
                        for (int e = 0; e < 32; e += 2) {
                            longlong2 v;
                            v.x = 256ll * (long long)(int)rh[e] + (long long)(int)rl[e];
                            v.y = 256ll * (long long)(int)rh[e + 1] + (long long)(int)rl[e + 1];
                            *reinterpret_cast<longlong2 *>(dst + e) = v;
                        }
                    }
                }
                rterm = rterm_next;
            }
        }
    }

    if (timed_out) {
        raise_timeout(P.status);
        __nanosleep(1000000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) { __syncwarp(); tmem_dealloc(tmem_base, (uint32_t)P.tmem_cols); }
}

// Adds the CTAs' partials, applies the zero-points and dequantises:
//   acc = raw - zg * SX - zx * SG + count * zx * zg
// Plain product [k][n]: SX / SG are the column sums, count = M.  kWgFinalizeLanes lanes per output element share its slices (an
// element's partials are few hundred bytes each, far apart: one thread walking them alone is bound by latency).
__global__ void __launch_bounds__(256) wgrad_finalize_kernel(const __grid_constant__ WgradParams P, int64_t total)
{
    pdl_wait();
    constexpr int kLanes = kWgFinalizeLanes;
    const int64_t e_raw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kLanes;
    const int part_lane = threadIdx.x % kLanes;
    const bool live = e_raw < total;
    const int64_t e = live ? e_raw : total - 1;           // (idle lanes of the last warp compute a duplicate and do not store)
    // (signed low bytes: the limbs hold g16 - 128, against the zero-point zg - 128)
    const long long zx = P.qx->zero_point, zg = P.qg->zero_point - (P.lo_signed ? 128 : 0);
    const int64_t k = e / P.N;
    const int n = (int)(e % P.N);
    const int at = (int)(k / 128), row = (int)(k % 128);  // accumulator tile, row in it
    // the CTAs of this element's item
    const int ag = at / P.ma, j = at % P.ma, tb = n / P.bn, col = n % P.bn;
    const int item = ag * P.tiles_b + tb;
    const int full_items = P.ctas_full / P.s_full;
    const int first = item < full_items ? item * P.s_full : P.ctas_full + (item - full_items) * P.s_last;
    const int slices = item < full_items ? P.s_full : P.s_last;
    long long raw = 0;
    const long long *src = P.part + (int64_t)first * P.part_stride + ((int64_t)j * 128 + row) * P.bn + col;
    int sl = part_lane;
    for (; sl + 7 * kLanes < slices; sl += 8 * kLanes) {
        long long v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcs(src + (int64_t)(sl + u * kLanes) * P.part_stride);
#pragma unroll
        for (int u = 0; u < 8; ++u) raw += v[u];
    }
    for (; sl < slices; sl += kLanes) raw += __ldcs(src + (int64_t)sl * P.part_stride);
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1) raw += __shfl_xor_sync(0xffffffffu, raw, o);
    if (!live || part_lane != 0) return;
    const long long SX = P.cx ? P.cx[k] : P.sx.at(k), SG = wg_plain_sum_g(P, n);
    const long long acc = raw - zg * SX - zx * SG + P.M * zx * zg;
    if (P.acc_out) P.acc_out[e] = acc;
    if (P.dW) P.dW[e] = __fmul_rn((float)acc, __fmul_rn(P.qx->scale, P.qg->scale));
}

// SX (of_x: over the positions of x that tap (r, s) sees) or SG (over the positions of g at which it is inside the image) in
// four parts: all positions, less the row and the column that are out, plus the corner that was taken off twice.
//   g sees the tap where p - pad + r is in [0, H): not in the first row for r < pad, not in the last for r > pad;
//   x is seen where h + pad - r is in [0, H):      not in the last row for r < pad, not in the first for r > pad.
__device__ __forceinline__ long long wg_tap_part(const WgradParams &P, bool of_x, int ch, int r, int s, int part)
{
    const int dr = r < P.pad ? -1 : r > P.pad ? 1 : 0, ds = s < P.pad ? -1 : s > P.pad ? 1 : 0;
    if (part == 0 && P.tot_x) {
        if (of_x) return P.tot_x[ch];
        return P.tot_g[ch] - (P.lo_signed && P.tot_g_plain ? 128ll * P.Nimg * P.H * P.W : 0);
    }
    if (part == 0) return of_x ? P.cx[ch] : 256 * P.chi[ch] + P.clo[ch];
    if ((part != 2 && dr == 0) || (part != 1 && ds == 0)) return 0;
    const int row = (dr > 0) != of_x ? 1 : 0, col = (ds > 0) != of_x ? 1 : 0;         // the row / column out: 0 first, 1 last
    const int edge = part == 1 ? row : part == 2 ? 2 + col : 4 + 2 * row + col;
    const int64_t at = (int64_t)edge * (of_x ? P.C : P.N) + ch;
    const long long v = of_x ? P.ex[at] : 256 * P.ehi[at] + P.elo[at];
    return part == 3 ? v : -v;
}

// The same for a convolution, output [n][tap][c].  A block takes 64 channels of one tap and NB output channels per group of 64 threads:
// SX and SG are added up once per block (once per element they are tens of loads each: 78 us for a 256 -> 256 channel 3x3 filter).
// Q = 4: the groups share the slices of the same NB output channels and meet in shared memory; Q = 1, for items of one or two slices:
// each takes all slices of NB channels of its own (three of four groups had nothing to load).
// Bound by latency: rounds of resident blocks, each a few dependent loads long.  So four blocks share an SM (one pointer for the NB
// columns of a tile, 128 values apart: at 124 registers, two blocks), eight or more loads are in flight per thread, and NB is as
// large as leaves four blocks per SM.  256 -> 256 channels, 8 slices: 16.5 -> 10.0 us; 512 -> 512 with
// 64 x 7 x 7 positions, 1 slice: 46.9 -> 11.0.
template <int NB, int Q>
__global__ void __launch_bounds__(256, 4) wgrad_conv_finalize_kernel(const __grid_constant__ WgradParams P)
{
    pdl_wait();
    constexpr int U = NB == 8 ? 2 : 8 / NB;                // slices in flight per output channel
    constexpr int NN = Q == 1 ? 4 * NB : NB;               // output channels of the block
    __shared__ long long s_part[Q == 1 ? 1 : NB][4][64], s_sx[4][64], s_sg[4][NN];
    const int cblocks = (P.C + 63) / 64;
    const int tap = (int)blockIdx.x / cblocks, cl = threadIdx.x & 63, c = ((int)blockIdx.x % cblocks) * 64 + cl;
    const int q = threadIdx.x >> 6;
    const int n0 = (int)blockIdx.y * NN, n_mine = n0 + (Q == 1 ? q * NB : 0);
    const int r = tap / P.S, s = tap % P.S, pad = P.pad;
    const bool c_ok = c < P.C && n_mine < P.N;
    // the CTAs of this channel's items
    const int at = (tap / P.a_chunks) * P.tiles_c + (c_ok ? c : 0) / P.rb_a, row = (tap % P.a_chunks) * P.rb_a + (c_ok ? c : 0) % P.rb_a;
    const int ag = at / P.ma, j = at % P.ma, full_items = P.ctas_full / P.s_full;
    long long raw[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) raw[i] = 0;
    if (c_ok) {
        // (N and a tile's columns are multiples of NB: these output channels lie in one tile)
        const int item = ag * P.tiles_b + n_mine / P.bn;
        const int first = item < full_items ? item * P.s_full : P.ctas_full + (item - full_items) * P.s_last;
        const int slices = item < full_items ? P.s_full : P.s_last;
        const long long *const src = P.part + (int64_t)first * P.part_stride + ((int64_t)j * P.bn + n_mine % P.bn) * 128 + row;
        for (int sl = Q == 1 ? 0 : q; sl < slices; sl += Q * U) {
            long long v[NB][U];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < NB; ++i) v[i][u] = sl + Q * u < slices ? __ldcs(src + (int64_t)(sl + Q * u) * P.part_stride + i * 128) : 0;
#pragma unroll
            for (int i = 0; i < NB; ++i)
#pragma unroll
                for (int u = 0; u < U; ++u) raw[i] += v[i][u];
        }
    }
    if (Q != 1) {
#pragma unroll
        for (int i = 0; i < NB; ++i) s_part[Q == 1 ? 0 : i][q][cl] = raw[i];
    }
    s_sx[q][cl] = c < P.C ? wg_tap_part(P, true, c, r, s, q) : 0;
    if (cl < NN) s_sg[q][cl] = wg_tap_part(P, false, min(n0 + cl, (int)P.N - 1), r, s, q);
    __syncthreads();
    // (signed low bytes: the limbs hold g16 - 128, against the zero-point zg - 128)
    const long long zx = P.qx->zero_point, zg = P.qg->zero_point - (P.lo_signed ? 128 : 0);
    const long long rows_ok = P.H - (r < pad ? pad - r : r - pad), cols_ok = P.W - (s < pad ? pad - s : s - pad);
    const long long count = (long long)P.Nimg * (rows_ok > 0 ? rows_ok : 0) * (cols_ok > 0 ? cols_ok : 0);
    const float scale = __fmul_rn(P.qx->scale, P.qg->scale);
    const long long xterm = count * zx * zg - zg * (s_sx[0][cl] + s_sx[1][cl] + s_sx[2][cl] + s_sx[3][cl]);
    auto finish = [&](int nl, long long part) {
        const int n = n0 + nl;
        if (n >= P.N || c >= P.C) return;
        const long long acc = part + xterm - zx * (s_sg[0][nl] + s_sg[1][nl] + s_sg[2][nl] + s_sg[3][nl]);
        const int64_t e = ((int64_t)n * P.taps + tap) * P.C + c;
        if (P.acc_out) P.acc_out[e] = acc;
        if (P.dW) P.dW[e] = __fmul_rn((float)acc, scale);
    };
    if (Q == 1) {
#pragma unroll
        for (int i = 0; i < NB; ++i) finish(q * NB + i, raw[i]);
    } else {
        for (int nl = q; nl < NB; nl += 4) finish(nl, s_part[nl][0][cl] + s_part[nl][1][cl] + s_part[nl][2][cl] + s_part[nl][3][cl]);
    }
}

// Pixel box of `rows` = bw x bh x bn positions (powers of two) that needs the fewest steps.
static void pick_pixel_box_w(int rows, int Nimg, int H, int W, int &bwl, int &bhl)
{
    long long best = -1;
    int lg = 0; while ((1 << lg) < rows) ++lg;
    for (int a = 0; a <= lg; ++a)
        for (int b = 0; a + b <= lg; ++b) {
            const int bw = 1 << a, bh = 1 << b, bn = rows >> (a + b);
            const long long tiles = (long long)((W + bw - 1) / bw) * ((H + bh - 1) / bh) * ((Nimg + bn - 1) / bn);
            const long long score = tiles * 64 - a * 8 - b;
            if (best < 0 || score < best) { best = score; bwl = a; bhl = b; }
        }
}

bool wgrad_conv_supported(const qbp_conv_desc *d)
{
    return d->stride == 1 && d->R == d->S && (d->R == 1 || d->R == 3) && d->pad == (d->R - 1) / 2 && d->N > 0 &&
           d->H > 0 && d->W > 0 && d->C > 0 && d->K > 0 && d->C % 32 == 0 && d->K % 32 == 0;
}

// Everything of the launch that does not depend on pointers: tiling, split, workspace.
struct WgradPlan {
    WgradParams P;
    int grid;
    size_t smem;
    int bw, bh, bn_img;
};

}  // namespace qbp

// Plain products of more than kWgPieceRows rows: the sums by atomics into a table, from as many blocks as the rows fill.  The 16
// pieces that a reader adds up would be longer than the whole product takes (2^20 rows, 128 x 32 columns: 521 us with pieces, 115
// with the table; the clearing it needs is what shorter ones save).  Such a product never finishes in one launch and is never the pair
// kernel's: only wgrad_finalize_kernel reads the sums.
constexpr int64_t kWgPieceRows = 65536;
size_t qbp::wgrad_sum_table(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K)
{
    if (!d) return M > kWgPieceRows ? (size_t)(K + 2 * N) : 0;
    return (size_t)(d->pad ? 9 : 1) * ((size_t)d->C + 2 * (size_t)d->K);
}
int qbp::wgrad_sum_jobs(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K, const int8_t *x, const int8_t *hi, const uint8_t *lo,
                        bool lo_signed, int64_t *tab, SumJob (&jobs)[6])
{
    const struct { const void *q; int64_t cols; int is_signed; } t[3] = {{x, K, 1}, {hi, N, 1}, {lo, N, lo_signed ? 1 : 0}};
    for (int i = 0; i < 3; ++i) { jobs[i] = SumJob{t[i].q, M, t[i].cols, kSumCols, t[i].is_signed, nullptr, 0, 0, tab}; if (tab) tab += t[i].cols; }
    if (!d || !d->pad) return 3;
    for (int i = 0; i < 3; ++i) { jobs[3 + i] = SumJob{t[i].q, M, t[i].cols, kSumEdges, t[i].is_signed, nullptr, d->H, d->W, tab}; if (tab) tab += 8 * t[i].cols; }
    return 6;
}

// Whether the product can take the gradient's per-channel totals itself (a spare chunk in its last A tile).
bool qbp::wgrad_self_totals(const qbp_conv_desc *d)
{
    if (!d || !wgrad_conv_supported(d)) return false;
    const int rb_a = d->C >= 128 ? 128 : d->C >= 64 ? 64 : 32;
    const int a_chunks = 128 / rb_a;
    return d->C % rb_a == 0 && (d->R * d->S) % a_chunks != 0;
}

namespace qbp {

static void plan_wgrad(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K, WgradPlan &pl, bool lo_signed = false)
{
    WgradParams &P = pl.P;
    P = WgradParams{};
    P.conv = d ? 1 : 0;
    P.M = M; P.N = N; P.K = K;
    // g side: one swizzled row holds bn output channels
    uint32_t rb_b = N >= 128 ? 128u : N >= 64 ? 64u : 32u;
    // (a short plain reduction -- done whole, see below -- whose tiles of half as many columns still fit the machine once: the
    // epilogue takes 1900 cycles per 32 columns)
    while (!d && M <= 8 * kWgRows && rb_b > 32 && ((K + 127) / 128) * ((N + rb_b / 2 - 1) / (rb_b / 2)) <= sm_count()) rb_b /= 2;
    P.bn = (int)rb_b;
    P.tiles_b = (int)((N + P.bn - 1) / P.bn);
    // x side: 128 MMA rows = a_chunks chunks of rb_a columns / channels
    const uint32_t rb_a = K >= 128 ? 128u : K >= 64 ? 64u : 32u;
    P.rb_a = (int)rb_a;
    P.a_chunks = 128 / (int)rb_a;
    if (!d) {
        P.a_tiles = (int)((K + 127) / 128);
        P.tiles_c = 1;
    } else {
        P.H = d->H; P.W = d->W; P.Nimg = d->N; P.pad = d->pad; P.R = d->R; P.S = d->S; P.C = d->C;
        P.taps = d->R * d->S;
        P.tiles_c = (d->C + (int)rb_a - 1) / (int)rb_a;
        P.a_tiles = ((P.taps + P.a_chunks - 1) / P.a_chunks) * P.tiles_c;
    }
    // reduction rows per stage: kWgRows (the ring is shallower than with 64, but a stage holds twice the MMAs)
    const uint32_t kr = kWgRows;
    P.kr = (int)kr;
    P.a_chunk_bytes = kr * rb_a;
    P.a = layout_mnmajor(kr, rb_a, (uint32_t)P.a_chunks, P.a_chunk_bytes);
    P.b = layout_mnmajor(kr, rb_b, 1, 0);
    P.idesc_hi = make_idesc(true, true, 1, 1, 128, (uint32_t)P.bn);
    P.idesc_lo = make_idesc(true, false, 1, 1, 128, (uint32_t)P.bn);
    P.lo_signed = lo_signed ? 1 : 0;
    P.b2_desc_lo = layout_mnmajor(kr, rb_b, 2, P.b.tile_bytes).desc_lo;      // the low tile follows the high one in a stage
    P.idesc_fused = make_idesc(true, true, 1, 1, 128, 2u * (uint32_t)P.bn);
    if (!d) {
        P.iters_total = (int)((M + kr - 1) / kr);
        pl.bw = pl.bh = pl.bn_img = 0;
    } else {
        int bwl = 0, bhl = 0;
        pick_pixel_box_w((int)kr, d->N, d->H, d->W, bwl, bhl);
        if (lo_signed && d->R == 3 && P.tiles_c == 1 && P.a_chunks <= 2) {
            // halo tiles: boxes 8 positions wide and 8 or 4 rows high, when that costs at most a fifth more steps
            // than the free choice of box
            const long long free_tiles = (long long)((d->W + (1 << bwl) - 1) >> bwl) * ((d->H + (1 << bhl) - 1) >> bhl) *
                                         ((d->N + ((int)kr >> (bwl + bhl)) - 1) / ((int)kr >> (bwl + bhl)));
            long long best = -1;
            for (int bh = 8; bh >= 4; bh >>= 1) {
                const long long t = (long long)((d->W + 7) / 8) * ((d->H + bh - 1) / bh) * ((d->N + 16 / bh - 1) / (16 / bh));
                if (best < 0 || t < best) { best = t; P.halo_bh = bh; }
            }
            if (best * 5 > free_tiles * 6) P.halo_bh = 0;
            if (P.halo_bh) {
                bwl = 3; bhl = P.halo_bh == 8 ? 3 : 2;
                P.halo_box_bytes = (uint32_t)(kWgHaloW * (P.halo_bh + 2) * (16 / P.halo_bh)) * rb_a;
                P.halo_bytes = (uint32_t)align_up((size_t)P.halo_box_bytes, 1024);
            }
        }
        P.bw_log2 = bwl; P.bh_log2 = bhl;
        pl.bw = 1 << bwl; pl.bh = 1 << bhl; pl.bn_img = (int)kr >> (bwl + bhl);
        P.tiles_w = (d->W + pl.bw - 1) / pl.bw; P.tiles_h = (d->H + pl.bh - 1) / pl.bh;
        P.iters_total = P.tiles_w * P.tiles_h * ((d->N + pl.bn_img - 1) / pl.bn_img);
        P.d_tiles_w = make_fastdiv(P.tiles_w); P.d_tiles_h = make_fastdiv(P.tiles_h);
    }
    // A tiles per CTA: at most what tensor memory holds (two accumulators of bn columns each), spread evenly over
    // the groups that takes (5 tiles: 3 + 2 rather than 4 + 1 -- a stage of few MMAs is bound by its fixed costs)
    const int ma_max = std::max(1, std::min({kWgMaxTiles, 512 / (2 * P.bn), P.a_tiles}));
    P.a_groups = (P.a_tiles + ma_max - 1) / ma_max;
    // (a plain product whose tiles do not fill the machine: one A tile per CTA)
    if (!d && (int64_t)P.a_tiles * P.tiles_b <= sm_count()) P.a_groups = P.a_tiles;
    // A convolution's reduction is split over the machine, and every CTA reads out and writes a partial of all its A tiles: more of
    // them share the gradient's tiles in the loop, fewer leave less to read out, write and add up.  In cycles: an operand row of the
    // loop 2.7 (what the copies reach), a tile's read-out 6000, the partials at 2.6 KB a cycle over the machine.  (20 images of
    // 19 x 19, 96 -> 160: kernel and finalize 22.9 + 14.7 us with two tiles, 18.9 + 12.8 with one, launches included; 64 images of
    // 28 x 28, 128 -> 128: 31 + 16 and 25 + 13; 256 of 14 x 14, 256 -> 256 stays with two: 52 + 21.)
    if (d && !P.halo_bh) {
        int64_t best = -1;
        int groups = P.a_groups;
        for (int ma = ma_max; ma >= 1; --ma) {
            const int64_t ag = (P.a_tiles + ma - 1) / ma, items = ag * P.tiles_b;
            const int64_t slices = std::max<int64_t>(1, std::min<int64_t>(sm_count() / items, P.iters_total));
            const int64_t waves = (items * slices + sm_count() - 1) / sm_count(), iters = (P.iters_total + slices - 1) / slices;
            const int64_t loop = iters * (int64_t)kr * (ma * P.a_chunks + 2) * 27 / 10, part = items * slices * ma * 128 * P.bn * 8;
            const int64_t cost = waves * (loop + ma * 6000) + part / 2600;
            if (best < 0 || cost < best) { best = cost; groups = (int)ag; }
        }
        P.a_groups = groups;
    }
    P.ma = (P.a_tiles + P.a_groups - 1) / P.a_groups;
    int cols = 32; while (cols < P.ma * 2 * P.bn) cols <<= 1;
    P.tmem_cols = cols;
    // pipeline: stages of kr rows; one commit releases `cg` stages (some 24 MMAs between commits while that leaves
    // three groups in the ring).  The CTAs of the last group (fewer A tiles) get a ring of their own shape.
    const int n_last = P.a_tiles - (P.a_groups - 1) * P.ma;                 // A tiles of the last group
    // (the region of ones of the halo variant sits behind the ring)
    const uint32_t ones_bytes = P.halo_bh ? P.halo_bytes : 0u;
    auto ring = [&](int tiles, int &stages, int &cg) {
        const uint32_t stage_bytes = (P.halo_bh ? P.halo_bytes : P.a_chunk_bytes * P.a_chunks * (uint32_t)tiles) + 2 * P.b.tile_bytes;
        stages = std::max(2, std::min<int>(kWgMaxStages, (int)((kWgSmem - 1024 - ones_bytes) / stage_bytes)));
        const int mmas = tiles * (int)(kr / 32) * 2;       // (in MMAs of bn columns: a fused one counts twice)
        cg = 1;
        while (cg * mmas < 24 && stages / (cg + 1) >= 3) ++cg;
        stages -= stages % cg;
        return (size_t)stages * stage_bytes + 1024;
    };
    const size_t smem_full = ring(P.ma, P.stages, P.cg);
    const size_t smem_last = ring(n_last, P.stages_last, P.cg_last);
    P.ones_off = (uint32_t)(std::max(smem_full, smem_last) - 1024);          // behind the longer of the two rings
    pl.smem = std::max(smem_full, smem_last) + ones_bytes;
    // split of the reductions: at most 65536 rows per CTA; with few items, enough slices to fill the machine
    // once, in proportion to an item's cost per reduction step: a fixed part (waits, the share of a commit)
    // worth about eight MMAs, plus its MMAs
    const int max_iters = 65536 / (int)kr;
    const int min_slices = (P.iters_total + max_iters - 1) / max_iters;
    auto cost = [&](int tiles) { return (int64_t)(8 + tiles * (int)(kr / 32) * 2); };
    const int64_t weight = ((int64_t)(P.a_groups - 1) * cost(P.ma) + cost(n_last)) * P.tiles_b;
    const int T = sm_count();
    auto slices_for = [&](int tiles) {
        int64_t s = (int64_t)T * cost(tiles) / weight;
        s = std::max<int64_t>(s, min_slices);
        s = std::max<int64_t>(1, std::min<int64_t>(s, P.iters_total));
        // a short plain reduction (at most 1024 rows) stays whole: no partials and no second kernel
        if (!d && P.iters_total <= 8) s = 1;
        return (int)s;
    };
    P.s_full = slices_for(P.ma);
    P.s_last = slices_for(n_last);
    P.ctas_full = (P.a_groups - 1) * P.tiles_b * P.s_full;
    pl.grid = P.ctas_full + P.tiles_b * P.s_last;
    P.direct = (!d && P.s_full == 1 && P.s_last == 1) ? 1 : 0;
    // (not a power of two apart: the CTAs write their blocks in step, and equal low address bits pile onto few L2 slices)
    P.part_stride = (int64_t)P.ma * 128 * P.bn + 272;
}

static size_t wgrad_ws_bytes(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K)
{
    const size_t table = wgrad_sum_table(d, M, N, K);
    const size_t sums = table ? align_up(sizeof(int64_t) * table, 256)
                              : align_up(sizeof(int32_t) * sum_elems(M, K, kSumCols), 256) + 2 * align_up(sizeof(int32_t) * sum_elems(M, N, kSumCols), 256);
    // (the split, and with it the partials, may differ between the two forms of the low limb: room for either)
    size_t part = 0;
    for (int lo_signed = 0; lo_signed < 2; ++lo_signed) {
        WgradPlan pl;
        plan_wgrad(d, M, N, K, pl, lo_signed != 0);
        part = std::max(part, pl.P.direct ? (size_t)0 : align_up(sizeof(int64_t) * (size_t)pl.grid * (size_t)pl.P.part_stride, 256));
    }
    return 256 + sums + part;
}

}  // namespace qbp

using namespace qbp;

extern "C" __attribute__((visibility("default"))) size_t qbp_wgrad_s16_workspace_bytes(const qbp_conv_desc *d, int64_t M,
                                                                                      int64_t N, int64_t K)
{
    if (d) {
        if (!wgrad_conv_supported(d)) return 0;
        M = (int64_t)d->N * d->H * d->W; N = d->K; K = d->C;
    }
    return wgrad_ws_bytes(d, M > 0 ? M : 1, N > 0 ? N : 1, K > 0 ? K : 1);
}

extern "C" __attribute__((visibility("default"))) int qbp_wgrad_s16(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K,
                                                                   const int8_t *x, const qbp_qparams *qx,
                                                                   const int8_t *g_hi, const uint8_t *g_lo,
                                                                   const qbp_qparams *qg16, int64_t *acc_out, float *dW,
                                                                   void *ws, size_t ws_bytes, void *stream)
{
    return wgrad_s16_impl(d, M, N, K, x, qx, g_hi, g_lo, qg16, acc_out, dW, nullptr, ws, ws_bytes, (cudaStream_t)stream);
}

int qbp::wgrad_s16_impl(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K, const int8_t *x, const qbp_qparams *qx,
                        const int8_t *g_hi, const uint8_t *g_lo, const qbp_qparams *qg16, int64_t *acc_out, float *dW,
                        int *ext_status, void *ws, size_t ws_bytes, cudaStream_t st, const int64_t *tot_x, const int64_t *tot_g16,
                        bool tot_g_filled, bool lo_signed, const SumJob *done_sums)
{
    if (!x || !g_hi || !g_lo || !qx || !qg16) return fail(QBP_ERR_INVALID_ARG, "wgrad_s16: NULL operand");
    if (!acc_out && !dW) return fail(QBP_ERR_INVALID_ARG, "wgrad_s16: acc_out and dW are both NULL");
    if (!aligned16(x) || !aligned16(g_hi) || !aligned16(g_lo))
        return fail(QBP_ERR_INVALID_ARG, "wgrad_s16: operands must be 16-byte aligned");
    if (d) {
        if (!wgrad_conv_supported(d))
            return fail(QBP_ERR_UNSUPPORTED_SHAPE,
                        "wgrad_s16: needs stride 1, R = S in {1,3}, pad = (R-1)/2, C and K multiples of 32");
        M = (int64_t)d->N * d->H * d->W; N = d->K; K = d->C;
        if (M >= (1ll << 30)) return fail(QBP_ERR_UNSUPPORTED_SHAPE, "wgrad: more than 2^30 positions");
    } else {
        if (M <= 0 || N <= 0 || K <= 0) return fail(QBP_ERR_INVALID_ARG, "wgrad_s16: M, N, K must be positive");
        if (N % 16 || K % 16) return fail(QBP_ERR_UNSUPPORTED_SHAPE, "wgrad_s16: N and K must be multiples of 16");
        if (M > (int64_t)INT32_MAX || N > (int64_t)INT32_MAX || K > (int64_t)INT32_MAX)
            return fail(QBP_ERR_UNSUPPORTED_SHAPE, "wgrad_s16: extent too large");
    }
    if (!ws || ws_bytes < wgrad_ws_bytes(d, M, N, K))
        return fail(QBP_ERR_WORKSPACE, "wgrad_s16: workspace of %zu bytes needed, %zu given", wgrad_ws_bytes(d, M, N, K), ws_bytes);

    WgradPlan pl;
    plan_wgrad(d, M, N, K, pl, lo_signed);
    WgradParams &P = pl.P;
    const int64_t outs = d ? (int64_t)d->K * d->R * d->S * d->C : K * N;
    WsCarver w(ws, ws_bytes);
    int *status = w.take<int>(1);
    if (ext_status) status = ext_status;         // the caller's sticky word: raised here, never cleared
    SumJob all[6], jobs[6];
    const size_t table = wgrad_sum_table(d, M, N, K);
    int64_t *tab = table && !done_sums ? w.take<int64_t>(table) : nullptr;
    const int nall = wgrad_sum_jobs(d, M, N, K, x, g_hi, g_lo, lo_signed, tab, all);
    for (int i = 0; i < nall; ++i) {
        if (done_sums) all[i] = done_sums[i];
        else if (!table) all[i].out = w.take<int32_t>(sum_elems(all[i]));
    }
    int64_t *part = P.direct ? nullptr : w.take<int64_t>((size_t)pl.grid * (size_t)P.part_stride);

    // most plain products run on CTA pairs (tiles across two SMs, the whole reduction in one pair), whose stores (TMA for dW, 16 bytes
    // at a time for acc_out) want both outputs on a 16-byte boundary; the single-CTA kernel takes any float- and int64-aligned ones
    const bool pair_kernel = !d && wgrad2_eligible(M, N, K) && aligned16(dW) && aligned16(acc_out);
    // code sums for the zero-point terms: of everything, or (the kernels that wrote the codes left their per-channel totals,
    // or the product takes the gradient's itself: a row of ones in its spare chunk) of the images' edges only
    int rc;
    const bool from_totals = d && tot_x && tot_g16 && (tot_g_filled || wgrad_self_totals(d));
    const int64_t *plain_tot_g = !d && !table && done_sums ? tot_g16 : nullptr;
    int njobs = 0;
    if (!done_sums)
        for (int i = from_totals ? 3 : 0; i < nall; ++i) jobs[njobs++] = all[i];
    if (!table) { P.sx = sums_of(all[0]); P.shi = sums_of(all[1]); P.slo = sums_of(all[2]); }
    else {
        P.cx = (const long long *)all[0].out64; P.chi = (const long long *)all[1].out64; P.clo = (const long long *)all[2].out64;
        if (nall == 6) { P.ex = (const long long *)all[3].out64; P.ehi = (const long long *)all[4].out64; P.elo = (const long long *)all[5].out64; }
        if (tab && (rc = launch_clear(tab, 2 * (int64_t)table, st))) return rc;
    }
    ZeroJobs zero{};
    if (!ext_status && (rc = zero.add(status, 1))) return rc;
    if (from_totals) {
        P.tot_x = (const long long *)tot_x; P.tot_g = (const long long *)tot_g16;
        P.tot_g_plain = tot_g_filled ? 1 : 0;
        if (!tot_g_filled) {
            P.ones_tot = (unsigned long long *)const_cast<int64_t *>(tot_g16);
            if (!done_sums && (rc = zero.add(P.ones_tot, 2 * N))) return rc;
        }
    }
    bool beside = false;
    if ((rc = launch_code_sums(jobs, njobs, st, zero, pair_kernel ? &beside : nullptr))) return rc;      // (the single-CTA kernel waits)
    if (pair_kernel)
        return launch_wgrad2(M, N, K, x, qx, g_hi, g_lo, qg16, acc_out, dW, P.sx, P.shi, P.slo, plain_tot_g, status, beside, st, lo_signed);
    if (!d) P.tot_g = (const long long *)plain_tot_g;

    P.part = (long long *)part; P.status = status;
    P.qx = qx; P.qg = qg16; P.acc_out = (long long *)acc_out; P.dW = dW; P.dW_vec = aligned16(dW) ? 1 : 0;
    const uint32_t kr = (uint32_t)P.kr, rb_a = (uint32_t)P.rb_a, rb_b = (uint32_t)P.bn;
    if (!d) {
        if ((rc = make_map_2d(&P.mapX, x, M, K, kr, rb_a))) return rc;
        if ((rc = make_map_2d(&P.mapHi, g_hi, M, N, kr, rb_b))) return rc;
        if ((rc = make_map_2d(&P.mapLo, g_lo, M, N, kr, rb_b))) return rc;
    } else {
        if ((rc = P.halo_bh ? make_map_nhwc(&P.mapX, x, d->N, d->H, d->W, d->C, pl.bn_img, pl.bh + 2, kWgHaloW, rb_a)
                            : make_map_nhwc(&P.mapX, x, d->N, d->H, d->W, d->C, pl.bn_img, pl.bh, pl.bw, rb_a))) return rc;
        if ((rc = make_map_nhwc(&P.mapHi, g_hi, d->N, d->H, d->W, d->K, pl.bn_img, pl.bh, pl.bw, rb_b))) return rc;
        if ((rc = make_map_nhwc(&P.mapLo, g_lo, d->N, d->H, d->W, d->K, pl.bn_img, pl.bh, pl.bw, rb_b))) return rc;
    }
    // the kernel instance for this pair of operand layouts
    void (*kernel)(const WgradParams) = nullptr;
    const int layout_id = (rb_a == 128 ? 0 : rb_a == 64 ? 1 : 2) * 3 + (rb_b == 128 ? 0 : rb_b == 64 ? 1 : 2);
    switch (layout_id) {
    case 0: kernel = qbp_wgrad_kernel<128, 128>; break;
    case 1: kernel = qbp_wgrad_kernel<128, 64>; break;
    case 2: kernel = qbp_wgrad_kernel<128, 32>; break;
    case 3: kernel = qbp_wgrad_kernel<64, 128>; break;
    case 4: kernel = qbp_wgrad_kernel<64, 64>; break;
    case 5: kernel = qbp_wgrad_kernel<64, 32>; break;
    case 6: kernel = qbp_wgrad_kernel<32, 128>; break;
    case 7: kernel = qbp_wgrad_kernel<32, 64>; break;
    default: kernel = qbp_wgrad_kernel<32, 32>; break;
    }
    static PerDeviceOnce configured[9];
    QBP_SMEM_OPT_IN(configured[layout_id], kernel, kWgSmem);
    QBP_TRACE_BEGIN(st);
    launch(kernel, pl.grid, kWgThreads, pl.smem, st, P);
    QBP_LAUNCH_OK("qbp_wgrad_kernel");
    if (d) {
        const int64_t per_n = (int64_t)P.taps * ((d->C + 63) / 64);
        const bool whole = std::max(P.s_full, P.s_last) <= 2;
        const int groups = whole ? 4 : 1;
        const int nb = per_n * (d->K / (8 * groups)) >= 4ll * sm_count() ? 8 : per_n * (d->K / (4 * groups)) >= 4ll * sm_count() ? 4 : 2;
        const dim3 grid((unsigned)per_n, (unsigned)((d->K + nb * groups - 1) / (nb * groups)));
        QBP_TRACE_BEGIN(st);
        if (whole) {
            if (nb == 8)      launch(wgrad_conv_finalize_kernel<8, 1>, grid, 256, 0, st, P);
            else if (nb == 4) launch(wgrad_conv_finalize_kernel<4, 1>, grid, 256, 0, st, P);
            else              launch(wgrad_conv_finalize_kernel<2, 1>, grid, 256, 0, st, P);
        } else {
            if (nb == 8)      launch(wgrad_conv_finalize_kernel<8, 4>, grid, 256, 0, st, P);
            else if (nb == 4) launch(wgrad_conv_finalize_kernel<4, 4>, grid, 256, 0, st, P);
            else              launch(wgrad_conv_finalize_kernel<2, 4>, grid, 256, 0, st, P);
        }
        QBP_LAUNCH_OK("wgrad_conv_finalize_kernel");
    } else if (!P.direct) {
        const int blocks = (int)((outs * kWgFinalizeLanes + 255) / 256);
        QBP_TRACE_BEGIN(st);
        launch(wgrad_finalize_kernel, blocks, 256, 0, st, P, outs);
        QBP_LAUNCH_OK("wgrad_finalize_kernel");
    }
    return QBP_OK;
}
