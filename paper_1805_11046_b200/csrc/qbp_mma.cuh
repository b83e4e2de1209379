// Declarations shared by the tensor-core product files: TMA tensor-map
// construction on the host, the parameter block of the tcgen05 kernels, and
// the small helper launchers (row/column sums of codes).
#pragma once

#include <cuda.h>

#include "qbp_common.cuh"

namespace qbp {

// ---- sums of stored codes (qbp_quant.cu) -------------------------------------
int launch_rowsum(const void *q, bool is_signed, int64_t rows, int64_t cols, int32_t *sums, cudaStream_t st);
// (cleared: sums is zero already)
int launch_colsum(const void *q, bool is_signed, int64_t rows, int64_t cols, int64_t *sums, cudaStream_t st, bool cleared = false);
// Clears 32-bit words in a kernel: a memset node between two kernels costs the stream 4 to 5 us, since neither overlaps it.
int launch_clear(void *p, int64_t words, cudaStream_t st);
// Sums of stored codes as a product takes them for its zero-point correction: element i is the sum of `pieces` int32
// values p[i], p[i + stride], ... (sums along the rows of a tensor in pieces of its columns, so that nothing has to start at
// zero and no atomics are needed).
struct CodeSums {
    const int32_t *p; int pieces; int64_t stride;
#ifdef __CUDACC__
    __device__ __forceinline__ long long at(int64_t i) const
    {
        long long s = 0;
#pragma unroll 8
        for (int k = 0; k < pieces; ++k) s += load_after_wait(p + (int64_t)k * stride + i);
        return s;
    }
#endif
};
inline CodeSums sums_of(const int32_t *p) { return CodeSums{p, 1, 0}; }
// Up to eight such sums in one launch (code_sums_kernel), by kind:
//   kSumRows   per row: out [rows]
//   kSumCols   per column over the rows, in pieces: out [sum_pieces(rows, cols)][cols]
//   kSumEdges  rows = the positions of N images of H x W, cols = channels: per channel over the positions of the first row, last
//              row, first column, last column and the four corners (first row: first, last column; last row: the same) of
//              every image: added to out64 [8][cols], which is zero beforehand
// out64 (kSumCols): the whole sums are added to out64 [cols], which is zero beforehand, instead.
// cols a multiple of 16, q 16-byte aligned, fewer than 2^31 rows.  zero: regions of 32-bit words the launch clears (a
// status word, sums that a later kernel adds to).
enum { kSumRows = 0, kSumCols = 1, kSumEdges = 2 };
struct SumJob { const void *q; int64_t rows, cols; int kind, is_signed; int32_t *out; int H = 0, W = 0; int64_t *out64 = nullptr; };
constexpr int kMaxSumJobs = 8;
int sum_pieces(int64_t rows, int64_t cols);
inline size_t sum_elems(int64_t rows, int64_t cols, int kind)
{
    return kind == kSumRows ? (size_t)rows : kind == kSumCols ? (size_t)sum_pieces(rows, cols) * (size_t)cols : 8 * (size_t)cols;
}
inline size_t sum_elems(const SumJob &j) { return sum_elems(j.rows, j.cols, j.kind); }
inline CodeSums sums_of(const SumJob &j)
{
    return j.kind == kSumRows ? sums_of(j.out) : CodeSums{j.out, sum_pieces(j.rows, j.cols), j.cols};
}
// beside (nullable): set when the product launched next may run beside this kernel (see launch()).  Sums of fewer than a megabyte
// take a microsecond or two, less than the product's launch, and sums of more than 32 want HBM for themselves: both let it go at their
// start, ahead of their own wait, and it waits for them in every role (weight gradient 8192 x 2048 x 4096 with its 67 MB 123.7 us beside them, 122.8 behind; linear layer
// 1024 x 2048 -> 1008 with 4 MB 77.6 and 78.3).
constexpr int64_t kSumsBesideMin = 1 << 20, kSumsBesideMax = 32 << 20;
int launch_code_sums(const SumJob *jobs, int count, cudaStream_t st, const ZeroJobs &zero = ZeroJobs{}, bool *beside = nullptr);

// ---- per-tensor range scan (qbp_quant.cu): leaves *nparts (min, max) pairs at ws, for RangeSrc::parts -------------
size_t range_scan_ws_bytes();
int range_scan(const float *x, int64_t n, void *ws, size_t ws_bytes, int *nparts, cudaStream_t st);

// ---- pieces the whole-layer composition chains without a pass of their own ------
// Range BN backward that also leaves per-block (min, max) of dx (qbp_rangebn.cu), and the gradient
// bifurcation that starts from such partials instead of scanning (qbp_quant.cu).
int rangebn_bwd_impl(const float *dy, const float *x, int64_t n, int64_t C, const float *gamma, const float *beta,
                     int relu, const float *save_mean, const float *save_min, const float *save_max, float *dx,
                     float *dgamma, float *dbeta, void *ws, size_t ws_bytes, float2 *range_parts, int *nparts,
                     cudaStream_t st);
size_t rangebn_range_parts_capacity(int64_t C);
// Range BN backward and the bifurcation of the gradient in two passes, the fp32 gradient optional (qbp_rangebn.cu).
bool rangebn_bwd_one_launch(int64_t n, int64_t C);
bool rangebn_bwd_bifurcate_supported(const float *dy, const float *x, const float *g_out, int64_t n, int64_t C);
int rangebn_bwd_bifurcate_impl(const float *dy, const float *x, int64_t n, int64_t C, const float *gamma, const float *beta,
                               int relu, const float *save_mean, const float *save_min, const float *save_max, float *g_out,
                               float *dgamma, float *dbeta, uint64_t seed, uint32_t id8, uint32_t id16, int8_t *q8,
                               qbp_qparams *qp8, int32_t *row_sums8, int8_t *hi, uint8_t *lo, qbp_qparams *qp16, bool lo_signed,
                               void *ws, size_t ws_bytes, cudaStream_t st, int64_t *tot16 = nullptr, void *clear = nullptr,
                               int64_t clear_words = 0, const SumJob *extra = nullptr, int extra_count = 0);
// (tot16 (nullable) [C]: per-channel totals of the stored 16-bit codes; clear: 32-bit words cleared at the start, tot16 among
// them; extra: code sums taken beside the per-channel reduction)
int bifurcate_with_range_partials(const float *g, int64_t rows, int64_t cols, uint64_t seed, uint32_t tensor_id8,
                                  uint32_t tensor_id16, int8_t *q8, qbp_qparams *qp8, int32_t *row_sums8, int8_t *hi,
                                  uint8_t *lo, qbp_qparams *qp16, const float2 *partials, int nparts, cudaStream_t st,
                                  int64_t *tot16 = nullptr, bool lo_signed = false);
// The layer's operands quantised to 8 bits (nearest rounding, clamping values = min and max): the activation (nullable) and the
// weights, in two launches.  row_sums [rows] / tot [cols] / col_sums [sum_pieces(rows, cols)][cols] (each nullable): wanted sums of the
// stored codes; *_left: whether the quantising kernel left them (it depends on the shape; the caller sums the codes up otherwise).
// tot is cleared either way, and so are clear_words 32-bit words at `clear`.  add_rows: row sums may be added up in pieces (slower
// than whole rows; worth it where no launch for other sums follows).
struct QuantOperand {
    const float *v; int64_t rows, cols; int8_t *q; qbp_qparams *qp; int32_t *row_sums; int64_t *tot; int32_t *col_sums;
    bool row_sums_left = false, tot_left = false, col_sums_left = false;
};
size_t quantize_operands_ws_bytes();
int quantize_operands(QuantOperand *x, QuantOperand *w, int *status, void *ws, size_t ws_bytes, cudaStream_t st, bool add_rows,
                      void *clear = nullptr, int64_t clear_words = 0);
bool quantizer_totals_supported(int64_t cols);
// The convolution products with the per-pixel channel sums of the input codes supplied by the caller
// (nullable: computed here) (qbp_mma.cu).
// Per-column (sum, min, max) of a product's fp32 output as partial rows [rows][N], one per CTA
// of the tensor-core kernel; `rows` is filled in by the launch.  colstat_rows_max(): the most rows a launch leaves.
struct ColStatParts { float *lo, *hi; double *sum; int rows; };
int colstat_rows_max();
int rangebn_fold_from_parts(int64_t n, int64_t C, const float *gamma, const float *beta, int relu, float *save_mean,
                            float *save_min, float *save_max, const ColStatParts &parts, qbp_qparams *qp8_out,
                            float4 *fold, cudaStream_t st);
// Optional tail of a product's epilogue: per-column normalisation (fold: (mean, scale, gamma, beta) per output
// column, as rangebn_fold_from_parts leaves them), ReLU, and 8-bit codes of the result with parameters *rq
// (q [M x N], row_sums [M] nullable).  keep_terms: the zero-point term kernels ran for the same operands in the
// call just before on the same workspace and are not run again.
// w_sums (nullable): the filter's code sums (forward [K * taps], layer gradient [taps * C]) are there already.
// extra [extra_count] (3 x 3): code sums of a later product, taken in the launch that makes this one's correction terms.
// beside: the launch before the call was code_sums_kernel (see launch()).
struct EpilogueTail { const float4 *fold; int relu; const qbp_qparams *rq; int8_t *q; int32_t *row_sums; int keep_terms; const CodeSums *w_sums;
                      const SumJob *extra = nullptr; int extra_count = 0; bool beside = false; };
size_t filter_sum_elems(const qbp_conv_desc *d);
SumJob filter_sum_job(const qbp_conv_desc *d, bool dgrad, const int8_t *w, int32_t *out);

// ext_status (here and below; nullable): a status word the caller owns and has cleared -- the product raises it when
// a bounded wait runs out and never clears it; NULL: the word is the first int of `ws`, cleared by the call itself.
int conv_s8_impl(int mode, const qbp_conv_desc *d, const int8_t *in, const qbp_qparams *q_in, const int8_t *wgt,
                 const qbp_qparams *q_w, int32_t *acc_out, float *out, const int32_t *in_chan_sum, ColStatParts *stats,
                 int *ext_status, void *ws, size_t ws_bytes, cudaStream_t st, const EpilogueTail *tail = nullptr);
int gemm_s8_impl(int transA, int transB, int64_t M, int64_t N, int64_t K, const int8_t *A, const qbp_qparams *qa,
                 const int8_t *B, const qbp_qparams *qb, int32_t *acc_out, float *C, const qbp_epilogue *ep,
                 int *ext_status, void *ws, size_t ws_bytes, cudaStream_t st, const CodeSums *a_sums = nullptr,
                 const CodeSums *b_sums = nullptr, bool beside = false);
// tot_x [C] / tot_g16 [K] (convolution; nullable, both or none): per-channel totals of the stored x codes and of the
// stored 16-bit gradient codes (256 * hi + lo) over all positions, left by the kernels that wrote the codes.  tot_g16 [N] alone:
// a plain product's, of at most kWgPieceRows rows.
// lo_signed: g_lo holds the low bytes with the top bit flipped, i.e. the signed bytes lo - 128 (lo_signed in
// bifurcate_with_range_partials): g16 - zg = 256 * hi + (lo - 128) - (zg - 128), so the two limbs have one operand
// type and run as one product of twice the columns (the x tile is read from shared memory once, not once per limb),
// with zg - 128 as the zero-point.
int wgrad_s16_impl(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K, const int8_t *x, const qbp_qparams *qx,
                   const int8_t *g_hi, const uint8_t *g_lo, const qbp_qparams *qg16, int64_t *acc_out, float *dW,
                   int *ext_status, void *ws, size_t ws_bytes, cudaStream_t st, const int64_t *tot_x = nullptr,
                   const int64_t *tot_g16 = nullptr, bool tot_g_filled = true, bool lo_signed = false,
                   const SumJob *done_sums = nullptr);
// The sums behind the zero-point terms.  Plain product: the columns of x, hi, lo in pieces (3 jobs), or, when that would make the
// pieces long, as for a convolution: added to one cleared table of int64 (tab: x [C], hi [N], lo [N]; 3 x 3: then [8][C], [8][N],
// [8][N] over the images' edges; 3 or 6 jobs); with totals (tot_x, tot_g16) the first three are not needed.  done_sums (above): the caller has run the needed
// ones into these buffers, and has cleared tot_g16 when tot_g_filled is false.
int wgrad_sum_jobs(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K, const int8_t *x, const int8_t *hi, const uint8_t *lo,
                   bool lo_signed, int64_t *tab, SumJob (&jobs)[6]);
size_t wgrad_sum_table(const qbp_conv_desc *d, int64_t M, int64_t N, int64_t K);        // int64 entries of tab (0: sums in pieces)
// tot_g_filled == false: tot_g16 is a cleared buffer [K] that the product fills itself (possible when wgrad_self_totals(d)).
bool wgrad_self_totals(const qbp_conv_desc *d);
// Shapes the convolution products / the convolution weight gradient implement.
bool conv_supported(const qbp_conv_desc *d);
bool wgrad_conv_supported(const qbp_conv_desc *d);
// Range BN forward from such partials instead of a statistics pass over x (qbp_rangebn.cu).
// out_range / rq (each nullable): the exact range of y / its 8-bit codes for the next layer (see qbp_requant); totals_cleared:
// rq->chan_sums is zero already.
int rangebn_fwd_from_parts(const float *x, int64_t n, int64_t C, const float *gamma, const float *beta, int relu, float *y,
                           float *save_mean, float *save_min, float *save_max, const ColStatParts &parts,
                           qbp_qparams *out_range, const qbp_requant *rq, cudaStream_t st, bool totals_cleared = false);

// ---- TMA tensor maps ---------------------------------------------------------
// A dense byte matrix [rows x cols] (cols innermost) read in boxes of
// box_cols x box_rows; box_cols in {32, 64, 128} selects the matching swizzle.
int make_map_2d(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_cols);
// A dense NHWC byte tensor read in boxes of box_c x bw x bh x bn.
int make_map_nhwc(CUtensorMap *map, const void *base, uint64_t N, uint64_t H, uint64_t W, uint64_t C, uint32_t bn,
                  uint32_t bh, uint32_t bw, uint32_t box_c);

// fp32 output matrix [rows x cols] stored by TMA in boxes of 32 rows x 32 columns (128-byte swizzled slabs).
int make_map_out_2d(CUtensorMap *map, float *base, uint64_t rows, uint64_t cols);
// fp32 NHWC output stored in boxes of 32 channels x (sw x sh x sn = 32 pixels).
int make_map_out_nhwc(CUtensorMap *map, float *base, uint64_t N, uint64_t H, uint64_t W, uint64_t C, uint32_t sn,
                      uint32_t sh, uint32_t sw);

// ---- the dense product on CTA pairs (qbp_mma2.cu) -------------------------------
bool gemm2_eligible(int transB, int64_t M, int64_t N, int64_t K);
int launch_gemm2(int transA, int transB, int64_t M, int64_t N, int64_t K, const int8_t *A, const qbp_qparams *qa,
                 const int8_t *B, const qbp_qparams *qb, int32_t *acc_out, float *C, const CodeSums &a_sums,
                 const CodeSums &b_sums, int *status, bool beside, cudaStream_t st);

// ---- the 3 x 3 convolution products on CTA pairs (qbp_conv2.cu); bwl / bhl: log2 of the position box's extents ----
bool conv2_eligible(const qbp_conv_desc *d, bool dgrad);
int launch_conv2(bool dgrad, const qbp_conv_desc *d, const int8_t *in, const qbp_qparams *q_in, const int8_t *wgt,
                 const qbp_qparams *q_w, int32_t *acc_out, float *out, const int32_t *rowterm, const int32_t *colterm,
                 ColStatParts *stats, int *status, int bwl, int bhl, bool beside, cudaStream_t st);
// ... and those whose output's statistics nobody wants
struct ConvTPlan { int npos, tiles_n, units, windows, stages; uint32_t window_bytes; double cost; };
bool conv2t_eligible(const qbp_conv_desc *d, bool dgrad, int bwl, int bhl, ConvTPlan &p);
int launch_conv2t(bool dgrad, const qbp_conv_desc *d, const int8_t *in, const qbp_qparams *q_in, const int8_t *wgt,
                  const qbp_qparams *q_w, int32_t *acc_out, float *out, const int32_t *rowterm, const int32_t *colterm,
                  const ConvTPlan &p, int *status, bool beside, cudaStream_t st);

// ---- the dense weight gradient on CTA pairs (qbp_wgrad2.cu) ----------------------
bool wgrad2_eligible(int64_t M, int64_t N, int64_t K);
int launch_wgrad2(int64_t M, int64_t N, int64_t K, const int8_t *x, const qbp_qparams *qx, const int8_t *g_hi,
                  const uint8_t *g_lo, const qbp_qparams *qg16, int64_t *acc_out, float *dW, const CodeSums &sx,
                  const CodeSums &shi, const CodeSums &slo, const int64_t *tot_g, int *status, bool beside, cudaStream_t st, bool lo_signed = false);

// ---- shared-memory operand descriptors ---------------------------------------
// How one operand tile of a pipeline stage is laid out and walked by the MMAs.
struct OperandLayout {
    uint32_t tile_bytes;    // bytes of this operand per stage
    uint32_t desc_lo;       // descriptor bits 16..31 (leading byte offset), address added at run time
    uint32_t desc_hi;       // descriptor bits 32..63 (stride byte offset, version, swizzle)
    uint32_t kstep;         // start-address advance per MMA (K = 32), in 16-byte units
    uint32_t major;         // 0 = K-major, 1 = MN-major (instruction descriptor bit)
};

// K-major tile: `rows` rows of `row_bytes` (32/64/128, swizzled alike) reduction bytes.
OperandLayout layout_kmajor(uint32_t rows, uint32_t row_bytes);
// MN-major tile: `krows` reduction rows of `row_bytes` (32/64/128) M/N bytes each;
// `chunks` such tiles side by side (chunk_stride bytes apart) widen M/N beyond row_bytes.
OperandLayout layout_mnmajor(uint32_t krows, uint32_t row_bytes, uint32_t chunks, uint32_t chunk_stride);

// ---- division by launch-time constants ----------------------------------------
// Division of a non-negative int (< 2^31) by a positive constant known at launch: multiply-high and
// shift (Granlund & Montgomery, "Division by invariant integers using multiplication").  The producer
// and MMA-issue threads run one dependent instruction at a time, so 32-bit divisions (some 25 dependent
// instructions each) per tile and per stage would dominate short tiles.
struct FastDiv {
    uint32_t mul, shr, d;
#ifdef __CUDACC__
    __device__ __forceinline__ int div(int n) const { return d == 1 ? n : (int)(__umulhi((uint32_t)n, mul) >> shr); }
    __device__ __forceinline__ void divmod(int n, int &q, int &r) const { q = div(n); r = n - q * (int)d; }
#endif
};
inline FastDiv make_fastdiv(int d)
{
    FastDiv f; f.d = (uint32_t)d; f.mul = 0; f.shr = 0;
    if (d > 1) {
        int lg = 0; while ((1ll << lg) < d) ++lg;
        const int p = 31 + lg;
        f.mul = (uint32_t)(((1ull << p) + (uint64_t)d - 1) / (uint64_t)d);
        f.shr = (uint32_t)(p - 32);
    }
    return f;
}

uint32_t make_idesc(bool a_signed, bool b_signed, uint32_t a_major, uint32_t b_major, uint32_t m, uint32_t n);

}  // namespace qbp
