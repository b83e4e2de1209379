"""GPU integer products (tcgen05 int8 GEMM, implicit-GEMM convolution, limb-split weight gradient)
vs the CPU oracle: int32 / int64 accumulators bit for bit, fp32 outputs identical (same single multiply)."""
import numpy as np
import pytest

from oracle import qbp_oracle as O
from paper_1805_11046_b200 import synth
from tests.util import random_codes, set_qparams, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import paper_1805_11046_b200.binding as binding
    return binding


def _qp(B, scale, zp):
    return set_qparams(B.new_qparams(1), scale, zp)


# ------------------------------------------------------------------ GEMM
GEMMS = [(128, 128, 128), (64, 128, 256), (64, 256, 128), (16, 16, 16), (208, 80, 144), (256, 384, 512),
         (384, 640, 1040), (128, 272, 33024)]


@pytest.mark.parametrize("M,N,K", GEMMS)
@pytest.mark.parametrize("tA,tB", [(False, False), (False, True), (True, False), (True, True)])
def test_gemm_s8(B, M, N, K, tA, tB):
    A = random_codes((K, M) if tA else (M, K), 1); Bm = random_codes((N, K) if tB else (K, N), 2)
    za, zb, sa, sb = 3, -128, 0.5, 0.25
    if K > 30000:                       # keep the exact sum inside int32: small codes at the longest legal K
        A = (A // 4).astype(np.int8); Bm = (Bm // 4).astype(np.int8); zb = -5
    acc, out, ws = B.qbp_gemm_s8(to_dev(A), _qp(B, sa, za), to_dev(Bm), _qp(B, sb, zb), transA=tA, transB=tB, want_acc=True)
    oacc, oout, bad = O.gemm_s8(A, za, Bm, zb, sa, sb, transA=tA, transB=tB)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc)
    assert np.array_equal(to_host(out), oout)


def test_gemm_extreme_codes_and_zero_points(B):
    M, N, K = 128, 128, 33024 // 2
    A = np.full((M, K), -128, np.int8); Bm = np.full((K, N), 127, np.int8)
    acc, _, ws = B.qbp_gemm_s8(to_dev(A), _qp(B, 1, 127), to_dev(Bm), _qp(B, 1, -128), want_acc=True, want_out=False)
    assert B.status_word(ws) == 0
    assert np.all(to_host(acc) == (-255) * 255 * K)


def test_gemm_dense_sweep_shape_sampled_rows(B):
    """4096^3 from the dense sweep, operands quantised from N(0,1); oracle on 192 sampled rows."""
    case = synth.dense_gemm(4096, 4096, 4096)
    qa, qpa = B.qbp_quantize_s8(to_dev(case["a"])); qb, qpb = B.qbp_quantize_s8(to_dev(case["b"]))
    oa = O.quantize(case["a"], 8); ob = O.quantize(case["b"], 8)
    assert np.array_equal(to_host(qa), oa.q) and np.array_equal(to_host(qb), ob.q)
    acc, out, ws = B.qbp_gemm_s8(qa, qpa, qb, qpb, want_acc=True)
    assert B.status_word(ws) == 0
    rows = np.unique(np.concatenate([[0, 127, 128, 4095, 3968], np.random.Generator(np.random.PCG64(5)).integers(0, 4096, 187)]))
    oacc, oout, bad = O.gemm_s8(oa.q[rows], oa.zero_point[0], ob.q, ob.zero_point[0], oa.scale[0], ob.scale[0])
    assert bad == 0
    assert np.array_equal(to_host(acc)[rows], oacc) and np.array_equal(to_host(out)[rows], oout)


def test_gemm_dense_sweep_8192_sampled_rows_and_corner_tiles(B):
    """8192^3 from the dense sweep in the benchmark's launch configuration (256 x 256 tiles, several tiles per CTA);
    oracle on 64 random rows plus the rows of the four corner tiles' edges."""
    n = 8192
    case = synth.dense_gemm(n, n, n)
    qa, qpa = B.qbp_quantize_s8(to_dev(case["a"])); qb, qpb = B.qbp_quantize_s8(to_dev(case["b"]))
    oa = O.quantize(case["a"], 8); ob = O.quantize(case["b"], 8)
    assert np.array_equal(to_host(qa), oa.q) and np.array_equal(to_host(qb), ob.q)
    acc, out, ws = B.qbp_gemm_s8(qa, qpa, qb, qpb, want_acc=True)
    assert B.status_word(ws) == 0
    rows = np.unique(np.concatenate([[0, 127, 128, 255, 256, n - 256, n - 129, n - 128, n - 1],
                                     np.random.Generator(np.random.PCG64(6)).integers(0, n, 64)]))
    oacc, oout, bad = O.gemm_s8(oa.q[rows], oa.zero_point[0], ob.q, ob.zero_point[0], oa.scale[0], ob.scale[0])
    assert bad == 0
    assert np.array_equal(to_host(acc[rows]), oacc) and np.array_equal(to_host(out[rows]), oout)


def _dense_gemm_sampled(B, M, N, K, seed, n_random=64):
    """One product of the dense sweep in the benchmark's launch configuration: operands quantised from N(0,1) on both
    sides (codes compared in full), accumulators and fp32 outputs compared on the rows at the tile edges plus
    n_random random rows, every column."""
    case = synth.dense_gemm(M, N, K, parts=("a", "b"))
    qa, qpa = B.qbp_quantize_s8(to_dev(case["a"])); qb, qpb = B.qbp_quantize_s8(to_dev(case["b"]))
    oa = O.quantize(case["a"], 8); ob = O.quantize(case["b"], 8)
    del case
    assert np.array_equal(to_host(qa), oa.q) and np.array_equal(to_host(qb), ob.q)
    acc, out, ws = B.qbp_gemm_s8(qa, qpa, qb, qpb, want_acc=True)
    assert B.status_word(ws) == 0
    rows = np.unique(np.concatenate([[0, 127, 128, 255, 256, 511, 512, M - 512, M - 257, M - 256, M - 129, M - 128, M - 1],
                                     np.random.Generator(np.random.PCG64(seed)).integers(0, M, n_random)]))
    oacc, oout, bad = O.gemm_s8(oa.q[rows], oa.zero_point[0], ob.q, ob.zero_point[0], oa.scale[0], ob.scale[0])
    assert bad == 0
    assert np.array_equal(to_host(acc[rows]), oacc) and np.array_equal(to_host(out[rows]), oout)


def test_gemm_dense_sweep_16384_sampled_rows(B):
    """The largest cube of the dense sweep (16384^3, 512 x 256 pair tiles, 32 x 64 of them over 74 CTA pairs)."""
    _dense_gemm_sampled(B, 16384, 16384, 16384, 8, n_random=32)


# (M, N, K) combinations of the sweep that are not cubes: tall, wide, deep and shallow ones
NONCUBE = [(4096, 16384, 8192), (16384, 4096, 4096), (8192, 4096, 16384), (4096, 8192, 16384)]


@pytest.mark.parametrize("M,N,K", NONCUBE)
def test_gemm_dense_sweep_noncube_sampled_rows(B, M, N, K):
    _dense_gemm_sampled(B, M, N, K, 9 + M // 4096 + N // 2048, n_random=48)


def _dense_wgrad_sampled(B, M, N, K, seed, n_cols):
    """The limb-split 16 x 8-bit product dW [K x N] = X [M x K]^T G [M x N] of the dense sweep: operands quantised from
    N(0,1) (nearest for the 8-bit side, stochastic for the 16-bit side, codes compared in full); int64
    accumulators and fp32 outputs compared on the output columns at the tile edges plus random ones, every row."""
    case = synth.dense_gemm(M, N, K, parts=("x", "g"))
    qx, qpx = B.qbp_quantize_s8(to_dev(case["x"]))
    q16, hi, lo, qpg = B.qbp_quantize_s16(to_dev(case["g"]), rounding=B.QBP_ROUND_STOCHASTIC, seed=3, tensor_id=7)
    ox = O.quantize(case["x"], 8); og = O.quantize(case["g"], 16, rounding=1, seed=3, tensor_id=7)
    del case
    assert np.array_equal(to_host(qx), ox.q) and np.array_equal(to_host(q16), og.q)
    del q16
    acc, dW, ws = B.qbp_wgrad_s16(qx, qpx, hi, lo, qpg, want_acc=True)
    assert B.status_word(ws) == 0
    cols = np.unique(np.concatenate([[0, 127, 128, N - 129, N - 128, N - 1],
                                     np.random.Generator(np.random.PCG64(seed)).integers(0, N, n_cols)]))
    oacc, oout = O.gemm_s16s8(ox.q, ox.zero_point[0], np.ascontiguousarray(og.q[:, cols]), og.zero_point[0], ox.scale[0], og.scale[0])
    assert np.array_equal(to_host(acc[:, cols]), oacc) and np.array_equal(to_host(dW[:, cols]), oout)


@pytest.mark.parametrize("n,n_cols", [(8192, 48), (16384, 16)])
def test_wgrad_dense_sweep_large_cubes_sampled_columns(B, n, n_cols):
    """8192^3 and 16384^3: the reduction over M is split over CTAs in chunks of at most 65536 rows and summed in int64."""
    _dense_wgrad_sampled(B, n, n, n, 10 + n // 8192, n_cols)


@pytest.mark.parametrize("M,N,K", NONCUBE)
def test_wgrad_dense_sweep_noncube_sampled_columns(B, M, N, K):
    _dense_wgrad_sampled(B, M, N, K, 20 + M // 4096 + K // 2048, 24)


# Shapes the CTA-pair kernel takes (at least eight rounds of 256 x 256 tiles over the SM pairs) with ragged edges in
# every dimension: 512 x 256 pair tiles, several rounds of them.
PAIR_GEMMS = [(8208, 8464, 208), (1104, 38000, 144), (2048, 19216, 400)]


@pytest.mark.parametrize("M,N,K", PAIR_GEMMS)
@pytest.mark.parametrize("tA,tB", [(False, False), (False, True), (True, False), (True, True)])
def test_gemm_s8_pair_kernel_ragged_sampled_rows(B, M, N, K, tA, tB):
    """Oracle on the rows at the tile and pair-half edges, the ragged last rows and 48 random ones; every column."""
    A = random_codes((K, M) if tA else (M, K), 11); Bm = random_codes((N, K) if tB else (K, N), 12)
    za, zb, sa, sb = -7, 19, 0.125, 0.5
    acc, out, ws = B.qbp_gemm_s8(to_dev(A), _qp(B, sa, za), to_dev(Bm), _qp(B, sb, zb), transA=tA, transB=tB, want_acc=True)
    assert B.status_word(ws) == 0
    edge = [0, 127, 128, 255, 256, 383, 384, 511, 512, M - 1, M - 2, (M // 512) * 512 - 1, (M // 256) * 256 - 1,
            min((M // 256) * 256, M - 1), min((M // 128) * 128, M - 1)]
    rows = np.unique(np.concatenate([edge, np.random.Generator(np.random.PCG64(M)).integers(0, M, 48)]))
    Arows = np.ascontiguousarray(A[:, rows]) if tA else A[rows]
    oacc, oout, bad = O.gemm_s8(Arows, za, Bm, zb, sa, sb, transA=tA, transB=tB)
    assert bad == 0
    assert np.array_equal(to_host(acc[rows]), oacc) and np.array_equal(to_host(out[rows]), oout)


# Products that fit the SM pairs once: pair tiles of 64, 128 and 256 columns, ragged in every dimension (the fourth has
# more than 2048 rows and still takes tiles of 256), and deep ones smaller than a tile; then two rounds of 256 x 256
# tiles of more than 2048 rows, and one of 512 x 256 tiles of fewer.
SMALL_PAIR_GEMMS = [(272, 304, 144), (256, 256, 1040), (2064, 1008, 144), (4368, 784, 272), (16, 64, 1024), (144, 208, 1040), (2320, 4112, 144), (592, 8208, 144)]


@pytest.mark.parametrize("M,N,K", SMALL_PAIR_GEMMS)
@pytest.mark.parametrize("tA,tB", [(False, False), (False, True), (True, False), (True, True)])
def test_gemm_s8_pair_kernel_narrow_tiles(B, M, N, K, tA, tB):
    A = random_codes((K, M) if tA else (M, K), 13); Bm = random_codes((N, K) if tB else (K, N), 14)
    za, zb, sa, sb = 23, -5, 0.25, 0.5
    acc, out, ws = B.qbp_gemm_s8(to_dev(A), _qp(B, sa, za), to_dev(Bm), _qp(B, sb, zb), transA=tA, transB=tB, want_acc=True)
    assert B.status_word(ws) == 0
    oacc, oout, bad = O.gemm_s8(A, za, Bm, zb, sa, sb, transA=tA, transB=tB)
    assert bad == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(out), oout)


# ------------------------------------------- column statistics from the epilogue
def _check_col_stats(out, stats):
    o = to_host(out).reshape(-1, out.shape[-1]).astype(np.float64)
    csum, cmin, cmax = (to_host(t) for t in stats)
    assert np.array_equal(cmin, o.min(axis=0).astype(np.float32)) and np.array_equal(cmax, o.max(axis=0).astype(np.float32))
    # partial sums of at most 32 fp32 values in fp32, the rest in fp64
    assert np.allclose(csum, o.sum(axis=0), rtol=0, atol=1e-6 * np.abs(o).sum(axis=0).max())


@pytest.mark.parametrize("M,N,K", [(128, 128, 128), (208, 80, 144), (1024, 256, 512), (2000, 64, 64)])
def test_gemm_epilogue_column_statistics(B, M, N, K):
    """Section 3: the sum, minimum and maximum of every output column, as the following Range BN needs them, taken
    from the fp32 outputs in the product's epilogue; the product itself is unchanged."""
    A = random_codes((M, K), 21); Bm = random_codes((K, N), 22)
    za, zb, sa, sb = 5, -9, 0.5, 0.125
    acc, out, ws, stats = B.qbp_gemm_s8(to_dev(A), _qp(B, sa, za), to_dev(Bm), _qp(B, sb, zb), want_acc=True, col_stats=True)
    oacc, oout, bad = O.gemm_s8(A, za, Bm, zb, sa, sb)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(out), oout)
    _check_col_stats(out, stats)


@pytest.mark.parametrize("N,H,W,C,K,R", [(2, 56, 56, 64, 64, 3), (3, 10, 12, 32, 48, 3), (4, 7, 7, 256, 128, 1), (2, 20, 17, 128, 32, 3)])
@pytest.mark.parametrize("mode", [0, 1])
def test_conv_epilogue_channel_statistics(B, N, H, W, C, K, R, mode):
    """The same for a convolution (ragged pixel boxes: positions outside the image must not count)."""
    pad = (R - 1) // 2
    d = B.conv_desc(N, H, W, C, K, R, R, 1, pad); od = O.conv_desc(N, H, W, C, K, R, R, 1, pad)
    inp = random_codes((N, H, W, C if mode == 0 else K), 23); w = random_codes((K, R, R, C), 24)
    zi, zw = -3, 11
    acc, out, ws, stats = B.qbp_conv_s8_implicit(mode, d, to_dev(inp), _qp(B, 0.5, zi), to_dev(w), _qp(B, 0.25, zw),
                                                 want_acc=True, col_stats=True)
    oacc, oout, bad = O.conv_s8(mode, od, inp, zi, w, zw, 0.5, 0.25)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(out), oout)
    _check_col_stats(out, stats)


@pytest.mark.parametrize("N,H,W,C,K,R,mode", [(8, 14, 14, 128, 512, 1, 0), (2, 9, 9, 64, 768, 1, 0), (2, 10, 10, 640, 64, 3, 1),
                                              (64, 28, 28, 128, 512, 1, 0), (64, 14, 14, 64, 768, 1, 0)])
def test_conv_epilogue_channel_statistics_of_wide_outputs(B, N, H, W, C, K, R, mode):
    """More than 256 output channels: several column tiles, each CTA keeping the statistics of the one it meets (two
    and three column tiles, a ragged last one, grids smaller than and as large as the device)."""
    pad = (R - 1) // 2
    d = B.conv_desc(N, H, W, C, K, R, R, 1, pad); od = O.conv_desc(N, H, W, C, K, R, R, 1, pad)
    inp = random_codes((N, H, W, C if mode == 0 else K), 25); w = random_codes((K, R, R, C), 26)
    zi, zw = 7, -2
    acc, out, ws, stats = B.qbp_conv_s8_implicit(mode, d, to_dev(inp), _qp(B, 0.5, zi), to_dev(w), _qp(B, 0.25, zw),
                                                 want_acc=True, col_stats=True)
    oacc, oout, bad = O.conv_s8(mode, od, inp, zi, w, zw, 0.5, 0.25)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(out), oout)
    _check_col_stats(out, stats)


def test_wgrad_dense_sweep_shape_sampled_columns(B):
    """The limb-split 16 x 8-bit product at 4096^3 (dense sweep): operands quantised from N(0,1) (nearest for the
    8-bit side, stochastic for the 16-bit side); oracle on 96 sampled output columns (all 4096 rows of each)."""
    n = 4096
    case = synth.dense_gemm(n, n, n)
    qx, qpx = B.qbp_quantize_s8(to_dev(case["x"]))
    q16, hi, lo, qpg = B.qbp_quantize_s16(to_dev(case["g"]), rounding=B.QBP_ROUND_STOCHASTIC, seed=3, tensor_id=7)
    ox = O.quantize(case["x"], 8); og = O.quantize(case["g"], 16, rounding=1, seed=3, tensor_id=7)
    assert np.array_equal(to_host(qx), ox.q) and np.array_equal(to_host(q16), og.q)
    acc, dW, ws = B.qbp_wgrad_s16(qx, qpx, hi, lo, qpg, want_acc=True)
    assert B.status_word(ws) == 0
    cols = np.unique(np.concatenate([[0, 127, 128, n - 1], np.random.Generator(np.random.PCG64(7)).integers(0, n, 92)]))
    oacc, oout = O.gemm_s16s8(ox.q, ox.zero_point[0], np.ascontiguousarray(og.q[:, cols]), og.zero_point[0], ox.scale[0], og.scale[0])
    assert np.array_equal(to_host(acc)[:, cols], oacc) and np.array_equal(to_host(dW)[:, cols], oout)


# ----------------------------------------------------------- convolution
CONVS = [(2, 8, 8, 64, 64, 1), (2, 8, 8, 64, 64, 3), (3, 10, 12, 32, 48, 3), (2, 14, 14, 128, 256, 3),
         (4, 7, 7, 256, 128, 1), (1, 1, 1, 16, 16, 3), (5, 9, 3, 80, 16, 3), (3, 28, 28, 128, 128, 3),
         (2, 56, 56, 64, 64, 3), (1, 5, 130, 16, 272, 3),
         # boxes loaded once with their border (taps as shifted windows): 128-, 64- and 32-byte channel chunks,
         # several chunks per tile, ragged boxes in both directions
         (2, 20, 17, 128, 32, 3), (2, 20, 17, 32, 128, 3), (1, 33, 9, 192, 32, 3), (2, 16, 8, 256, 16, 3),
         (1, 40, 24, 16, 64, 3)]


@pytest.mark.parametrize("N,H,W,C,K,R", CONVS)
@pytest.mark.parametrize("mode", [0, 1])
def test_conv_s8(B, N, H, W, C, K, R, mode):
    pad = (R - 1) // 2
    d = B.conv_desc(N, H, W, C, K, R, R, 1, pad); od = O.conv_desc(N, H, W, C, K, R, R, 1, pad)
    inp = random_codes((N, H, W, C if mode == 0 else K), 3); w = random_codes((K, R, R, C), 4)
    zi, zw = 7, -128
    acc, out, ws = B.qbp_conv_s8_implicit(mode, d, to_dev(inp), _qp(B, 0.5, zi), to_dev(w), _qp(B, 0.25, zw), want_acc=True)
    oacc, oout, bad = O.conv_s8(mode, od, inp, zi, w, zw, 0.5, 0.25)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc)
    assert np.array_equal(to_host(out), oout)


# --------------------------------------------------------- weight gradient
def _g16(shape, seed):
    return random_codes(shape, seed, -32768, 32767, np.int16)


# (the last four run on CTA pairs: ragged in every dimension, a short and a long reduction)
WGRADS = [(128, 128, 128), (64, 128, 256), (1000, 64, 64), (70000, 32, 48), (4096, 256, 384), (130, 16, 16),
          (1000, 272, 400), (520, 528, 256), (2064, 1040, 784), (4096, 2304, 512)]


@pytest.mark.parametrize("M,N,K", WGRADS)
def test_wgrad_plain(B, M, N, K):
    X = random_codes((M, K), 5); G = _g16((M, N), 6)
    hi, lo = O.limb_split(G)
    zx, zg = -128, 32767
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, zx), to_dev(hi), to_dev(lo), _qp(B, 0.25, zg), want_acc=True)
    oacc, oout = O.gemm_s16s8(X, zx, G, zg, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


@pytest.mark.parametrize("M,N,K", [(48, 64, 18960), (528, 112, 18960), (512, 128, 18944), (64, 144, 18960)])
def test_wgrad_pair_kernel_more_row_tiles_than_pairs(B, M, N, K):
    """Outputs whose 256-row tiles alone fill the SM pairs or do not fit them once: tiles as wide as the columns there are."""
    test_wgrad_plain_pair_kernel_narrow_tiles(B, M, N, K)


@pytest.mark.parametrize("M,N,K", [(640, 64, 528), (656, 272, 304), (624, 512, 512), (624, 496, 512), (558, 1328, 1568), (1162, 1328, 1568)])
def test_wgrad_either_side_of_the_pair_kernels_rule(B, M, N, K):
    """The fewest rows for small and middle outputs, one step short of the latter, tiles that would stay 256 columns wide where the
    single-CTA kernel's fit the SMs once."""
    test_wgrad_plain_pair_kernel_narrow_tiles(B, M, N, K)


# The CTA-pair kernel where it fits the SM pairs once: tiles of 64, 128 and 256 columns, ragged in every dimension, fewer
# reduction steps than the ring has stages and more; outputs smaller than a tile, the fewest rows; the last is just too deep for it.
@pytest.mark.parametrize("M,N,K", [(528, 272, 304), (2064, 256, 256), (560, 1008, 2064), (1536, 784, 4368), (1040, 208, 160),
                                   (512, 64, 528), (16, 1024, 1024), (3312, 256, 256)])
def test_wgrad_plain_pair_kernel_narrow_tiles(B, M, N, K):
    X = random_codes((M, K), 7); G = _g16((M, N), 8)
    hi, lo = O.limb_split(G)
    zx, zg = 11, -77
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, zx), to_dev(hi), to_dev(lo), _qp(B, 0.25, zg), want_acc=True)
    oacc, oout = O.gemm_s16s8(X, zx, G, zg, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


def test_wgrad_long_reduction_extreme_codes(B):
    """131072 rows of extreme codes: each CTA's int32 chunk stays in range, the int64 total is exact."""
    M, N, K = 131072, 32, 32
    X = np.full((M, K), -128, np.int8); G = np.full((M, N), 32767, np.int16)
    G[::2] = -32768
    hi, lo = O.limb_split(G)
    acc, _, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 1, 127), to_dev(hi), to_dev(lo), _qp(B, 1, 0), want_acc=True, want_out=False)
    assert B.status_word(ws) == 0
    assert np.all(to_host(acc) == (-255) * (32767 - 32768) * (M // 2))


def test_wgrad_pair_kernel_longest_reduction_extreme_codes(B):
    """65536 rows, the most one CTA pair accumulates in int32: every low-limb product at 128 * 255, every high-limb
    product at 128 * 128; the int64 combination must still be exact."""
    M, N, K = 65536, 256, 256
    X = np.full((M, K), -128, np.int8); G = np.full((M, N), -32513, np.int16)        # hi = -128, lo = 255
    hi, lo = O.limb_split(G)
    assert hi.min() == hi.max() == -128 and lo.min() == lo.max() == 255
    acc, _, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 1, 0), to_dev(hi), to_dev(lo), _qp(B, 1, 0), want_acc=True, want_out=False)
    assert B.status_word(ws) == 0
    assert np.all(to_host(acc) == (-128) * (-32513) * M)


WCONVS = [(2, 8, 8, 64, 64, 1), (2, 8, 8, 64, 64, 3), (3, 10, 12, 32, 96, 3), (2, 14, 14, 128, 256, 3),
          (4, 7, 7, 256, 128, 1), (1, 1, 1, 32, 32, 3), (2, 28, 28, 128, 128, 3), (3, 9, 5, 96, 160, 3)]


@pytest.mark.parametrize("N,H,W,C,K,R", WCONVS)
def test_wgrad_conv(B, N, H, W, C, K, R):
    pad = (R - 1) // 2
    d = B.conv_desc(N, H, W, C, K, R, R, 1, pad); od = O.conv_desc(N, H, W, C, K, R, R, 1, pad)
    X = random_codes((N, H, W, C), 7); G = _g16((N, H, W, K), 8)
    hi, lo = O.limb_split(G)
    zx, zg = 5, -300
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, zx), to_dev(hi), to_dev(lo), _qp(B, 0.25, zg), d=d, want_acc=True)
    oacc, oout = O.conv_wgrad_s16(od, X, zx, G, zg, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


# ------------------------------------------- ReLU and requantisation in the epilogue (no Range BN after the product)
def _check_requant(B, out_dev, q_dev, qp_dev, rs_dev, oout, relu, rng):
    want = np.maximum(oout, 0) if relu else oout
    if out_dev is not None:
        assert np.array_equal(to_host(out_dev), want)
    o = O.quantize(want, 8, range_in=rng)                # values beyond the clamp saturate
    s_, z_, lo_, hi_ = B.read_qparams(qp_dev)
    assert s_[0] == o.scale[0] and z_[0] == o.zero_point[0] and lo_[0] == o.vmin[0] and hi_[0] == o.vmax[0]
    assert np.array_equal(to_host(q_dev), o.q)
    if rs_dev is not None:
        assert np.array_equal(to_host(rs_dev), o.q.reshape(-1, o.q.shape[-1]).astype(np.int32).sum(1))


@pytest.mark.parametrize("M,N,K", [(128, 128, 128), (208, 80, 144), (1024, 256, 512), (2000, 64, 64), (384, 640, 256)])
@pytest.mark.parametrize("relu,keep_out", [(True, True), (False, False), (True, False)])
def test_gemm_epilogue_relu_and_requantisation(B, M, N, K, relu, keep_out):
    import torch
    A = random_codes((M, K), 31); Bm = random_codes((K, N), 32)
    za, zb, sa, sb = 5, -9, 0.5, 0.125
    _, oout, bad = O.gemm_s8(A, za, Bm, zb, sa, sb)
    assert bad == 0
    hi = np.float32(0.6 * oout.max()); lo = np.float32(0.0 if relu else 0.5 * oout.min())      # a clamp that cuts the tails
    q = torch.empty((M, N), dtype=torch.int8, device="cuda"); qp = B.new_qparams(1); rs = torch.empty(M, dtype=torch.int32, device="cuda")
    res = B.qbp_gemm_s8(to_dev(A), _qp(B, sa, za), to_dev(Bm), _qp(B, sb, zb), want_out=keep_out, relu=relu,
                        requant=(B.range_qparams(lo, hi), q, qp, rs))
    assert B.status_word(res[2]) == 0
    _check_requant(B, res[1] if keep_out else None, q, qp, rs, oout, relu, (lo, hi))


@pytest.mark.parametrize("N_,H,W,C_,K_,R", [(2, 56, 56, 64, 64, 3), (3, 10, 12, 32, 48, 3), (4, 7, 7, 256, 128, 1), (1, 5, 130, 16, 272, 3)])
@pytest.mark.parametrize("mode", [0, 1])
def test_conv_epilogue_relu_and_requantisation(B, N_, H, W, C_, K_, R, mode):
    import torch
    pad = (R - 1) // 2
    d = B.conv_desc(N_, H, W, C_, K_, R, R, 1, pad); od = O.conv_desc(N_, H, W, C_, K_, R, R, 1, pad)
    inp = random_codes((N_, H, W, C_ if mode == 0 else K_), 33); w = random_codes((K_, R, R, C_), 34)
    zi, zw = -3, 11
    _, oout, bad = O.conv_s8(mode, od, inp, zi, w, zw, 0.5, 0.25)
    assert bad == 0
    hi = np.float32(0.7 * oout.max()); lo = np.float32(0.0)
    q = torch.empty(oout.shape, dtype=torch.int8, device="cuda"); qp = B.new_qparams(1)
    rs = torch.empty(oout.size // oout.shape[-1], dtype=torch.int32, device="cuda")
    res = B.qbp_conv_s8_implicit(mode, d, to_dev(inp), _qp(B, 0.5, zi), to_dev(w), _qp(B, 0.25, zw), relu=True,
                                 requant=(B.range_qparams(lo, hi), q, qp, rs))
    assert B.status_word(res[2]) == 0
    _check_requant(B, res[1], q, qp, rs, oout, True, (lo, hi))


@pytest.mark.parametrize("M,N,K", [(128, 128, 128), (208, 80, 144), (1024, 512, 256)])
@pytest.mark.parametrize("tA,tB", [(False, False), (False, True), (True, False), (True, True)])
def test_gemm_with_caller_code_sums(B, M, N, K, tA, tB):
    """The code sums along the reduction handed in (as a chain of calls has them from the quantiser): same product,
    and no sum kernel in the launch list."""
    A = random_codes((K, M) if tA else (M, K), 41); Bm = random_codes((N, K) if tB else (K, N), 42)
    za, zb, sa, sb = 3, -11, 0.5, 0.25
    a_sums = (A.astype(np.int32).sum(0 if tA else 1)).astype(np.int32); b_sums = (Bm.astype(np.int32).sum(1 if tB else 0)).astype(np.int32)
    B.trace_enable(True)
    acc, out, ws = B.qbp_gemm_s8(to_dev(A), _qp(B, sa, za), to_dev(Bm), _qp(B, sb, zb), transA=tA, transB=tB, want_acc=True,
                                 a_sums=to_dev(a_sums), b_sums=to_dev(b_sums))
    names = [n for n, _ in B.trace_records()]
    B.trace_enable(False)
    assert "rowsum_kernel" not in names and "colsum_kernel" not in names
    oacc, oout, bad = O.gemm_s8(A, za, Bm, zb, sa, sb, transA=tA, transB=tB)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(out), oout)


@pytest.mark.parametrize("mode", ["fprop", "dgrad"])
def test_conv_at_full_size_is_reproducible(B, mode):
    """The 64-channel 3x3 convolution of the benchmark, twenty times on the same codes: every run must write the same
    bits.  (Integer accumulators and one fp32 scale leave no room for run-to-run differences; a difference means a
    race -- one was found this way: an output slab refilled while the store of the tile before was still reading it,
    in tiles whose rows lie partly outside the image.)  Each run starts from an output filled with NaN."""
    import torch
    cfg = synth.conv3x3_layer()
    c = cfg["conv"]
    d = B.conv_desc(c["N"], c["H"], c["W"], c["C"], c["K"], c["R"], c["S"], c["stride"], c["pad"])
    src = to_dev(cfg["x"] if mode == "fprop" else cfg["dy"])
    q_in, p_in = B.qbp_quantize_s8(src)
    w = to_dev(cfg["w"])
    q_w, p_w = B.qbp_quantize_s8(w.reshape(c["K"], -1))
    out = torch.empty((c["N"], c["H"], c["W"], 64), dtype=torch.float32, device="cuda")
    ref = None
    for rep in range(20):
        out.fill_(float("nan"))
        B.qbp_conv_s8_implicit(B.QBP_CONV_FPROP if mode == "fprop" else B.QBP_CONV_DGRAD, d, q_in, p_in, q_w.reshape(w.shape), p_w, out=out)
        torch.cuda.synchronize()
        bits = out.view(torch.int32)
        if ref is None:
            ref = bits.clone()
            assert not bool(torch.isnan(out).any())
        else:
            assert int((bits != ref).sum()) == 0, f"run {rep} differs from run 0"


# ------------------------------------------- the weight gradient's two ways of finishing
@pytest.mark.parametrize("M,N,K,shift", [(16, 16, 16, 0), (64, 128, 256, 0), (64, 128, 256, 1), (496, 112, 1008, 0), (1024, 144, 272, 0),
                                         (1040, 128, 272, 0)])
def test_wgrad_plain_whole_and_split_reductions(B, M, N, K, shift):
    """At most 1024 rows stay whole (the product applies the zero-points itself), one more step of rows is split; one A
    tile per CTA while the tiles do not fill the machine; dW on a 16-byte boundary and 4 bytes off it."""
    import torch
    X = random_codes((M, K), 51); G = np.random.Generator(np.random.PCG64(52)).integers(-32768, 32768, (M, N)).astype(np.int16)
    hi, lo = O.limb_split(G)
    dW = torch.full((K * N + 4,), float("nan"), dtype=torch.float32, device="cuda")[shift:shift + K * N].view(K, N)
    acc, _, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, -7), to_dev(hi), to_dev(lo), _qp(B, 0.25, 311), want_acc=True, dW=dW)
    oacc, oout = O.gemm_s16s8(X, -7, G, 311, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


@pytest.mark.parametrize("N,H,W,C,K,R", [(2, 6, 6, 32, 32, 1), (2, 9, 7, 96, 160, 3), (2, 7, 9, 160, 192, 3), (3, 6, 5, 256, 256, 3)])
def test_wgrad_conv_finalize_block_shapes(B, N, H, W, C, K, R):
    """The kernel that adds the partials with two, four and eight output channels per block; channel blocks half filled and
    spanning two accumulator tiles."""
    pad = (R - 1) // 2
    d = B.conv_desc(N, H, W, C, K, R, R, 1, pad); od = O.conv_desc(N, H, W, C, K, R, R, 1, pad)
    X = random_codes((N, H, W, C), 53); G = np.random.Generator(np.random.PCG64(54)).integers(-32768, 32768, (N, H, W, K)).astype(np.int16)
    hi, lo = O.limb_split(G)
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, 9), to_dev(hi), to_dev(lo), _qp(B, 0.25, -77), d=d, want_acc=True)
    oacc, oout = O.conv_wgrad_s16(od, X, 9, G, -77, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


@pytest.mark.parametrize("N,H,W,C,K,R", [(2, 7, 7, 512, 512, 3), (3, 5, 4, 416, 480, 3), (1, 6, 6, 256, 544, 3), (2, 4, 4, 1056, 1024, 1), (9, 8, 8, 480, 96, 3)])
def test_wgrad_conv_finalize_of_whole_items(B, N, H, W, C, K, R):
    """Many output tiles, one or two slices each: every group of threads finishes output channels of its own (several groups of them per
    block, ragged channels on either side, one slice and two, the groups sharing slices beside them)."""
    test_wgrad_conv_finalize_block_shapes(B, N, H, W, C, K, R)


@pytest.mark.parametrize("M", [1, 31, 127, 128, 255, 256, 257, 4095, 8200])
@pytest.mark.parametrize("N,K", [(16, 144), (272, 16)])
def test_wgrad_code_sums_in_pieces_of_the_rows(B, M, N, K):
    """The zero-point terms come from column sums taken in up to 16 pieces of the rows, in strips of 128 columns: one and
    several pieces, uneven ones, strips of one 16-column group and partly filled; signed and unsigned bytes."""
    X = random_codes((M, K), 61); G = np.random.Generator(np.random.PCG64(62)).integers(-32768, 32768, (M, N)).astype(np.int16)
    hi, lo = O.limb_split(G)
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, -101), to_dev(hi), to_dev(lo), _qp(B, 0.25, 12345), want_acc=True)
    oacc, oout = O.gemm_s16s8(X, -101, G, 12345, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


@pytest.mark.parametrize("M", [65535, 65536, 65537, 300001])
@pytest.mark.parametrize("N,K", [(16, 144), (144, 32)])
def test_wgrad_code_sums_of_long_reductions(B, M, N, K):
    """Beyond 65536 rows the column sums are added up in a table instead of pieces: either side of that, many rows."""
    test_wgrad_code_sums_in_pieces_of_the_rows(B, M, N, K)


@pytest.mark.parametrize("N,H,W,C,K", [(600, 1, 3, 32, 64), (5, 7, 1, 160, 32), (150, 2, 4, 64, 288), (700, 3, 3, 32, 32)])
def test_wgrad_conv_edge_sums(B, N, H, W, C, K):
    """The zero-point terms of a 3x3 weight gradient from the operands' sums over all positions less those over the images'
    edges: images of one row or column (both edges at once), edges in one and several pieces, strips of 32, 64 and 128
    channels, partly filled ones."""
    d = B.conv_desc(N, H, W, C, K, 3, 3, 1, 1); od = O.conv_desc(N, H, W, C, K, 3, 3, 1, 1)
    X = random_codes((N, H, W, C), 71); G = np.random.Generator(np.random.PCG64(72)).integers(-32768, 32768, (N, H, W, K)).astype(np.int16)
    hi, lo = O.limb_split(G)
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, -90), to_dev(hi), to_dev(lo), _qp(B, 0.25, 2077), d=d, want_acc=True)
    oacc, oout = O.conv_wgrad_s16(od, X, -90, G, 2077, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


@pytest.mark.parametrize("side", [1, 2])
def test_wgrad_conv_corner_sums_of_many_small_images(B, side):
    """So many images that the low bytes of one corner alone add up to more than an int32 holds (255 * N > 2^31): constant
    codes, whose accumulators are a count of positions times one product."""
    import torch
    N, C, zx, zg = (1 << 31) // 255 + 128, 32, -90, 2077
    d = B.conv_desc(N, side, side, C, C, 3, 3, 1, 1)
    code = lambda v, dt: torch.full((N, side, side, C), v, dtype=dt, device="cuda")
    acc, _, ws = B.qbp_wgrad_s16(code(1, torch.int8), _qp(B, 0.5, zx), code(0, torch.int8), code(255, torch.uint8), _qp(B, 0.25, zg), d=d,
                                 want_acc=True, want_out=False)
    assert B.status_word(ws) == 0
    seen = np.array([side - 1, side, side - 1], np.int64)          # rows (columns) that each tap row (column) sees
    want = N * np.outer(seen, seen) * (1 - zx) * (255 - zg)
    assert np.array_equal(to_host(acc), np.broadcast_to(want[None, :, :, None], (C, 3, 3, C)))


# ------------------------------------------- 3x3 convolutions of many channels (CTA pairs)
@pytest.mark.parametrize("N,H,W,C,K", [(1, 1, 1, 96, 96), (2, 5, 6, 96, 160), (3, 9, 7, 128, 256), (2, 14, 14, 288, 112), (1, 8, 16, 256, 400),
                                       (40, 28, 28, 128, 256), (90, 14, 14, 256, 512)])
@pytest.mark.parametrize("mode", [0, 1])
def test_conv_pairs(B, N, H, W, C, K, mode):
    """One box and an odd number of boxes per column of tiles, channel chunks and column tiles partly filled on either side, tiles of
    128 and of 256 channels (the last two fill the machine), more tiles than pairs; accumulators, output and statistics."""
    d = B.conv_desc(N, H, W, C, K, 3, 3, 1, 1); od = O.conv_desc(N, H, W, C, K, 3, 3, 1, 1)
    inp = random_codes((N, H, W, C if mode == 0 else K), 81); w = random_codes((K, 3, 3, C), 82)
    zi, zw = -31, 14
    acc, out, ws, stats = B.qbp_conv_s8_implicit(mode, d, to_dev(inp), _qp(B, 0.5, zi), to_dev(w), _qp(B, 0.25, zw), want_acc=True, col_stats=True)
    assert B.status_word(ws) == 0
    a, o = to_host(acc).ravel(), to_host(out).ravel()
    idx = np.arange(a.size) if a.size <= 1 << 19 else np.unique(np.concatenate(
        [[0, a.size - 1], np.random.Generator(np.random.PCG64(83)).integers(0, a.size, 1 << 14)]))
    oacc, oout, bad = O.conv_s8(mode, od, inp, zi, w, zw, 0.5, 0.25, idx=idx.astype(np.int64))
    assert bad == 0 and np.array_equal(a[idx], oacc) and np.array_equal(o[idx], oout)
    assert np.array_equal(o, a.astype(np.float32) * np.float32(0.125))
    _check_col_stats(out, stats)


@pytest.mark.parametrize("N,H,W,C,K", [(5, 1, 9, 96, 128), (130, 9, 1, 128, 96), (300, 1, 1, 256, 112), (70, 2, 2, 96, 96), (2, 15, 15, 128, 256),
                                       (1, 3, 96, 96, 272), (2, 3, 97, 96, 128), (1, 6, 130, 160, 96), (3, 1, 200, 96, 96), (1, 2, 255, 128, 128),
                                       (20, 19, 19, 96, 160), (40, 28, 28, 128, 128), (64, 14, 14, 512, 512)])
@pytest.mark.parametrize("mode", [0, 1])
def test_conv_channels_as_rows(B, N, H, W, C, K, mode):
    """Products without statistics.  Images of one row or column (no padding that way, fewer taps), of a tile's exact size, one and
    several panels of columns with a narrower last one, channel chunks partly filled, one and several tiles of a CTA, of one and several tiles of channels."""
    d = B.conv_desc(N, H, W, C, K, 3, 3, 1, 1); od = O.conv_desc(N, H, W, C, K, 3, 3, 1, 1)
    inp = random_codes((N, H, W, C if mode == 0 else K), 84); w = random_codes((K, 3, 3, C), 85)
    acc, out, ws = B.qbp_conv_s8_implicit(mode, d, to_dev(inp), _qp(B, 0.5, 17), to_dev(w), _qp(B, 0.25, -23), want_acc=True)
    assert B.status_word(ws) == 0
    a, o = to_host(acc).ravel(), to_host(out).ravel()
    idx = np.arange(a.size) if a.size <= 1 << 19 else np.unique(np.concatenate(
        [[0, a.size - 1], np.random.Generator(np.random.PCG64(86)).integers(0, a.size, 1 << 14)]))
    oacc, oout, bad = O.conv_s8(mode, od, inp, 17, w, -23, 0.5, 0.25, idx=idx.astype(np.int64))
    assert bad == 0 and np.array_equal(a[idx], oacc) and np.array_equal(o[idx], oout)
    assert np.array_equal(o, a.astype(np.float32) * np.float32(0.125))


# ------------------------------------------------- products that leave most of the machine idle: smaller tiles
@pytest.mark.parametrize("M,N,K", [(48, 4736, 64), (48, 4752, 64), (128, 9488, 32), (240, 96, 160), (2304, 240, 48), (2432, 240, 48),
                                   (16, 37888, 16), (16, 37904, 16)])
@pytest.mark.parametrize("tB", [False, True])
def test_gemm_tiles_that_fit_the_machine_once(B, M, N, K, tB):
    """128-row tiles of 32, 64, 128 and 256 columns are taken while they fit 148 SMs once, each size just inside and just outside;
    a CTA's only tile is read out by all epilogue groups, its columns in chunks that do not divide evenly among them."""
    A = random_codes((M, K), 61); Bm = random_codes((N, K) if tB else (K, N), 62)
    acc, out, ws = B.qbp_gemm_s8(to_dev(A), _qp(B, 0.5, 7), to_dev(Bm), _qp(B, 0.25, -19), transB=tB, want_acc=True)
    oacc, oout, bad = O.gemm_s8(A, 7, Bm, -19, 0.5, 0.25, transB=tB)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(out), oout)


@pytest.mark.parametrize("M,N,K", [(2400, 3600, 1040), (2400, 3600, 4096), (18960, 64, 1040), (18960, 128, 1040), (37904, 64, 1040), (37904, 112, 1040), (37904, 144, 1040), (65520, 64, 1024),
                                   (65536, 64, 1024), (65536, 80, 1024)])
@pytest.mark.parametrize("tA,tB", [(False, False), (False, True), (True, False)])
def test_gemm_pair_kernel_more_row_tiles_than_pairs(B, M, N, K, tA, tB):
    """Outputs whose 256-row tiles alone do not fit the SM pairs once: 512 x 256 tiles, 256-row tiles as wide as the columns, the
    single-CTA kernel; first, two of as many rounds' worth of large as of small tiles; sampled rows, those at the edges of the first and last tiles among them."""
    rows = np.unique(np.concatenate([[0, 127, 128, 255, 256, 511, 512, M - 1, M - 16, M - 17, M // 512 * 512 - 1, M // 256 * 256 - 1],
                                     np.random.Generator(np.random.PCG64(66)).integers(0, M, 120)]))
    A = random_codes((M, K), 67); Bm = random_codes((N, K) if tB else (K, N), 68)
    acc, out, ws = B.qbp_gemm_s8(to_dev(A.T if tA else A), _qp(B, 0.5, 7), to_dev(Bm), _qp(B, 0.25, -19), transA=tA, transB=tB, want_acc=True)
    oacc, oout, bad = O.gemm_s8(A[rows], 7, Bm, -19, 0.5, 0.25, transB=tB)
    assert bad == 0 and B.status_word(ws) == 0
    assert np.array_equal(to_host(acc)[rows], oacc) and np.array_equal(to_host(out)[rows], oout)


@pytest.mark.parametrize("M,N,K", [(64, 32, 128), (128, 4736, 16), (128, 4752, 16), (1024, 1184, 512), (1024, 1200, 512), (144, 176, 240)])
def test_wgrad_tiles_that_fit_the_machine_once(B, M, N, K):
    """Short reductions over tiles of 32, 64 and 128 columns, each size just inside and just outside one wave."""
    X = random_codes((M, K), 63); G = _g16((M, N), 64)
    hi, lo = O.limb_split(G)
    acc, dW, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, -3), to_dev(hi), to_dev(lo), _qp(B, 0.25, 1234), want_acc=True)
    oacc, oout = O.gemm_s16s8(X, -3, G, 1234, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)


@pytest.mark.parametrize("dw_off,acc_off", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("M,N,K", [(2048, 208, 1024), (48, 1024, 1024), (528, 272, 304), (1040, 128, 272), (2048, 64, 48)])
def test_wgrad_outputs_off_the_vector_boundary(B, M, N, K, dw_off, acc_off):
    """dW one float, acc_out one int64 behind a 16-byte boundary, as slices of flat buffers are: shapes that the kernel on CTA pairs
    takes where both lie on one, and shapes that it does not take; what lies before and behind the slices stays."""
    import torch
    X = random_codes((M, K), 65); G = _g16((M, N), 66)
    hi, lo = O.limb_split(G)
    flat_w = torch.full((K * N + 8,), 7.0, dtype=torch.float32, device="cuda"); flat_a = torch.full((K * N + 4,), 7, dtype=torch.int64, device="cuda")
    dW, acc = flat_w[dw_off:dw_off + K * N].view(K, N), flat_a[acc_off:acc_off + K * N].view(K, N)
    assert dW.data_ptr() % 16 == 4 * dw_off and acc.data_ptr() % 16 == 8 * acc_off
    _, _, ws = B.qbp_wgrad_s16(to_dev(X), _qp(B, 0.5, -3), to_dev(hi), to_dev(lo), _qp(B, 0.25, 1234), acc_out=acc, dW=dW)
    oacc, oout = O.gemm_s16s8(X, -3, G, 1234, 0.5, 0.25)
    assert B.status_word(ws) == 0
    assert np.array_equal(to_host(acc), oacc) and np.array_equal(to_host(dW), oout)
    for flat, off in ((flat_w, dw_off), (flat_a, acc_off)):
        assert bool((flat[:off] == 7).all()) and bool((flat[off + K * N:] == 7).all())


@pytest.mark.parametrize("N,H,W,C,K,R", [(1, 8, 16, 128, 128, 3), (2, 12, 12, 128, 160, 3), (6, 16, 16, 256, 96, 1), (5, 11, 13, 96, 160, 3)])
def test_wgrad_conv_one_tile_per_block_and_ragged_columns(B, N, H, W, C, K, R):
    """Reductions short enough that each block takes one tile of 128 rows, from a single step on; output channels that leave most
    of the last tile's columns out."""
    test_wgrad_conv_finalize_block_shapes(B, N, H, W, C, K, R)
