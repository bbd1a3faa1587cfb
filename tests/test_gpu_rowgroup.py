"""The row-group kernel of the row-split family: one group of lanes per row, one or four lane sets, loads of 16, 8, 4 or 2
bytes by what width and operands allow.  Rows at the edges of a batch, of a group of lanes and of the longest sum one lane
set may take (512 terms), with empty rows between them."""
import numpy as np
import pytest

import workloads as W
pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    import paper_2608_05033_b200 as sd
    from test_gpu_parity import check
    from util import DeviceWorkload, run_spmm


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [5, 8, 12, 31, 34, 64, 97, 132, 260, 521])
@pytest.mark.parametrize("edges", [[0, 1, 7, 8, 9, 15], [11, 12, 13, 0, 31, 33], [0, 1, 31, 32, 33, 512], [64, 127, 0, 513, 2047, 2048]])
def test_row_group_lengths_widths_and_alignment(edges, N, dtype):
    rng = np.random.default_rng(N + len(edges))
    M, K = 203, 2100
    lengths = rng.permutation(np.resize(edges, M))
    w = W.random_csr(M, K, N, lengths, seed=N, dtype=dtype, alpha=-0.75, beta=0.5)
    dw = DeviceWorkload(w)
    plan = dw.plan(family=sd.SD_ROWSPLIT)
    for kw in (dict(), dict(pad_b=3, pad_c=5), dict(offset=1), dict(offset=2, pad_b=2)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
        again, _ = run_spmm(plan, w, **kw)
        assert np.array_equal(got, again)
    got, _ = run_spmm(plan, w, c_fill=np.full((M, N), np.nan, np.float32), beta=0.0)
    check(w, got, beta=0.0)
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [16, 32, 128, 192, 256])
@pytest.mark.parametrize("edges", [[5], [0, 1, 2, 9], [15, 16, 17, 31], [39, 40, 47, 0], [63, 64, 65, 128]])
def test_whole_widths_at_the_lines_of_the_rule(edges, N, dtype):
    """Enough rows to fill the GPU, lengths on both sides of the lines between the row kernels, of one length and of several; every
    lane has columns (16 to 256) or some have none (192).  A non-finite row of B reaches only the rows that name it."""
    rng = np.random.default_rng(N + len(edges))
    M, K = 12007, 700
    w = W.random_csr(M, K, N, rng.permutation(np.resize(edges, M)), seed=N, dtype=dtype, alpha=-0.75, beta=0.5)
    plan = DeviceWorkload(w).plan(family=sd.SD_ROWSPLIT)
    got, intact = run_spmm(plan, w)
    assert intact
    check(w, got)
    assert np.array_equal(got, run_spmm(plan, w)[0])
    w.B[0] = np.inf if dtype == W.SD_F32 else 0x7F80
    named = np.zeros(M, bool)
    named[np.repeat(np.arange(M), np.diff(w.rowptr))[w.colind == 0]] = True
    got, _ = run_spmm(plan, w)
    assert np.isfinite(got[~named]).all() and not np.isfinite(got[named]).any()
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [8, 16, 20, 24, 32, 36, 40, 48, 72, 128, 136, 264])
@pytest.mark.parametrize("M,length", [(11, 5), (90001, 5), (90001, 1), (700000, 3)])
def test_rows_of_one_length(M, length, N, dtype):
    """Short rows of one length: one or two vectors per lane by width and size, idle lanes in the last vector."""
    if M > 100000 and N > 24:
        M = 13_000_000 // N   # either side of 40 MB of C
    K = 1200
    w = W.random_csr(M, K, N, np.full(M, length), seed=N, dtype=dtype, alpha=0.5, beta=-1.5)
    plan = DeviceWorkload(w).plan(family=sd.SD_ROWSPLIT)
    for kw in (dict(), dict(pad_b=8, pad_c=4)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    assert np.array_equal(got, run_spmm(plan, w, **kw)[0])
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("mean", [1, 5, 20, 70])
def test_two_and_four_columns_from_any_offset(mean, N, dtype):
    """A row of B as one load where base and pitch allow it, with four columns also a row of C as one store."""
    rng = np.random.default_rng(mean)
    w = W.random_csr(901, 800, N, rng.poisson(mean, 901), seed=mean, dtype=dtype, alpha=1.5, beta=-0.5)
    plan = DeviceWorkload(w).plan(family=sd.SD_ROWSPLIT)
    for kw in (dict(), dict(offset=1), dict(offset=2), dict(pad_b=1), dict(pad_b=2, pad_c=1), dict(pad_b=4, pad_c=4), dict(offset=4)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    plan.close()


# 16-byte loads per row of B, columns of A, usual and longest row
@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("loads,K,usual,longest", [(2, 9000, 24, 30), (2, 260000, 24, 30), (2, 260000, 36, 40), (4, 9000, 24, 30), (8, 9000, 16, 64), (8, 9000, 33, 40), (8, 130000, 24, 30),
                                                   (8, 130000, 36, 40), (8, 130000, 24, 120), (16, 9000, 24, 30), (16, 9000, 36, 40),
                                                   (16, 9000, 36, 300), (16, 9000, 70, 80), (32, 9000, 20, 30)])
def test_lane_sets_on_matrices_that_fill_the_gpu(loads, K, usual, longest, dtype):
    """More lanes than the GPU holds at five CTAs per SM (189,440), so that the rule goes by loads, mean length, longest row and size of B:
    130,000 columns at eight loads are 16.6 MB, 260,000 at two 8.3."""
    N = loads * (4 if dtype == W.SD_F32 else 8)
    M = 200_000 // min(32, loads)
    rng = np.random.default_rng(loads + usual)
    lengths = rng.integers(usual - 3, usual + 4, M)
    lengths[[0, M // 2, M - 1]] = longest, longest - 1, 0
    w = W.random_csr(M, K, N, lengths, seed=loads, dtype=dtype, alpha=-0.75, beta=0.5)
    plan = DeviceWorkload(w).plan(family=sd.SD_ROWSPLIT)
    got, intact = run_spmm(plan, w)
    assert intact
    check(w, got)
    assert np.array_equal(got, run_spmm(plan, w)[0])
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("loads", [1, 2, 4, 6, 8, 12, 20, 33])
@pytest.mark.parametrize("length", [4, 6, 12, 15])
@pytest.mark.parametrize("near", [False, True])
def test_rows_of_one_length_that_share_rows_of_b(near, length, loads, dtype):
    """Neighbouring rows name neighbouring columns, four nonzeros and more per occupied 16x16 block, or any: either side of the lines
    between the plain and the row-group kernel, with more lanes than the GPU holds."""
    N = loads * (4 if dtype == W.SD_F32 else 8)
    M, K = 200_000 // min(32, loads) + 3, 5000
    w = W.random_csr(M, K, N, np.full(M, length), seed=loads, dtype=dtype, alpha=0.5, beta=-1.5)
    if near:
        w.colind[:] = (np.arange(M)[:, None] // 4 % (K - length) + np.arange(length)).reshape(-1)
    plan = DeviceWorkload(w).plan(family=sd.SD_ROWSPLIT)
    assert (w.colind.size >= 4 * plan.info().nnzb16) == near
    got, intact = run_spmm(plan, w)
    assert intact
    check(w, got)
    assert np.array_equal(got, run_spmm(plan, w)[0])
    plan.close()
