"""One to four columns: a warp owns a range of nonzeros, a lane adds up eight or four consecutive ones, carries join the ranges.  On
matrices whose nonzeros crowd into few columns the kernel keeps those columns' rows of B in shared memory, with columns outside, empty
rows, a row over many ranges."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    import paper_2608_05033_b200 as sd
    from test_gpu_parity import check
    from util import DeviceWorkload, dev, run_spmm


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [2, 3])
def test_frequent_columns_in_shared_memory(N, dtype):
    rng = np.random.default_rng(N)
    M, K = 5203, 70001
    rows = []
    for i in range(M):
        n = 0 if i % 37 == 5 else 30000 if i == 11 else 700
        rows.append(np.unique((K * rng.random(n) ** 5).astype(np.int32)))
    rowptr = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int32)
    cols = np.concatenate(rows).astype(np.int32)
    assert cols.size > 4096 * 600
    vals, B = rng.standard_normal(cols.size).astype(np.float32), rng.standard_normal((K, N)).astype(np.float32)
    C = rng.standard_normal((M, N)).astype(np.float32)
    if dtype == W.SD_BF16:
        vals, B = W.f32_to_bf16_bits(vals), W.f32_to_bf16_bits(B).reshape(K, N)
    w = W.Workload("frequent_columns", M, K, N, rowptr, cols, vals, B, C, -0.75, 0.5, dtype, {})
    plan = DeviceWorkload(w).plan(family=sd.SD_MERGE)
    assert plan.info().plan_bytes > 8 * cols.size      # a row index and a renamed column per nonzero
    for kw in (dict(), dict(pad_b=3, pad_c=1), dict(offset=1)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    again, _ = run_spmm(plan, w, **kw)
    assert np.array_equal(got, again)
    got, _ = run_spmm(plan, w, c_fill=np.full((M, N), np.nan, np.float32), beta=0.0)
    check(w, got, beta=0.0)
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("edges", [[0, 1, 7, 8, 9, 0, 15], [255, 256, 257, 1, 0, 511], [1], [1000, 3, 0, 0, 2048, 5]])
def test_one_column_runs_and_aligned_arrays(edges, offset, dtype):
    lengths = np.resize(edges, 301)
    w = W.random_csr(301, 2500, 1, lengths, seed=len(edges), dtype=dtype, alpha=1.5, beta=-0.5)
    colind, vals = (dev(np.concatenate([np.zeros(offset, a.dtype), a]))[offset:] for a in (w.colind, w.vals))
    plan = sd.Plan(dev(w.rowptr), colind, vals, w.M, w.K, 1, dtype=dtype, family=sd.SD_MERGE)
    got, intact = run_spmm(plan, w)
    assert intact
    check(w, got)
    assert np.array_equal(got, run_spmm(plan, w)[0])
    got, _ = run_spmm(plan, w, c_fill=np.full((w.M, 1), np.nan, np.float32), beta=0.0)
    check(w, got, beta=0.0)
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("M,length,empty", [(1, 3, 0), (1, 700000, 0), (40, 1, 0), (3, 256, 0), (5, 129, 1), (9000, 61, 0), (700000, 1, 0), (60000, 9, 7)])
def test_ranges_of_warps(M, length, empty, N, dtype):
    """One to thousands of warps with a step each or several: a single row over all of them, rows that end with a lane's items, a
    step or a range, rows of one nonzero, empty rows (every seventh), the last step partly filled; operands at any offset."""
    lengths = np.full(M, length)
    lengths[::5] += 3 if length > 1 else 0
    if empty:
        lengths[1::7] = 0
    K = 1500000 if M == 1 else 4000
    w = W.random_csr(M, K, N, lengths, seed=M + N, dtype=dtype, alpha=1.25, beta=-0.5)
    plan = DeviceWorkload(w).plan(family=sd.SD_MERGE)
    for kw in (dict(), dict(pad_b=4 - N, pad_c=1), dict(offset=1)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    assert np.array_equal(got, run_spmm(plan, w, **kw)[0])
    got, _ = run_spmm(plan, w, c_fill=np.full((M, N), np.nan, np.float32), beta=0.0)
    check(w, got, beta=0.0)
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("empty", [False, True])
def test_columns_and_values_from_any_offset(empty, N, dtype):
    """Slices of a longer CSR: columns that begin at every entry of a 32-byte piece, values at the same, at another and, as new values
    of the same plan, at a third; the first row shorter and longer than what is missing of the piece; rows without nonzeros."""
    for first in (1, 2400):
        lengths = np.random.default_rng(first).integers(1, 60, 701)
        lengths[[0, 350]] = first, 2400
        if empty:
            lengths[::7] = 0
        w = W.random_csr(701, 2500, N, lengths, seed=N + first, dtype=dtype, alpha=1.5, beta=-0.5)
        w.B[0] = np.inf if dtype == W.SD_F32 else 0x7F80   # no row names column 0: items that are no nonzeros must not bring it in
        w.colind[w.colind == 0] = 1
        rowptr, column, value = dev(w.rowptr), {}, {}
        for off in range(9):
            column[off], value[off] = (dev(np.concatenate([np.zeros(off, a.dtype), a, np.zeros(8, a.dtype)]))[off:] for a in (w.colind, w.vals))
        for co, vo in [(off, off) for off in range(8)] + [(0, 1), (1, 0), (4, 0), (0, 4), (3, 8), (2, 6)]:
            plan = sd.Plan(rowptr, column[co], value[vo], w.M, w.K, N, dtype=dtype, family=sd.SD_MERGE)
            got, intact = run_spmm(plan, w)
            assert intact
            check(w, got)
            plan.update_values(value[(vo + 3) % 8])
            assert np.array_equal(got, run_spmm(plan, w)[0])
            plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N,empty,offset", [(1, False, 0), (1, False, 3), (1, True, 0), (1, True, 5), (4, True, 1)])
def test_frequent_columns_of_one_and_four_columns(N, empty, offset, dtype):
    """One column from 4,096,000 nonzeros on, rows told by a bit per nonzero or, with empty rows among them, by a row index; four bf16
    columns from 2,457,600 on, four fp32 columns without frequent ones; slices of a longer CSR."""
    rng = np.random.default_rng(N + offset)
    M, K = 9203, 70001
    rows = []
    for i in range(M):
        n = 0 if empty and i % 37 == 5 else 30000 if i == 11 else 700
        rows.append(np.unique((K * rng.random(n) ** 5).astype(np.int32)))
    rowptr = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int32)
    cols = np.concatenate(rows).astype(np.int32)
    assert cols.size > 4096 * 1000
    vals, B = rng.standard_normal(cols.size).astype(np.float32), rng.standard_normal((K, N)).astype(np.float32)
    C = rng.standard_normal((M, N)).astype(np.float32)
    if dtype == W.SD_BF16:
        vals, B = W.f32_to_bf16_bits(vals), W.f32_to_bf16_bits(B).reshape(K, N)
    w = W.Workload("frequent_columns", M, K, N, rowptr, cols, vals, B, C, -0.75, 0.5, dtype, {})
    colind, values = (dev(np.concatenate([np.zeros(offset, a.dtype), a]))[offset:] for a in (cols, vals))
    plan = sd.Plan(dev(rowptr), colind, values, M, K, N, dtype=dtype, family=sd.SD_MERGE)
    renamed = 0 if N == 4 and dtype == W.SD_F32 else 4
    rows_told = 0.625 if N == 1 and not empty else 4
    assert (rows_told + renamed) * cols.size < plan.info().plan_bytes < (rows_told + renamed + 1) * cols.size
    for kw in (dict(), dict(pad_b=3, pad_c=1), dict(offset=1)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    assert np.array_equal(got, run_spmm(plan, w, **kw)[0])
    got, _ = run_spmm(plan, w, c_fill=np.full((M, N), np.nan, np.float32), beta=0.0)
    check(w, got, beta=0.0)
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("lengths", [[1], [1, 2, 3], [7, 8, 9, 1, 1], [2, 300, 1, 5]])
@pytest.mark.parametrize("empty", [False, True])
def test_one_column_updates_c(empty, lengths, dtype):
    """beta != 0 at one column: a lane has up to seven complete rows, whose old values it reads together, and the end of one that began
    before; C with a pitch."""
    rows = np.resize(lengths, 3001)
    if empty:
        rows[2::5] = 0
    w = W.random_csr(3001, 700, 1, rows, seed=len(lengths), dtype=dtype, alpha=-0.5, beta=0.75)
    plan = DeviceWorkload(w).plan(family=sd.SD_MERGE)
    for kw in (dict(), dict(pad_c=2), dict(pad_b=1, offset=1)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    assert np.array_equal(got, run_spmm(plan, w, **kw)[0])
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("M,length,empty", [(39, 300_000, False), (650_000, 18, True), (1, 11_000_000, False)])
def test_one_column_of_many_steps(M, length, empty, dtype):
    """More than eight steps of 256 nonzeros for each of 32 warps per SM (9.7 M nonzeros) without frequent columns: gathers of 32 consecutive
    nonzeros, dealt out through shared memory; columns and values from an odd offset; a last step that is not whole."""
    lengths = np.full(M, length)
    if empty:
        lengths[::9] = 0
    K = 1_500_000
    rng = np.random.default_rng(M)
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    colind = rng.integers(0, K, rowptr[-1]).astype(np.int32)   # repeated and in any order
    vals, B = rng.standard_normal(colind.size).astype(np.float32), rng.standard_normal((K, 1)).astype(np.float32)
    C = rng.standard_normal((M, 1)).astype(np.float32)
    if dtype == W.SD_BF16:
        vals, B = W.f32_to_bf16_bits(vals), W.f32_to_bf16_bits(B).reshape(K, 1)
    w = W.Workload("many_steps", M, K, 1, rowptr, colind, vals, B, C, 1.5, -0.5, dtype, {})
    colind, vals = (dev(np.concatenate([np.zeros(3, a.dtype), a]))[3:] for a in (colind, vals))
    plan = sd.Plan(dev(rowptr), colind, vals, M, K, 1, dtype=dtype, family=sd.SD_MERGE)
    assert plan.info().plan_bytes < 5 * colind.numel()   # no renamed columns
    got, intact = run_spmm(plan, w)
    assert intact
    check(w, got)
    assert np.array_equal(got, run_spmm(plan, w)[0])
    plan.close()
