"""One column with a lane per eight nonzeros or, where the arrays are not aligned, per 32; two and three columns on a matrix whose nonzeros crowd into few columns: the kernel that keeps those columns' rows of B in
shared memory, with columns outside, empty rows, a row over many chunks."""
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
