"""The BSR-16 kernel on the warp-level tensor-core instructions: one or two strips of B per warp, one to four warps per
block-row, ring slots that wrap, block-rows of zero to more than 32 blocks per warp, a last block-row and a last block column
that are not whole, a last strip that is not whole."""
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
@pytest.mark.parametrize("Mb,N", [(5, 8), (5, 40), (5, 136), (5, 1032), (700, 64), (700, 136), (700, 264), (700, 520), (2400, 264)])
def test_block_rows_strips_and_edges(Mb, N, dtype):
    rng = np.random.default_rng(Mb + N)
    M, K = 16 * Mb - 5, 16 * 150 - 9
    blocks = rng.choice([0, 1, 2, 3, 4, 9], Mb)
    blocks[:3] = [150, 0, 33]
    rows, cols = [], []
    for i in range(Mb):
        J = np.sort(rng.choice(150, blocks[i], replace=False))
        if blocks[i] and i % 2:
            J[-1] = 149                                   # the block that reaches past the last column
            J = np.unique(J)
        c = (J[:, None] * 16 + np.arange(16)).reshape(-1)
        for r in range(16 * i, min(16 * i + 16, M)):
            keep = c[(c < K) & (rng.random(c.size) < 0.8)]
            rows.append(np.full(keep.size, r)), cols.append(keep)
    rows, cols = np.concatenate(rows), np.concatenate(cols).astype(np.int32)
    rowptr = np.zeros(M + 1, np.int32)
    np.cumsum(np.bincount(rows, minlength=M), out=rowptr[1:])
    vals, B = rng.standard_normal(cols.size).astype(np.float32), rng.standard_normal((K, N)).astype(np.float32)
    C = rng.standard_normal((M, N)).astype(np.float32)
    if dtype == W.SD_BF16:
        vals, B = W.f32_to_bf16_bits(vals), W.f32_to_bf16_bits(B).reshape(K, N)
    w = W.Workload("block_rows", M, K, N, rowptr, cols, vals, B, C, -0.75, 0.5, dtype, {})
    plan = DeviceWorkload(w).plan(family=sd.SD_BSR_TC)
    for kw in (dict(), dict(pad_b=8, pad_c=4)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    again, _ = run_spmm(plan, w, **kw)
    assert np.array_equal(got, again)
    got, _ = run_spmm(plan, w, c_fill=np.full((M, N), np.nan, np.float32), beta=0.0)
    check(w, got, beta=0.0)
    plan.close()


@pytest.mark.parametrize("dtype,N", [(W.SD_F32, 8), (W.SD_F32, 20), (W.SD_F32, 48), (W.SD_BF16, 16), (W.SD_BF16, 40)])
def test_automatic_row_split_plan_of_blocks(dtype, N):
    """Below the width of the block family an automatic plan of a blocked matrix is a row-split plan and runs the row kernels,
    with aligned operands and with others, also after new values and when it is loaded."""
    w = W.g4_block(Mb=90, Kb=70, N=N, nblocks=500, dtype=dtype)
    dw = DeviceWorkload(w)
    plan = dw.plan()
    assert plan.info().family == sd.SD_ROWSPLIT
    for kw in (dict(), dict(pad_b=8, pad_c=4), dict(pad_b=1, pad_c=1), dict(offset=1)):
        got, intact = run_spmm(plan, w, **kw)
        assert intact
        check(w, got)
    want, _ = run_spmm(plan, w)
    loaded = sd.Plan.load(plan.save(), dw.rowptr, dw.colind, dw.vals)
    assert np.array_equal(run_spmm(loaded, w)[0], want)
    new = np.random.default_rng(N).standard_normal(w.nnz).astype(np.float32)
    w.vals = W.f32_to_bf16_bits(new) if dtype == W.SD_BF16 else new
    vals = torch.from_numpy(w.vals.view(np.int16) if dtype == W.SD_BF16 else w.vals).cuda()
    for p in (plan, loaded):
        p.update_values(vals)
        check(w, run_spmm(p, w)[0])
        p.close()


@pytest.mark.parametrize("poison", [np.inf, np.nan])
@pytest.mark.parametrize("dtype,N", [(W.SD_F32, 8), (W.SD_F32, 48), (W.SD_F32, 72), (W.SD_BF16, 16), (W.SD_BF16, 40)])
def test_automatic_row_split_plan_of_blocks_keeps_non_finite_rows_of_b_apart(dtype, N, poison):
    """Row k of B holds Inf or NaN: it reaches exactly the rows with an entry in column k, and an Inf stays one."""
    base = W.g4_block(Mb=40, Kb=30, N=N, nblocks=150, seed=3, dtype=W.SD_F32)
    rng = np.random.default_rng(N)
    keep = rng.random(base.nnz) < 0.75
    rows = np.repeat(np.arange(base.M), np.diff(base.rowptr))[keep]
    cols, vals = base.colind[keep], np.abs(base.vals[keep]) + np.float32(0.5)
    rowptr = np.zeros(base.M + 1, np.int32)
    np.cumsum(np.bincount(rows, minlength=base.M), out=rowptr[1:])
    bad = rng.choice(base.K, 6, replace=False)
    B = np.abs(base.B)
    clean = B.copy()
    B[bad], clean[bad] = poison, 0.0
    if dtype == W.SD_BF16:
        vals, B, clean = W.f32_to_bf16_bits(vals), W.f32_to_bf16_bits(B).reshape(B.shape), W.f32_to_bf16_bits(clean).reshape(B.shape)
    w = W.Workload("poisoned_blocks", base.M, base.K, N, rowptr, cols, vals, B, None, 1.0, 0.0, dtype, {})
    named = np.zeros(base.M, bool)
    named[rows[np.isin(cols, bad)]] = True
    assert named.any() and not named.all()
    plan = DeviceWorkload(w).plan()
    assert plan.info().family == sd.SD_ROWSPLIT
    got, intact = run_spmm(plan, w)
    assert intact
    assert np.all(np.isnan(got[named]) if np.isnan(poison) else np.isposinf(got[named]))
    ref = W.Workload("clean", base.M, base.K, N, rowptr, cols, vals, clean, None, 1.0, 0.0, dtype, {})
    got[named] = run_spmm(plan, ref)[0][named]   # the other rows against the oracle
    check(ref, got)
    plan.close()


@pytest.mark.parametrize("N", [32, 128, 256])
@pytest.mark.parametrize("per_row", [1, 9, 36, 140])
def test_fp32_error_does_not_grow_with_the_blocks_of_a_row(per_row, N):
    """Positive operands, so that nothing cancels and a bias of the sums shows.  Relative error (2-norm): the low parts that are
    dropped or cut, about 2^-22 of a product; at most two truncated additions of 2^-23 inside a block; one addition rounded to nearest
    per block, 2^-25 sqrt(blocks) together.  2.4e-7 + 1.2e-7 + 0.3e-7 sqrt(140 / 3), rounded up: 6e-7."""
    Mb, Kb = 60, 150
    rng = np.random.default_rng(per_row)
    cols = np.concatenate([np.tile(np.sort(rng.choice(Kb, per_row, replace=False))[:, None] * 16 + np.arange(16), (16, 1, 1)).reshape(-1) for _ in range(Mb)]).astype(np.int32)
    M, K = 16 * Mb, 16 * Kb
    rowptr = (np.arange(M + 1) * 16 * per_row).astype(np.int32)
    vals, B = rng.uniform(0.25, 1, cols.size).astype(np.float32), rng.uniform(0.25, 1, (K, N)).astype(np.float32)
    w = W.Workload("positive_blocks", M, K, N, rowptr, cols, vals, B, None, 1.0, 0.0, W.SD_F32, {})
    plan = DeviceWorkload(w).plan(family=sd.SD_BSR_TC)
    got, _ = run_spmm(plan, w)
    A = np.zeros((M, K))
    A[np.repeat(np.arange(M), 16 * per_row), cols] = vals
    want = A @ B.astype(np.float64)
    assert np.linalg.norm(got - want) <= 6e-7 * np.linalg.norm(want)
    plan.close()


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("holes", [0, 1])
def test_block_values_from_any_offset(dtype, holes):
    """Whole vectors of a block's row come as one load where they are aligned, entry by entry otherwise: arrays that start at
    every element of a 16-byte piece, whole blocks and blocks with a few absent entries, bit-exact."""
    import oracle
    w = W.g4_block(Mb=20, Kb=15, N=64, nblocks=90, dtype=dtype)
    rowptr, colind = w.rowptr, w.colind
    if holes:
        keep = np.random.default_rng(1).random(colind.size) > 0.02
        rowptr = np.concatenate([[0], np.cumsum(keep)])[rowptr].astype(np.int32)
        colind = colind[keep]
    vals = np.random.default_rng(2).standard_normal(colind.size).astype(np.float32)
    if dtype == W.SD_BF16:
        vals = W.f32_to_bf16_bits(vals)
    ref = oracle.bsr16(rowptr, colind, vals, w.M, w.K)[2].tobytes()
    rowptr_d, colind_d = torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda()
    old = torch.zeros(colind.size, device="cuda", dtype=torch.float32 if dtype == W.SD_F32 else torch.int16)
    plan = sd.Plan(rowptr_d, colind_d, old, w.M, w.K, w.N, dtype=dtype, family=sd.SD_BSR_TC)
    bits = vals.view(np.int16) if dtype == W.SD_BF16 else vals
    for off in range(8):
        new = torch.from_numpy(np.concatenate([np.zeros(off, bits.dtype), bits])).cuda()
        plan.update_values(new[off:])
        assert sd.sd_plan_get_bsr(plan.handle)[2].tobytes() == ref
        plan.update_values(old)
    plan.close()
