"""Sums of long rows: a term of 1 first, then terms that a running sum of 1 rounds away.  A kernel that adds k of them in one
accumulator loses k half-units of the last place; the bound is what the longest chain of additions that the kernel
may have is allowed to lose, half a unit (2^-24 of the sum, all terms being positive) per addition."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    import paper_2608_05033_b200 as sd


def absorbing_rows(lengths, small, K, dtype):
    """Rows of lengths.numel() >= 1: the first value 1, the others `small`; columns repeat 0 .. K - 1."""
    rowptr = torch.zeros(lengths.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lengths, 0, out=rowptr[1:])
    nnz = int(rowptr[-1])
    vals = torch.full((nnz,), small, dtype=torch.float32 if dtype == W.SD_F32 else torch.bfloat16, device="cuda")
    vals[rowptr[:-1]] = 1.0
    colind = torch.arange(K, dtype=torch.int32, device="cuda").repeat(nnz // K + 1)[:nnz]
    return rowptr.to(torch.int32), colind, vals


# 16-byte loads per row of B (41: 41 columns, element by element), usual and longest row
@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("loads,usual,longest", [(2, 5, 500), (2, 20, 2000), (6, 24, 500), (6, 80, 2000), (8, 24, 1000), (16, 24, 500), (16, 36, 1000),
                                                 (16, 45, 2000), (32, 24, 500), (32, 45, 2000), (64, 10, 500), (64, 45, 2000), (41, 24, 500),
                                                 (41, 50, 2000)])
def test_row_group_chains(loads, usual, longest, dtype):
    """Rows of every lane set of the row-group kernel up to the longest it takes, 512 per set that the rule asks for: at most 64
    products in one accumulator, then a second one, the sum over at most four sets, and alpha."""
    N = 41 if loads == 41 else loads * (4 if dtype == W.SD_F32 else 8)
    lanes = min(32, 1 << (loads - 1).bit_length())
    M = 200_000 // lanes
    lengths = torch.full((M,), usual, dtype=torch.int64, device="cuda")
    lengths[::M // 5] = longest
    lengths[7::M // 5] = longest - 3
    rowptr, colind, vals = absorbing_rows(lengths, 2.0 ** -25, 300, dtype)
    scale = 2.0 ** (torch.arange(N, device="cuda") % 3)
    B = scale.expand(300, N).to(vals.dtype).contiguous()
    C = torch.full((M, N), float("nan"), device="cuda")
    plan = sd.Plan(rowptr, colind, vals, M, 300, N, family=sd.SD_ROWSPLIT)
    plan.spmm(B, C)
    exact = (1.0 + (lengths - 1).double() * 2.0 ** -25)[:, None] * scale.double()
    additions = 64 + torch.ceil(lengths / 64) + 4
    off = ((C.double() - exact).abs() / exact).amax(1)
    worst = (off / (additions * 2.0 ** -24)).max().item()
    plan.close()
    assert worst <= 1.0


@pytest.mark.parametrize("dtype", [W.SD_F32, W.SD_BF16])
@pytest.mark.parametrize("N,empty", [(1, False), (1, True), (3, False)])
def test_ranges_of_many_steps(N, empty, dtype):
    """One to four columns: a warp has 660 steps and more of 256 nonzeros (128 at three columns), rows are 700 steps long.  A lane adds
    eight, the scan over the lanes five, the open sum one per step of a range, at most 64; a row lies in up to 13 ranges, whose sums
    meet one by one in the end, and a dozen for the scans of the carries and scaling."""
    step = 256 if N <= 2 else 128
    length = 700 * step + 5
    lengths = torch.full((900_000_000 // length,), length, dtype=torch.int64, device="cuda")
    if step == 128:
        lengths = lengths[: lengths.numel() // 2]
    M = lengths.numel()
    rowptr, colind, vals = absorbing_rows(lengths, 2.0 ** -25 / step, 1000, dtype)
    if empty:
        rowptr, M = torch.cat([rowptr, rowptr[-1:]]), M + 1
    B = torch.ones(1000, N, dtype=vals.dtype, device="cuda")
    C = torch.full((M, N), float("nan"), device="cuda")
    plan = sd.Plan(rowptr, colind, vals, M, 1000, N, family=sd.SD_MERGE)
    plan.spmm(B, C)
    plan.close()
    exact = 1.0 + (length - 1) * 2.0 ** -25 / step
    additions = 8 + 5 + 64 + 13 + 12
    assert ((C[: lengths.numel()].double() - exact).abs() / exact).max().item() <= additions * 2.0 ** -24
    assert not empty or (C[-1] == 0).all()
