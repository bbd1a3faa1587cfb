"""What this library is timed on: the work its users have it do, through `paper_2608_05033_b200`'s public calls.

A case is one product C = alpha*A*B + beta*C as a program makes it ("op"):

  product  the plan exists and is reused: one `Plan.spmm` with device operands (inference, forward and backward of an
           aggregation with a symmetric adjacency, every iteration of a solver)
  values   the pattern stays and the values are new: `Plan.update_values`, then the product (trained weights of a
           block-sparse layer, edge weights that change from step to step)
  pattern  the pattern is new too: `Plan(...)`, its summary, the product, `Plan.close` (a sampled subgraph per step)
  host     the dense operands live in pinned host memory: `Plan.spmm_host`

on one of five kinds of matrix ("kind"), the five synthetic workloads of the benchmark, drawn on the GPU:

  uniform  Poisson row lengths, distinct uniform columns
  stencil  5-point Laplacian of a square grid
  rmat     symmetrised R-MAT graph with self-loops, D^-1/2 (A + I) D^-1/2 values
  block    dense 16x16 blocks at random block positions, each entry kept with probability `fill`
  ranks    rank-size row lengths (exponent 1.2, capped), distinct uniform columns

Dense widths run from 1 (a matrix-vector product) to 256 and take any value in between: 41 is a class count, 8 to 256
are the layer widths of the graph-network benchmark.  Values and B are fp32, or bf16 with fp32 accumulation; C is fp32.
"""
import math

import numpy as np
import torch

import paper_2608_05033_b200 as sd

# quadrant probabilities of the R-MAT generator (the lower right one is what is left)
RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19
# the rank-size law of the skewed workload, per 4,194,304 rows: the r-th longest row has SCALE * r^-EXPONENT nonzeros
RANKS_ROWS, RANKS_SCALE, RANKS_EXPONENT, RANKS_CAP = 4_194_304, 2.4e7, 1.2, 200_000


def listed():
    return [
        # the smallest call there is: everything is launch latency
        dict(name="uniform_2k_n32", op="product", kind="uniform", M=2048, K=2048, mean=8, N=32, dtype="f32", beta=0.0),
        # one operator of an iterative method on a regular grid, several right-hand sides, C updated in place
        dict(name="stencil_1m_n64_beta", op="product", kind="stencil", n=1024, N=64, dtype="f32", beta=0.5),
        # aggregation of a graph network's hidden layer over a power-law graph
        dict(name="rmat20_n128", op="product", kind="rmat", scale=20, edges=16, N=128, dtype="f32", beta=0.0),
        # the same with half-width features
        dict(name="rmat19_n64_bf16", op="product", kind="rmat", scale=19, edges=16, N=64, dtype="bf16", beta=0.0),
        # its last layer: one column per class, rows of B that start at any multiple of four bytes
        dict(name="rmat17_n41", op="product", kind="rmat", scale=17, edges=16, N=41, dtype="f32", beta=0.0),
        # matrix-vector product over a graph (centrality, power iteration)
        dict(name="rmat20_n1", op="product", kind="rmat", scale=20, edges=16, N=1, dtype="f32", beta=0.0),
        # a block-sparse layer in both value types
        dict(name="block_64k_n256", op="product", kind="block", Mb=4096, Kb=4096, blocks=33554, fill=1.0, N=256, dtype="f32", beta=0.0),
        dict(name="block_64k_n256_bf16", op="product", kind="block", Mb=4096, Kb=4096, blocks=33554, fill=1.0, N=256, dtype="bf16", beta=0.0),
        # the most skewed rows: 91 % of them hold 1 to 4 nonzeros, the longest 200,000
        dict(name="ranks_4m_n32", op="product", kind="ranks", M=RANKS_ROWS, N=32, dtype="f32", beta=0.0),
        # a block-sparse layer in training: new weights before every product
        dict(name="block_32k_n128_bf16_values", op="values", kind="block", Mb=2048, Kb=2048, blocks=16384, fill=1.0, N=128, dtype="bf16", beta=0.0),
        # a new sampled graph: analysis, plan, one product
        dict(name="rmat16_n32_pattern", op="pattern", kind="rmat", scale=16, edges=16, N=32, dtype="f32", beta=0.0),
        # dense operands in host memory, there and back
        dict(name="rmat17_n128_host", op="host", kind="rmat", scale=17, edges=16, N=128, dtype="f32", beta=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A dense width in [lo, hi]: a usual one, a multiple of eight, or any."""
    how = rng.random()
    if how < 0.5:
        return rng.choice([n for n in (1, 2, 4, 8, 16, 32, 64, 128, 256) if lo <= n <= hi])
    n = _log_int(rng, lo, hi)
    return min(hi, max(8, 8 * round(n / 8))) if how < 0.75 else n


def draw(rng):
    op = rng.choice(["product"] * 9 + ["values", "pattern", "host"])
    kind = rng.choice(["uniform", "stencil", "rmat", "rmat", "block", "block", "ranks"])
    c = dict(op=op, kind=kind)
    big = op in ("product", "values")
    if kind == "uniform":
        c["M"] = _log_int(rng, 1000, 1_000_000 if big else 150_000)
        c["K"] = _log_int(rng, max(1000, c["M"] // 2), min(1_000_000, 2 * c["M"]))
        c["N"] = _width(rng, 1, 128)
        c["mean"] = _log_int(rng, 3, min(48, max(4, 1_500_000_000 // (c["M"] * c["N"]))))
    elif kind == "stencil":
        c["n"] = _log_int(rng, 64, 1024 if big else 400)
        c["N"] = _width(rng, 1, 64)
    elif kind == "rmat":
        c["scale"] = rng.randint(12, 20 if big else 17)
        c["edges"] = _log_int(rng, 4, 16)
        c["N"] = _width(rng, 1, 128 if c["scale"] > 18 else 256)
    elif kind == "block":
        c["Mb"] = _log_int(rng, 128, 4096 if big else 1024)
        c["Kb"] = _log_int(rng, max(128, c["Mb"] // 2), min(4096, 2 * c["Mb"]))
        c["blocks"] = _log_int(rng, 4 * c["Mb"], 12 * c["Mb"])
        c["fill"] = rng.choice([1.0, 1.0, 0.75, 0.5])
        c["N"] = _width(rng, 8, 256)
    else:
        c["M"] = _log_int(rng, 20_000, RANKS_ROWS if big else 200_000)
        c["N"] = _width(rng, 1, 32 if c["M"] > 1_000_000 else 128)
    c["dtype"] = rng.choice(["f32", "f32", "bf16"])
    c["beta"] = rng.choice([0.0, 0.0, 0.0, 0.5])
    return c


# ---- the matrices, as (rowptr, colind, vals, M, K) on the GPU -----------------------------------
def _csr(rows, cols, M):
    rowptr = torch.zeros(M + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(rows, minlength=M), 0, out=rowptr[1:])
    return rowptr.to(torch.int32), cols.to(torch.int32)


def _distinct_columns(gen, lengths, K):
    """Keys row * K + column, ascending: lengths[i] distinct uniform columns in row i (repeated ones are drawn again)."""
    rows = torch.repeat_interleave(torch.arange(lengths.numel(), device="cuda"), lengths)
    base = rows * K
    key = torch.sort(base + torch.randint(0, K, (rows.numel(),), device="cuda", generator=gen)).values
    while True:
        again = torch.nonzero(key[1:] == key[:-1]).flatten()
        if again.numel() == 0:
            return rows, key - base
        key[again] = base[again] + torch.randint(0, K, (again.numel(),), device="cuda", generator=gen)
        key = torch.sort(key).values


def _ranks_lengths(M):
    """Row lengths by rank; the law's scale and cap follow the row count, so that any M has the same shape."""
    rank = np.arange(1, M + 1, dtype=np.float64)
    share = M / RANKS_ROWS
    top = max(1, min(int(RANKS_CAP * share), M // 4))
    return np.clip(np.floor(RANKS_SCALE * share ** RANKS_EXPONENT * rank ** -RANKS_EXPONENT), 1, top).astype(np.int64)


def _matrix(c, gen):
    kind = c["kind"]
    if kind == "uniform":
        M, K = c["M"], c["K"]
        lengths = torch.poisson(torch.full((M,), float(c["mean"]), device="cuda"), generator=gen).long().clamp_(0, K // 2)
        rows, cols = _distinct_columns(gen, lengths, K)
        vals = torch.rand(cols.numel(), device="cuda", generator=gen) * 2 - 1
    elif kind == "ranks":
        M = K = c["M"]
        lengths = torch.from_numpy(_ranks_lengths(M)).cuda()[torch.randperm(M, device="cuda", generator=gen)]
        rows, cols = _distinct_columns(gen, lengths, K)
        vals = torch.rand(cols.numel(), device="cuda", generator=gen) * 2 - 1
    elif kind == "stencil":
        n = c["n"]
        M = K = n * n
        i = torch.arange(M, device="cuda")
        x, y = i % n, i // n
        there = torch.stack([y > 0, x > 0, x >= 0, x < n - 1, y < n - 1], 1)
        rows = i[:, None].expand(M, 5)[there]
        cols = torch.stack([i - n, i - 1, i, i + 1, i + n], 1)[there]
        vals = torch.tensor([-1.0, -1.0, 4.0, -1.0, -1.0], device="cuda").expand(M, 5)[there]
    elif kind == "rmat":
        M = K = n = 1 << c["scale"]
        ne = c["edges"] * n
        src = torch.zeros(ne, dtype=torch.int64, device="cuda")
        dst = torch.zeros_like(src)
        for _ in range(c["scale"]):
            u = torch.rand(ne, device="cuda", generator=gen)
            low = u >= RMAT_A + RMAT_B
            right = ((u >= RMAT_A) & ~low) | (u >= RMAT_A + RMAT_B + RMAT_C)
            src = 2 * src + low
            dst = 2 * dst + right
        keep = src != dst
        src, dst = src[keep], dst[keep]
        i = torch.arange(n, device="cuda")
        key = torch.unique(torch.cat([src * n + dst, dst * n + src, i * n + i]))
        rows, cols = key // n, key % n
        scale = torch.bincount(rows, minlength=n).double().rsqrt()
        vals = (scale[rows] * scale[cols]).float()
    else:
        Mb, Kb = c["Mb"], c["Kb"]
        M, K = 16 * Mb, 16 * Kb
        at = torch.randperm(Mb * Kb, device="cuda", generator=gen)[: c["blocks"]]
        r, q = torch.arange(16, device="cuda")[:, None], torch.arange(16, device="cuda")[None, :]
        rows = (at // Kb * 16)[:, None, None] + r
        key = (rows * K + (at % Kb * 16)[:, None, None] + q).reshape(-1)
        if c["fill"] < 1.0:
            key = key[torch.rand(key.numel(), device="cuda", generator=gen) < c["fill"]]
        key = torch.sort(key).values
        rows, cols = key // K, key % K
        vals = torch.randn(key.numel(), device="cuda", generator=gen)
    rowptr, colind = _csr(rows, cols, M)
    return rowptr, colind, vals, M, K


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rowptr, colind, vals, M, K = _matrix(case, gen)
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    N, op = case["N"], case["op"]
    s = dict(op=op, beta=case["beta"], M=M, K=K, N=N, rowptr=rowptr, colind=colind, vals=vals.to(dtype).contiguous())
    B = torch.randn(K, N, device="cuda", generator=gen).to(dtype)
    # beta = 0.5 updates C in place: repeated passes on one state converge
    C = torch.randn(M, N, device="cuda", generator=gen)
    if op == "host":
        s["B"], s["C"] = B.cpu().pin_memory(), C.cpu().pin_memory()
    else:
        s["B"], s["C"] = B, C
    if op != "pattern":
        s["plan"] = sd.Plan(rowptr, colind, s["vals"], M, K, N)
    if op == "values":
        s["new_vals"] = (torch.randn(s["vals"].numel(), device="cuda", generator=gen) * vals.abs()).to(dtype)
    return s


def _summary(info):
    """The structure summary: every count of it, as one array of whole numbers."""
    one = [info.M, info.K, info.N, info.nnz, info.sum_r2, info.max_r, info.empty_rows, info.sum_span, info.max_span,
           info.sum_gap, info.diag, info.unsorted_rows, info.long_rows, info.nnz_long_rows, info.nnzb16,
           info.nnz_dense_blocks]
    return np.array(one + list(info.row_hist) + list(info.blk_hist), dtype=np.int64)


def run(s):
    op = s["op"]
    if op == "host":
        return s["plan"].spmm_host(s["B"], s["C"], 1.0, s["beta"])
    if op == "pattern":
        plan = sd.Plan(s["rowptr"], s["colind"], s["vals"], s["M"], s["K"], s["N"])
        C = plan.spmm(s["B"], s["C"], 1.0, s["beta"])
        summary = _summary(plan.info())
        plan.close()
        return {"C": C, "summary": summary}
    if op == "values":
        s["plan"].update_values(s["new_vals"])
    return s["plan"].spmm(s["B"], s["C"], 1.0, s["beta"])


# ---- what a pass cannot do without --------------------------------------------------------------
def _rmat_nnz(scale, edges):
    """Expected nonzeros of the symmetrised, deduplicated graph with self-loops: a cell that i levels put on the
    diagonal's upper left, j off the diagonal and the rest on its lower right has probability a^i b^j d^(scale-i-j)."""
    ne, d = edges << scale, 1.0 - RMAT_A - RMAT_B - RMAT_C
    cells = 0.0
    for i in range(scale + 1):
        for j in range(1, scale - i + 1):
            k = scale - i - j
            p = RMAT_A ** i * RMAT_B ** j * d ** k
            cells += math.comb(scale, i) * math.comb(scale - i, j) * 2.0 ** j * -math.expm1(-2.0 * p * ne)
    return (1 << scale) + int(cells)


def _sizes(c):
    kind = c["kind"]
    if kind == "uniform":
        return c["M"], c["K"], c["M"] * c["mean"]
    if kind == "stencil":
        return c["n"] ** 2, c["n"] ** 2, 5 * c["n"] ** 2 - 4 * c["n"]
    if kind == "rmat":
        return 1 << c["scale"], 1 << c["scale"], _rmat_nnz(c["scale"], c["edges"])
    if kind == "block":
        return 16 * c["Mb"], 16 * c["Kb"], int(256 * c["blocks"] * c["fill"])
    return c["M"], c["M"], int(_ranks_lengths(c["M"]).sum())


def work(case):
    """A's values, indices and row pointers read once, B read once, C written once and read once when beta != 0."""
    M, K, nnz = _sizes(case)
    N, es = case["N"], 2 if case["dtype"] == "bf16" else 4
    moved = nnz * (es + 4) + 4 * (M + 1) + K * N * es + 4 * M * N * (2 if case["beta"] else 1)
    return {"bytes": moved, "flops": 2 * nnz * N}


def tolerance(case):
    """Sums in fp32 for both value types (products of bf16 values are exact in fp32); the counts of a summary agree exactly."""
    return {"rel": 1e-5, "max": 4e-4}
