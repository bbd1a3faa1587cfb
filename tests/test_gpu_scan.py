"""The structure scan at the edges of its tables: block-rows of as many nonzeros as a warp's, a small and a large CTA's table
takes, and one more or less; matrices as wide as the counter tables, the warp table's words and beyond; rows out of order,
repeated columns, empty rows, and column arrays that start at any entry of a 16-byte piece.  Every count agrees exactly."""
import numpy as np
import pytest

import oracle
pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if torch.cuda.is_available():
    import paper_2608_05033_b200 as sd
    from util import dev


def block_row(rng, n, K, order):
    """Row lengths and columns of 16 rows with n nonzeros together, some rows empty."""
    lengths = rng.multinomial(n, rng.dirichlet(np.full(16, 0.4)))
    cols = []
    for r in lengths:
        c = rng.choice(K, size=r, replace=False) if r <= K else rng.integers(0, K, r)
        if order == "dense":
            c = (int(rng.integers(0, K)) + np.arange(r)) % K
        if order == "repeated":
            c = rng.integers(0, min(K, 700), r)
        cols.append(c if order == "any" else np.sort(c))
    return lengths, np.concatenate(cols)


@pytest.mark.parametrize("order", ["ascending", "dense", "any", "repeated"])
@pytest.mark.parametrize("K", [16, 5000, 262144, 262160, 524288, 524304, 67108840, 67108865])
def test_counts_at_the_edges_of_the_tables(K, order):
    rng = np.random.default_rng(K % 1000 + len(order))
    sizes = [0, 1, 3, 4, 5, 127, 128, 129, 999, 1000, 1001, 4095, 4096, 4097, 8191, 8193, 20000]
    if order in ("ascending", "any"):   # distinct columns
        sizes = [n for n in sizes if n <= 2 * K]
    lengths, cols = zip(*(block_row(rng, n, K, order) for n in rng.permutation(np.resize(sizes, 160))))
    lengths = np.concatenate(lengths)[:-5]   # the last block-row is short
    M = lengths.size
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    colind = np.concatenate(cols)[:rowptr[-1]].astype(np.int32)
    ref = oracle.summary(rowptr, colind, M, K, 1).as_dict()
    for off in range(4):
        c = dev(np.concatenate([np.zeros(off, np.int32), colind, np.zeros(1, np.int32)]))
        vals = torch.zeros(colind.size + 1, device="cuda")
        plan = sd.Plan(dev(rowptr), c[off:], vals, M, K, 1, family=sd.SD_ROWSPLIT)
        mine = plan.info().as_dict()
        plan.close()
        assert {k: mine[k] for k in ref} == ref


@pytest.mark.parametrize("K", [67108832, 67108833, 2 ** 27 + 5])
@pytest.mark.parametrize("where", ["last", "any"])
def test_highest_block_columns_of_the_warp_tables(where, K):
    """The last matrix whose block columns share a word with a count (2^22 - 2 of them), the first that is wider and a much wider one:
    block-rows of half as many, as many and more nonzeros as a warp takes, in the last block columns or anywhere."""
    rng = np.random.default_rng(K % 1000)
    lengths, cols = [], []
    for n in rng.permutation(np.resize([1, 5, 499, 500, 501, 999, 1000, 1001, 4097], 200)):
        r = rng.multinomial(n, np.full(16, 1 / 16))
        lengths.append(r)
        for k in r:
            low = K - 5000 if where == "last" else 0
            cols.append(np.sort(low + rng.choice(K - low, size=k, replace=False) if K - low < 10000 else np.unique(rng.integers(low, K, 2 * k))[:k]))
            assert cols[-1].size == k
    lengths, colind = np.concatenate(lengths), np.concatenate(cols).astype(np.int32)
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    ref = oracle.summary(rowptr, colind, lengths.size, K, 1).as_dict()
    plan = sd.Plan(dev(rowptr), dev(colind), torch.zeros(colind.size, device="cuda"), lengths.size, K, 1, family=sd.SD_ROWSPLIT)
    mine = plan.info().as_dict()
    plan.close()
    assert {k: mine[k] for k in ref} == ref
