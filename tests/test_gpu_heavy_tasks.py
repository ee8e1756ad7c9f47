"""Heavy rows summed without staged products, at the sizes where their kernels change hands: rounds of rows of B, granules
of columns, granules cut into sub-ranges.  Against the oracle, with its tolerance (tau * sum|a*b|)."""
import numpy as np
import pytest

import gen
from parity import check_product

pytestmark = pytest.mark.gpu


def _csr(row_lists, n_cols, rng, dtype):
    rp = np.zeros(len(row_lists) + 1, np.int64)
    np.cumsum([len(r) for r in row_lists], out=rp[1:])
    col = np.concatenate([np.sort(np.asarray(r, np.int32)) for r in row_lists] + [np.zeros(0, np.int32)]).astype(np.int32)
    return gen.CSR(len(row_lists), n_cols, rp, col, rng.uniform(-1, 1, col.size).astype(dtype))


def _row(rng, n_cols, n, hot):
    """n distinct columns, most of them among the first `hot`."""
    a = rng.choice(hot, min(hot, (3 * n) // 4), replace=False)
    return np.unique(np.concatenate([a, rng.integers(0, n_cols, n - a.size)]))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_cols", [3000, 16384, 16385, 49157, 262144])
def test_rows_of_every_length_over_granules(dtype, n_cols):
    # rows of A around the rounds of 256 and 512 rows of B and of 1024 (counted by many warps); rows of B from 0 entries to
    # a third of the columns; hot columns, so that granules go over the size at which they are cut into sub-ranges
    rng = np.random.default_rng(n_cols)
    m = 2300
    sizes = rng.choice([0, 1, 2, 31, 32, 33, 63, 64, 65, 130, 300], m)
    sizes[[5, 900]] = n_cols // 3
    B = _csr([_row(rng, n_cols, int(k), 1500) if k else [] for k in sizes], n_cols, rng, dtype)
    rows = [rng.choice(m, k, replace=False) for k in (1, 2, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1537, 2300)]
    A = _csr(rows + [[5], [5, 900], []], m, rng, dtype)
    C, info, stats = check_product(A, B, tau=16)
    assert info.rows_heavy >= 18
    if n_cols == 16385:  # several batches
        check_product(A, B, tau=16, stage_elems=int(info.products_max_row) + 7)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_products_that_cancel_keep_their_entry(dtype):
    # every entry of C is a sum of +x and -x, or of zeros of either sign: the entry stays, with the value 0
    rng = np.random.default_rng(3)
    n_cols = 20000
    cols = np.sort(rng.choice(n_cols, 9000, replace=False)).astype(np.int32)
    v = rng.uniform(-1, 1, cols.size).astype(dtype)
    v[::7] = 0.0
    v[::14] = -0.0
    B = gen.CSR(2, n_cols, np.array([0, cols.size, 2 * cols.size]), np.concatenate([cols, cols]), np.concatenate([v, -v]).astype(dtype))
    A = gen.CSR(2, 2, np.array([0, 2, 3]), np.array([0, 1, 1], np.int32), np.array([2, 2, -1], dtype))
    C, info, stats = check_product(A, B, tau=16)
    assert C.nnz == 2 * cols.size and not C.val[:cols.size].any()
