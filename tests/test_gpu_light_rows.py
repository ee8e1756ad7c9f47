"""Row analysis and light rows at the sizes where their kernels change hands: tiles of entries and rows, widths of the
one-warp sort, the merge of few short rows.  Against the oracle, with its tolerance (tau * sum|a*b|)."""
import numpy as np
import pytest
import torch

import gen
import oracle
from helpers import random_csr
from parity import check_product, compare_rows
from test_gpu_scratch_and_errors import allocator  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def _csr(row_lists, n_cols, rng, dtype):
    rp = np.zeros(len(row_lists) + 1, np.int64)
    np.cumsum([len(r) for r in row_lists], out=rp[1:])
    col = np.concatenate([np.sort(np.asarray(r, np.int32)) for r in row_lists] + [np.zeros(0, np.int32)]).astype(np.int32)
    return gen.CSR(len(row_lists), n_cols, rp, col, rng.uniform(-1, 1, col.size).astype(dtype))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_cols", [700, 1 << 21, (1 << 23) + 5, (1 << 27) + 1])  # 32-bit and 64-bit sort keys
def test_sorted_rows_around_every_width(dtype, n_cols):
    # row r of B has 2**r entries from some 600 columns, so that columns repeat; rows of A spell their product counts in binary
    rng = np.random.default_rng(n_cols % 1000)
    pool = np.unique(np.concatenate([[0, n_cols - 1], rng.choice(n_cols, 600, replace=False) if n_cols < 1000 else rng.integers(0, n_cols, 600)]))
    B = _csr([rng.choice(pool, 1 << r, replace=False) for r in range(10)] + [[]], n_cols, rng, dtype)
    sizes = [0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 800, 1023]
    A = _csr([[r for r in range(10) if n >> r & 1] + [10] for n in sizes] * 3, 11, rng, dtype)
    C, info, stats = check_product(A, B, tau=700)  # sorted and heavy rows
    assert info.rows_heavy == 6
    check_product(A, B, tau=8)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_cols", [3000, (1 << 23) + 5])
def test_hashed_rows_around_every_class(dtype, n_cols):
    # rows above what one warp sorts, next to sorted and heavy ones; few and many entries for their products
    rng = np.random.default_rng(n_cols % 1000)
    pool = rng.choice(n_cols, 2500, replace=False)
    B = _csr([rng.choice(pool if r % 2 else pool[: (1 << r) + 3], 1 << r, replace=False) for r in range(12)] + [[]], n_cols, rng, dtype)
    sizes = [1, 700, 1023, 1024, 1025, 1100, 2047, 2048, 2049, 4000, 4095]
    A = _csr([[r for r in range(12) if n >> r & 1] for n in sizes] * 3, 13, rng, dtype)
    B2 = _csr([rng.choice(pool, 600, replace=False) for _ in range(14)], n_cols, rng, dtype)
    A2 = _csr([rng.choice(14, k, replace=False) for k in (1, 2, 6, 7, 13, 14)], 14, rng, dtype)
    for X, Y in ((A, B), (A2, B2)):
        ip = oracle.row_products(X, Y)
        for tau in (1500, 4095, 8192):
            C, info, stats = check_product(X, Y, tau=tau)
            assert info.light_bin_rows[7] == int(((ip > 1024) & (ip <= tau)).sum()) > 0


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("lists", [1, 2, 4, 5, 8])
def test_merged_rows(dtype, lists):
    # enough rows for one thread each; alone in the matrix (counted, then written to C) and next to longer rows (staged)
    rng = np.random.default_rng(lists)
    n, m = (1 << 16) + 77, 5000
    B = _csr([rng.choice(40 + 7 * i % 4000, int(rng.integers(0, 9)), replace=False) for i in range(3000)], m, rng, dtype)
    rows = [rng.choice(3000, int(k), replace=False) for k in rng.integers(0, lists + 1, n)]
    A = _csr(rows, 3000, rng, dtype)
    C, info, stats = check_product(A, B)
    assert info.rows_heavy == 0
    rows[5], rows[n - 1] = np.arange(40), np.arange(300)
    check_product(_csr(rows, 3000, rng, dtype), B, tau=400)


def test_rows_of_every_length_across_tiles():
    # a hub row over many tiles, runs of empty rows longer than a tile, rows that end exactly at a tile's edge
    import paper_2607_22866_b200 as gm
    rng = np.random.default_rng(4)
    B = random_csr(rng, 6000, 900, 0.01, np.float32)
    for lengths in ([6000, 0, 0, 5000, 1], [0] * 5000 + [1] + [0] * 5000, [511, 1, 0, 512, 1023, 0] * 40, [3] * 400 + [2045, 2048, 2047] * 90):
        A = _csr([rng.choice(6000, k, replace=False) for k in lengths], 6000, rng, np.float32)
        dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
        ref = oracle.row_products(A, B)
        plan = gm.spgemm_plan(dA, dB)
        assert np.array_equal(plan.row_products().cpu().numpy(), ref)
        info = plan.info()
        assert info.products_total == ref.sum() and info.rows_empty == int((ref == 0).sum()) and info.rows_heavy == int((ref > info.params.tau).sum())
        assert info.nnz_a_heavy == int(np.asarray(lengths)[ref > info.params.tau].sum())
        out = torch.full((A.n_rows,), -1, dtype=torch.int64, device="cuda")
        assert np.array_equal(gm.row_products_noalloc(dA, dB, out).cpu().numpy(), ref)
    check_product(A, B)


@pytest.mark.parametrize("n_cols", [1 << 24, (1 << 24) + 1])  # 32-bit prefix sums, and the first width with 64-bit ones
@pytest.mark.parametrize("n_rows", [40000, 80000])  # small and large tiles
def test_row_products_of_full_rows(n_rows, n_cols):
    # every entry of A meets a full row of B: a warp of a large tile adds up 256 of them, 2^32 products at 2^24 columns
    import paper_2607_22866_b200 as gm
    A = gm.DeviceCSR(n_rows, 1, torch.arange(n_rows + 1, device="cuda"), torch.zeros(n_rows, dtype=torch.int32, device="cuda"),
                     torch.ones(n_rows, device="cuda"))
    B = gm.DeviceCSR(1, n_cols, torch.tensor([0, n_cols], device="cuda"), torch.arange(n_cols, dtype=torch.int32, device="cuda"),
                     torch.ones(n_cols, device="cuda"))
    out = torch.full((n_rows,), -1, dtype=torch.int64, device="cuda")
    gm.row_products_noalloc(A, B, out)
    assert bool((out == n_cols).all())


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 255, 256, 257, 5000, (1 << 16) + 300, (1 << 20) + 1])
@pytest.mark.parametrize("longest", [4, 40])
def test_light_rows_find_their_place_by_themselves(n, longest, dtype):
    # no heavy rows: groups of 256 rows and one more, rows without entries at either end, a kept plan executed again, and one row
    # more than may do without a prefix sum
    import paper_2607_22866_b200 as gm
    rng = np.random.default_rng(n)
    m = 3000
    B = _csr([rng.choice(m, int(k), replace=False) for k in rng.integers(0, 6, m)], m, rng, dtype)
    k = rng.integers(0, longest, n)
    k[rng.random(n) < 0.3] = 0
    k[n // 2] = longest
    starts = rng.integers(0, m - longest, n)
    rp = np.zeros(n + 1, np.int64)
    np.cumsum(k, out=rp[1:])
    col = np.repeat(starts - rp[:-1], k) + np.arange(rp[-1])
    A = gen.CSR(n, m, rp, col.astype(np.int32), rng.uniform(-1, 1, rp[-1]).astype(dtype))
    ref = oracle.spgemm(A, B)
    plan = gm.spgemm_plan(gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B))
    assert plan.info().rows_heavy == 0
    for _ in range(3):
        compare_rows(gm.spgemm_execute(plan), ref, dtype)


@pytest.mark.parametrize("n_cols", [1 << 24, (1 << 24) + 1])  # 32-bit prefix sums, and the first width with 64-bit ones
def test_row_analysis_with_many_tiles_to_a_block(n_cols):
    # some ten tiles for every block, so that its warps look up the rows of four tiles at a time, thrice; hub rows over several tiles
    import paper_2607_22866_b200 as gm
    rng = np.random.default_rng(6)
    n, m = 9_000_000, 4000
    k = rng.integers(0, 3, n)
    k[[0, n // 3, n - 1]] = m
    k[n // 2:n // 2 + 50000] = 0
    rp = np.zeros(n + 1, np.int64)
    np.cumsum(k, out=rp[1:])
    col = (np.arange(rp[-1]) - np.repeat(rp[:-1], k) + np.repeat(np.where(k == m, 0, rng.integers(0, m - 3, n)), k)).astype(np.int32)
    length = rng.integers(0, 30, m)
    b_rp = np.zeros(m + 1, np.int64)
    np.cumsum(length, out=b_rp[1:])
    A = gm.DeviceCSR(n, m, torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), torch.ones(col.size, device="cuda"))
    B = gm.DeviceCSR(m, n_cols, torch.from_numpy(b_rp).cuda(), torch.from_numpy((np.arange(b_rp[-1]) - np.repeat(b_rp[:-1], length)).astype(np.int32)).cuda(),
                     torch.ones(int(b_rp[-1]), device="cuda"))
    before = np.zeros(col.size + 1, np.int64)
    np.cumsum(length[col], out=before[1:])
    ref = before[rp[1:]] - before[rp[:-1]]
    plan = gm.spgemm_plan(A, B)
    assert np.array_equal(plan.row_products().cpu().numpy(), ref)
    info = plan.info()
    assert info.products_total == ref.sum() and info.products_max_row == ref.max() and info.rows_empty == int((ref == 0).sum()) and info.rows_heavy == 3


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("rows", ["merged", "sorted"])
def test_c_takes_what_its_entries_take(rows, dtype):
    # no heavy rows, several products per entry of C, 64 to 512 MB for all of them: nothing is held for those, at no time
    import paper_2607_22866_b200 as gm
    if rows == "merged":
        A = gen.laplacian_2d(700, dtype=dtype)
    else:
        n, w = 40000, 19
        i = np.arange(n)[:, None] + np.arange(w) - w // 2
        A = _csr([r[(r >= 0) & (r < n)] for r in i], n, np.random.default_rng(1), dtype)
    dA = gm.DeviceCSR.from_host(A)
    ref = oracle.spgemm(A, A)
    plan = gm.spgemm_plan(dA, dA)
    entry = 4 + np.dtype(dtype).itemsize
    assert plan.info().rows_heavy == 0 and 64 << 20 < plan.info().c_nnz_upper * entry < 512 << 20
    for _ in range(2):
        torch.cuda.synchronize()
        torch.cuda.reset_peak_memory_stats()
        before = torch.cuda.memory_allocated()
        C = gm.spgemm_execute(plan)
        peak = torch.cuda.max_memory_allocated() - before
        compare_rows(C, ref, dtype)
        assert peak <= ref.nnz * entry + (A.n_rows + 1) * 8 + (4 << 20)
        del C


@pytest.mark.parametrize("n", [3000, (1 << 16) + 300])  # sorted rows; merged rows
def test_light_rows_after_a_refusal(allocator, n):
    # the room for every product is refused: C takes what it needs.  C is refused: the next execute starts from cleared sums.
    import paper_2607_22866_b200 as gm
    A = gen.erdos_renyi_k(n, 4, seed=n, dtype=np.float32)
    dA = gm.DeviceCSR.from_host(A)
    ref = oracle.spgemm(A, A)
    plan = gm.spgemm_plan(dA, dA)
    upper = plan.info().c_nnz_upper
    assert plan.info().rows_heavy == 0 and ref.nnz < upper
    for refuse, ok in ((lambda b: b >= upper * 4, True), (lambda b: b < n * 8 or b > (n + 1) * 8, False), (lambda b: False, True),
                       (lambda b: b >= upper * 4, True), (lambda b: False, True)):
        allocator.refuse = staticmethod(refuse)
        if ok:
            C = gm.spgemm_execute(plan)
            allocator.refuse = staticmethod(lambda b: False)
            compare_rows(C, ref, np.float32)
        else:
            with pytest.raises(gm.GmError) as ei:
                gm.spgemm_execute(plan)
            assert ei.value.status == -5


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_cols", [700, 1 << 21, (1 << 27) + 1])  # 32-bit and 64-bit sort keys
def test_sorted_rows_around_the_widths_between_powers_of_two(dtype, n_cols):
    # 3, 5 and 6 keys a lane: rows of up to 96, 160 and 192 products, and one more or less; columns repeat
    rng = np.random.default_rng(n_cols % 1000)
    pool = np.unique(np.concatenate([[0, n_cols - 1], rng.choice(n_cols, 600, replace=False) if n_cols < 1000 else rng.integers(0, n_cols, 600)]))
    sizes = [64, 65, 66, 94, 95, 96, 97, 98, 129, 145, 158, 159, 160, 161, 162, 190, 191, 192, 193, 194]
    B = _csr([rng.choice(pool, 1 << r, replace=False) for r in range(8)], n_cols, rng, dtype)
    A = _csr([[r for r in range(8) if n >> r & 1] for n in sizes] * 7, 8, rng, dtype)
    C, info, stats = check_product(A, B)  # rows placed by the sums of their groups
    assert info.rows_heavy == 0 and info.rows_light == A.n_rows
    rows = [[r for r in range(8) if n >> r & 1] for n in sizes] + [[8]]
    B2 = _csr([B.col[B.row_ptr[r]:B.row_ptr[r + 1]] for r in range(8)] + [pool], n_cols, rng, dtype)
    C, info, stats = check_product(_csr(rows, 9, rng, dtype), B2, tau=256)  # next to a heavy row
    assert info.rows_heavy == 1
