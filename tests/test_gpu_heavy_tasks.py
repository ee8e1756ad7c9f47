"""Heavy rows summed without staged products, at the sizes where their kernels change hands: rounds of rows of B, granules
of columns, granules cut into sub-ranges.  Against the oracle, with its tolerance (tau * sum|a*b|)."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2607_22866_b200 as gm
from parity import check_product, compare_rows, make_opts, run_gpu

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


@pytest.mark.parametrize("mid", [0, 16])  # hand-over to the dense accumulator: default, and nearly everything
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_products_that_underflow_keep_their_entry(dtype, mid):
    # products of either sign that round to zero, or to a subnormal, alone in their column and next to others.  The bound:
    # each of at most four products is off by half the smallest subnormal, sums of subnormals are exact, and the oracle's
    # result is rounded once.
    rng = np.random.default_rng(11)
    n_cols, info = 20000, np.finfo(dtype)
    tiny = dtype(1e-30) if dtype == np.float32 else dtype(1e-200)  # (its square underflows)
    B = _csr([rng.choice(n_cols, 6000, replace=False) for _ in range(4)], n_cols, rng, dtype)
    B.val[:] = np.where(B.val < 0, -tiny, tiny)
    sub = info.smallest_subnormal / tiny * 8  # times tiny: a few subnormals
    A = gen.CSR(4, 4, np.array([0, 1, 2, 4, 8]), np.array([0, 1, 2, 3, 0, 1, 2, 3], np.int32),
                np.array([-tiny, tiny, tiny, -tiny, -sub, tiny, -tiny, sub], dtype))
    C, plan, _ = run_gpu(A, B, tau=16, mid_chunk_max=mid, small_chunk_max=mid, validate_inputs=1)
    ref = oracle.spgemm(A, B)
    assert plan.rows_heavy == 4
    assert np.array_equal(C.row_ptr.cpu().numpy(), ref.row_ptr) and np.array_equal(C.col.cpu().numpy(), ref.col)
    assert np.all(np.abs(C.val.cpu().numpy().astype(np.longdouble) - ref.val) <= 4 * info.smallest_subnormal)


@pytest.mark.parametrize("n_rows", [1, 2, 1023, 1024, 1025, 4095, 4096, 4097, 16383, 16384, 16385])
def test_small_products_counted_by_one_block(n_rows):
    # the one-block launches around the sums: one heavy row, and 16384 rows of A and one more (separate launches); heavy
    # rows first, last and between empty and light ones; a kept plan executed again gives the same structure
    rng = np.random.default_rng(n_rows)
    m, n_cols = 500, 40000
    B = _csr([_row(rng, n_cols, int(k), 2000) for k in rng.integers(20, 60, m)], n_cols, rng, np.float32)
    heavy = {0, n_rows - 1, n_rows // 2, n_rows // 3}
    rows = [rng.choice(m, 40 + i % 3 * 100, replace=False) if i in heavy else rng.choice(m, i % 3, replace=False) for i in range(n_rows)]
    A = _csr(rows, m, rng, np.float32)
    C, info, stats = check_product(A, B, tau=512)
    assert info.rows_heavy == len(heavy)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
    plan = gm.spgemm_plan(dA, dB, opts=make_opts(tau=512))
    for _ in range(2):
        D = gm.spgemm_execute(plan)
        assert D.row_ptr.equal(C.row_ptr) and D.col.equal(C.col)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("lengths", [(1,), (1, 2, 3), (31, 32, 33), (63, 64, 65), (1, 127, 128, 129), (1, 500)])
def test_pieces_shorter_and_longer_than_the_windows(dtype, lengths):
    # rows of B of the lengths at which a round of windows starts, ends or holds many of them: up to 128 pieces in one
    # round, a piece that starts at the first product of a window or of the next round, pieces longer than a round
    rng = np.random.default_rng(sum(lengths))
    m, n_cols = 1500, 30000
    B = _csr([_row(rng, n_cols, lengths[i % len(lengths)], 900) for i in range(m)], n_cols, rng, dtype)
    rows = [rng.choice(m, k, replace=False) for k in (64, 65, 127, 128, 129, 255, 256, 257, 384, 385, 700, 1499)] + [np.arange(m)]
    A = _csr(rows, m, rng, dtype)
    C, info, stats = check_product(A, B, tau=16)
    assert info.rows_heavy == len(rows)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("stage", [0, 1 << 20])  # one batch, several
def test_debug_mode_finds_products_outside_their_task(dtype, stage):
    # columns of B that change behind the plan's back: debug mode reports it before anything is summed, and with the columns
    # of the plan the same plan computes the product
    A = gen.rmat(12, 16, seed=8, dtype=dtype)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(A)
    plan = gm.spgemm_plan(dA, dB, opts=make_opts(tau=256, chunk_width=512, validate_inputs=1, stage_elems=stage))
    assert plan.info().heavy_tasks == 1 and (plan.info().n_batches > 1) == (stage > 0)
    col = dB.col.clone()
    for bad in (torch.full_like(col, 5), A.n_cols - 1 - col):
        dB.col.copy_(bad)
        with pytest.raises(gm.GmError) as ei:
            gm.spgemm_execute(plan)
        assert ei.value.status == -10
    dB.col.copy_(col)
    compare_rows(gm.spgemm_execute(plan), oracle.spgemm(A, A), dtype)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ctas", [0, 1, 2, 4, 8])
def test_accumulators_per_sm_as_asked(dtype, ctas):
    # few products to a hand-over, so that the dense accumulator takes most tasks; several batches
    A = gen.rmat(13, 16, seed=8, dtype=dtype)
    C, info, _ = check_product(A, A, tau=256, acc_ctas_per_sm=ctas, small_chunk_max=32, mid_chunk_max=64, stage_elems=1 << 22)
    assert info.heavy_tasks == 1 and info.task_ctas_per_sm == (ctas or 3)


@pytest.mark.parametrize("n_rows_b,tasks", [(1000, 1), (30_000_000, 0)])
def test_tables_per_row_of_b_stay_small(n_rows_b, tasks):
    # boundaries of eight granules for 30 M rows of B are more than a gigabyte, for products that take a megabyte: staged
    rng = np.random.default_rng(6)
    n_cols = 131072
    B = _csr([_row(rng, n_cols, 300, 5000) for _ in range(1000)], n_cols, rng, np.float32)
    A = _csr([rng.choice(1000, k, replace=False) for k in (3, 40, 200, 1000)], n_rows_b, rng, np.float32)
    rp = torch.full((n_rows_b + 1,), int(B.nnz), dtype=torch.int64, device="cuda")
    rp[:1001] = torch.from_numpy(B.row_ptr).cuda()
    dA = gm.DeviceCSR.from_host(A)
    dB = gm.DeviceCSR(n_rows_b, n_cols, rp, torch.from_numpy(B.col).cuda(), torch.from_numpy(B.val).cuda())
    C, info, _ = gm.spgemm(dA, dB)
    assert info.rows_heavy == 4 and info.heavy_tasks == tasks
    assert info.workspace_bytes < 3 << 29
    compare_rows(C, oracle.spgemm(gen.CSR(4, 1000, A.row_ptr, A.col, A.val), B), np.float32)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("mid", [0, 600, 2048, 4096])
def test_products_kept_between_the_passes(dtype, mid):
    # tasks around half of the products that a mid-size block holds (kept for the second pass), over several rounds of rows of B;
    # a large one after a small one finds its slots empty
    rng = np.random.default_rng(mid)
    n_cols, m = 30000, 4600
    B = _csr([rng.choice(n_cols, 8 if i < 4300 else 1, replace=False) for i in range(m)], n_cols, rng, dtype)
    sizes = [300, 301, 511, 512, 513, 1023, 1024, 1025, 1500, 2047, 2048, 2049, 3000, 4095, 4096, 4097] * 6
    rows = [np.concatenate([rng.choice(4300, n // 8, replace=False), 4300 + rng.choice(300, n % 8, replace=False)]) for n in sizes]
    A = _csr(rows, m, rng, dtype)
    C, info, stats = check_product(A, B, tau=256, mid_chunk_max=mid)
    assert info.heavy_tasks == 1 and stats.mid_chunk_products > 0


@pytest.mark.parametrize("opts", [dict(), dict(level0_multisplit=1), dict(level0_multisplit=1, chunk_width=32, max_fanout=4)])
def test_gather_goes_over_more_tiles_than_it_has_blocks(opts):
    # 160 products to an entry of C: 19531 tiles of products, 148 SMs of 128 blocks each; in one staging buffer and in two
    n, m = 1000, 400
    rng = np.random.default_rng(7)
    A = _csr([np.arange(m)] * n, m, rng, np.float32)
    B = _csr([np.arange(m)] * m, m, rng, np.float32)
    C, info, stats = run_gpu(A, B, **opts)
    assert info.rows_heavy == n and info.n_batches == 1 and info.products_heavy > 148 * 128 * 8192
    assert C.nnz == n * m and np.array_equal(C.col.cpu().numpy(), np.tile(np.arange(m), n))
    a, b = A.val.reshape(n, m).astype(np.float64), B.val.reshape(m, m).astype(np.float64)
    assert np.all(np.abs(C.val.cpu().numpy().reshape(n, m) - a @ b) <= 1e-5 * (np.abs(a) @ np.abs(b)))


@pytest.mark.parametrize("n_long", [1, 2, 147, 148, 149, 300])
def test_counting_long_rows_with_all_blocks(n_long):
    # rows of A above 1024 entries share the blocks that count them: one row has all of them, from 149 on a group of blocks has several
    rng = np.random.default_rng(n_long)
    m, n_cols = 6000, 30000
    B = _csr([_row(rng, n_cols, int(k), 3000) for k in rng.integers(4, 24, m)], n_cols, rng, np.float32)
    longest = [m, 1025, 2048, 2049, 1024] if n_long < 10 else [1025, 1300, 1026, 2049]
    A = _csr([rng.choice(m, longest[i % len(longest)], replace=False) for i in range(n_long)] + [rng.choice(m, 200, replace=False)] * 3, m, rng, np.float32)
    C, info, stats = check_product(A, B, tau=512, chunk_width=8192)
    assert info.heavy_tasks == 1 and info.rows_heavy == n_long + 3 and info.params.chunks_required > 1
