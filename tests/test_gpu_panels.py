"""Neighbouring heavy rows with much the same columns, summed together: sizes of panels, of their column sets and of the
groups of columns they reach, against the oracle with its tolerance (tau * sum|a*b|)."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2607_22866_b200 as gm
from parity import check_product, compare_rows, make_opts, run_gpu
from test_gpu_scratch_and_errors import allocator  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def _csr(row_lists, n_cols, rng, dtype):
    rp = np.zeros(len(row_lists) + 1, np.int64)
    np.cumsum([len(r) for r in row_lists], out=rp[1:])
    col = np.concatenate([np.sort(np.asarray(r, np.int32)) for r in row_lists] + [np.zeros(0, np.int32)]).astype(np.int32)
    return gen.CSR(len(row_lists), n_cols, rp, col, rng.uniform(-1, 1, col.size).astype(dtype))


def _blocks(rng, sizes, per_row, fill, n_cols, dtype):
    """Consecutive row blocks of the given sizes; the rows of one draw their columns from the same per_row columns."""
    rows = []
    for n in sizes:
        pool = rng.choice(n_cols, per_row, replace=False)
        rows += [pool[rng.random(per_row) < fill] for _ in range(n)]
    return _csr(rows, n_cols, rng, dtype)


def _spans(rng, n_rows, n_cols, n_spans, width, fill, dtype):
    """Rows made of a few runs of neighbouring columns, which begin at one of some twenty places."""
    rows = []
    places = np.append(rng.integers(0, max(1, n_cols - width), 20), max(0, n_cols - width))
    for _ in range(n_rows):
        at = rng.choice(places, n_spans)
        c = np.unique(np.concatenate([a + np.nonzero(rng.random(width) < fill)[0] for a in at]))
        rows.append(c[c < n_cols])
    return _csr(rows, n_cols, rng, dtype)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_mid,n_cols", [(300, 130), (700, 4001), (3000, 70001)])
def test_panels_of_every_size(dtype, n_mid, n_cols):
    # row blocks below and above what a panel holds, next to rows of their own; column sets that end in the middle of a round
    rng = np.random.default_rng(n_cols)
    sizes = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 40, 63, 64, 65, 1, 100] * 18
    A = _blocks(rng, sizes, 113, 0.8, n_mid, dtype)
    B = _spans(rng, n_mid, n_cols, 2, 90, 0.7, dtype)
    C, info, stats = check_product(A, B, tau=64)
    assert info.heavy_tasks == 1 and stats.panel_rows > 0.7 * info.rows_heavy
    # several batches: panels end where a batch does
    big = int(info.products_max_row) * 191 + 5
    C2, info2, stats2 = check_product(A, B, tau=64, stage_elems=big)
    assert info2.n_batches > 3 and stats2.panel_rows > 0


@pytest.mark.parametrize("dtype,most", [(np.float32, 704), (np.float64, 384)])
@pytest.mark.parametrize("more", [None, 0, 1])
@pytest.mark.parametrize("rows", [5000, 27000])
def test_column_sets_at_their_limits(dtype, most, more, rows):
    # as many columns as a panel may have and one more (then the rows are tasks); units of a few groups and of whole panels
    rng = np.random.default_rng(most)
    n = 60 if more is None else most + more
    A = _blocks(rng, [32] * (rows // 32) + [rows % 32], n, 1.0, n, dtype)
    B = _spans(rng, n, 900, 2, 40, 0.6, dtype) if rows > 10000 else _spans(rng, n, 4000, 3, 100, 0.9, dtype)
    C, info, stats = check_product(A, B, tau=300)
    # (the last rows of all can be too few for the groups they reach)
    assert stats.panel_rows == 0 if more == 1 else stats.panel_rows > rows - 32


def test_rows_of_b_without_entries_and_scattered_ones():
    # U holds rows of B that are empty, short and long; scattered rows of B leave the panel to the tasks
    rng = np.random.default_rng(5)
    A = _blocks(rng, [32] * 120, 120, 0.9, 400, np.float32)
    B = _spans(rng, 400, 5000, 3, 100, 0.9, np.float32)
    rp, keep = B.row_ptr, rng.random(400) < 0.7
    B = _csr([B.col[rp[i]:rp[i + 1]] if keep[i] else [] for i in range(400)], 5000, rng, np.float32)
    C, info, stats = check_product(A, B, tau=100)
    assert stats.panel_rows == info.rows_heavy
    D = _csr([rng.choice(60000, 190, replace=False) for _ in range(400)], 60000, rng, np.float32)
    C, info, stats = check_product(A, D, tau=100)
    assert stats.panel_rows == 0 and info.heavy_tasks == 1


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_infinities_nans_and_zeros_stay_where_they_are(dtype):
    # an infinity or a NaN must not reach entries that no stored product of it belongs to; zeros of either sign are entries
    rng = np.random.default_rng(9)
    A = _blocks(rng, [32] * 180, 100, 0.85, 200, dtype)
    B = _spans(rng, 200, 700, 2, 120, 0.8, dtype)
    for M, n in ((A, 800), (B, 25)):
        at = rng.choice(M.val.size, n, replace=False)
        M.val[at] = rng.choice([np.inf, -np.inf, np.nan, 0.0, -0.0], n)
    C, info, stats = run_gpu(A, B, tau=64)
    assert stats.panel_rows == info.rows_heavy == A.n_rows
    a, b = np.zeros((A.n_rows, 200)), np.zeros((200, 700))
    has_a, has_b = np.zeros(a.shape, bool), np.zeros(b.shape, bool)
    for M, d, h in ((A, a, has_a), (B, b, has_b)):
        r = np.repeat(np.arange(M.n_rows), np.diff(M.row_ptr))
        d[r, M.col], h[r, M.col] = M.val, True
    want, bound = np.zeros((A.n_rows, 700)), np.zeros((A.n_rows, 700))
    with np.errstate(invalid="ignore"):
        for i in range(A.n_rows):
            k = np.nonzero(has_a[i])[0]
            p = np.where(has_b[k], a[i, k, None] * b[k], 0.0)
            want[i], bound[i] = p.sum(0), np.abs(p).sum(0)
    has = (has_a.astype(np.float32) @ has_b.astype(np.float32)) > 0
    rp, col, val = C.row_ptr.cpu().numpy(), C.col.cpu().numpy(), C.val.cpu().numpy()
    r = np.repeat(np.arange(A.n_rows), np.diff(rp))
    assert np.array_equal(np.flatnonzero(has), r * 700 + col)
    w, t = want[r, col], bound[r, col]
    fin = np.isfinite(w)
    assert fin.any() and not fin.all()
    assert np.array_equal(np.isnan(val), np.isnan(w)) and np.array_equal(val[~fin & ~np.isnan(w)], w[~fin & ~np.isnan(w)].astype(dtype))
    tol = 1e-5 if dtype == np.float32 else 1e-12
    assert np.all(np.abs(val[fin] - w[fin]) <= tol * t[fin])
    assert not np.any(np.signbit(val[val == 0]))


def test_a_kept_plan_with_new_values():
    rng = np.random.default_rng(2)
    A = _blocks(rng, [20] * 600, 90, 0.8, 500, np.float32)
    B = _spans(rng, 500, 2000, 2, 60, 0.8, np.float32)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
    plan = gm.spgemm_plan(dA, dB)
    first = gm.spgemm_execute(plan)
    v0 = first.val.clone()
    dA.val.mul_(2.0)
    second = gm.spgemm_execute(plan)
    assert plan.stats().panel_rows == A.n_rows
    assert torch.equal(first.col, second.col) and torch.equal(second.val, v0 * 2)


def test_no_room_for_the_panels_lists(allocator):
    # their memory is refused: the rows are tasks like the others
    rng = np.random.default_rng(3)
    A = _blocks(rng, [30] * 400, 90, 0.8, 500, np.float32)
    B = _spans(rng, 500, 2000, 2, 70, 0.8, np.float32)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
    ref = oracle.spgemm(A, B)
    for refused in (False, True):
        if refused:
            allocator.refuse = staticmethod(lambda n: 30 * A.nnz < n < 70 * A.nnz)
        plan = gm.spgemm_plan(dA, dB)
        allocator.refuse = staticmethod(lambda n: False)
        compare_rows(gm.spgemm_execute(plan), ref, np.float32)
        assert plan.stats().panel_rows == 0 if refused else plan.stats().panel_rows > 0.9 * A.n_rows


def _held(allocator, plan, *results):
    """What the plan has from the allocator: all but the results."""
    mine = {t.data_ptr() for C in results for t in (C.row_ptr, C.col, C.val)}
    return sum(n for p, n in allocator.held.items() if p not in mine)


@pytest.mark.parametrize("n_rows", [8000, 20000])  # tasks listed by one block, and by many
def test_rows_that_are_not_alike_take_no_lists(allocator, n_rows):
    # the same rows in another order, no two neighbours alike: planned as if there were no panels
    rng = np.random.default_rng(n_rows)
    A = _blocks(rng, [20] * (n_rows // 20), 150, 0.8, 4000, np.float32)
    B = _spans(rng, 4000, 3000, 2, 50, 0.9, np.float32)
    rows = np.split(A.col, A.row_ptr[1:-1])
    shuffled = _csr([rows[i] for i in rng.permutation(n_rows)], 4000, rng, np.float32)
    dB, held = gm.DeviceCSR.from_host(B), []
    for M in (A, shuffled):
        allocator.held.clear()
        plan = gm.spgemm_plan(gm.DeviceCSR.from_host(M), dB)
        torch.cuda.synchronize()
        assert plan.info().products_heavy >= 1 << 26
        held.append(_held(allocator, plan))
        C = gm.spgemm_execute(plan)
        assert plan.stats().panel_rows > 0.9 * n_rows if M is A else plan.stats().panel_rows == 0
        if M is shuffled:
            compare_rows(C, oracle.spgemm(M, B), np.float32)
    assert held[1] < held[0] - 40 * A.nnz


@pytest.mark.parametrize("n_rows", [8000, 20000])
def test_lists_of_no_panel_are_given_back(allocator, n_rows):
    # rows alike, but with more columns than a panel may have: nothing of the lists is left after the first product
    rng = np.random.default_rng(n_rows)
    A = _blocks(rng, [32] * (n_rows // 32), 705, 1.0, 705, np.float32)
    B = _spans(rng, 705, 3000, 1, 30, 0.6, np.float32)
    plan = gm.spgemm_plan(gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B))
    C = gm.spgemm_execute(plan)
    before = plan.info().workspace_bytes
    assert plan.stats().panel_rows == 0 and plan.info().products_heavy >= 1 << 26
    stage = plan.info().stage_elems * 8
    assert _held(allocator, plan, C) == before < stage + 30 * A.nnz + (8 << 20)
    compare_rows(gm.spgemm_execute(plan), oracle.spgemm(A, B), np.float32)


@pytest.mark.parametrize("batches", [False, True])
@pytest.mark.parametrize("n_rows", [8000, 20000])
def test_c_is_refused_beside_the_lists(allocator, n_rows, batches):
    # there is room for C or for the panels' lists: the lists go, and the rows are tasks from then on; not even that much room: an error,
    # and the plan goes on when there is room again
    rng = np.random.default_rng(n_rows)
    A = _blocks(rng, [20] * (n_rows // 20), 150, 0.8, 4000, np.float32)
    B = _spans(rng, 4000, 3000, 2, 50, 0.9, np.float32)
    ref = oracle.spgemm(A, B)
    c_bytes = ref.nnz * 8 + (n_rows + 1) * 8
    opts = make_opts(stage_elems=1 << 25, c_capacity=ref.nnz) if batches else None
    plan = gm.spgemm_plan(gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B), opts=opts)
    torch.cuda.synchronize()
    assert (plan.info().n_batches > 1) == batches

    def check():
        C = gm.spgemm_execute(plan)
        compare_rows(C, ref, np.float32)
        for t in (C.row_ptr, C.col, C.val):
            allocator.held.pop(t.data_ptr())

    check()
    assert plan.stats().panel_rows > 0.9 * n_rows
    for room in (c_bytes - 30 * A.nnz, 0, c_bytes, None):
        most = sum(allocator.held.values()) + room if room is not None else 1 << 40
        allocator.refuse = staticmethod(lambda n: sum(allocator.held.values()) + n > most)
        if room == 0:
            with pytest.raises(gm.GmError) as ei:
                gm.spgemm_execute(plan)
            assert ei.value.status == -5
        else:
            check()
            assert plan.stats().panel_rows == 0
    allocator.refuse = staticmethod(lambda n: False)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("what", ["A swapped", "A twice", "A ends inside", "B shuffled", "B twice"])
def test_rows_that_do_not_ascend_are_left_to_the_tasks(what, dtype):
    # against the contract, but the sums by tasks give the right product here (one granule of columns), and so they go on
    rng = np.random.default_rng(len(what))
    A = _blocks(rng, [25] * 480, 100, 0.85, 600, dtype)
    B = _spans(rng, 600, 900, 2, 60, 0.8, dtype)
    M, some = (A, [r for r in range(A.n_rows) if r // 25 % 3 == 0]) if what[0] == "A" else (B, range(0, 600, 7))
    col = M.col.copy()
    for r in some:
        s, e = M.row_ptr[r], M.row_ptr[r + 1]
        if what.endswith("shuffled"):
            col[s:e] = rng.permutation(col[s:e])
        elif what.endswith("swapped"):
            col[s + 40:s + 42] = col[s + 40:s + 42][::-1].copy()
        elif what.endswith("twice"):
            col[s + 5] = col[s + 4]
        else:  # the last column first: the row's ends leave out nearly all the others
            col[s:e] = np.roll(col[s:e], 1)
    a, b = np.zeros((A.n_rows, 600)), np.zeros((600, 900))
    X = gen.CSR(M.n_rows, M.n_cols, M.row_ptr, col, M.val)
    for S, d in ((X if M is A else A, a), (X if M is B else B, b)):
        np.add.at(d, (np.repeat(np.arange(S.n_rows), np.diff(S.row_ptr)), S.col), S.val.astype(np.float64))
    C, info, stats = run_gpu(X if M is A else A, X if M is B else B, tau=64)
    assert info.heavy_tasks == 1 and (stats.panel_rows == 0 if M is B else 0.6 * A.n_rows < stats.panel_rows <= A.n_rows)
    assert stats.panel_rows > 0.9 * A.n_rows if what == "A swapped" else stats.panel_rows < 0.7 * A.n_rows
    rp, cc, val = C.row_ptr.cpu().numpy(), C.col.cpu().numpy(), C.val.cpu().numpy()
    got = np.zeros((A.n_rows, 900))
    got[np.repeat(np.arange(A.n_rows), np.diff(rp)), cc] = val
    assert rp[-1] == np.count_nonzero((a != 0).astype(np.float32) @ (b != 0).astype(np.float32))
    tol = 1e-5 if dtype == np.float32 else 1e-12
    assert np.all(np.abs(got - a @ b) <= tol * (np.abs(a) @ np.abs(b)))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("stage", [0, 1 << 25])
def test_debug_mode_checks_the_products_of_panels(dtype, stage):
    # columns of B, and of A, that have changed since the plan; all of them in range, products per row as they were
    rng = np.random.default_rng(8)
    A = _blocks(rng, [31] * 500, 96, 0.85, 600, dtype)
    B = _spans(rng, 600, 900, 2, 60, 0.8, dtype)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
    plan = gm.spgemm_plan(dA, dB, opts=make_opts(tau=64, validate_inputs=1, stage_elems=stage))
    assert plan.info().heavy_tasks == 1 and (plan.info().n_batches > 1) == (stage > 0)
    ref = oracle.spgemm(A, B)
    for _ in range(2):
        compare_rows(gm.spgemm_execute(plan), ref, dtype)
        assert plan.stats().panel_rows > 0.9 * A.n_rows
    one = dB.col.clone()
    one[B.row_ptr[300]:B.row_ptr[301]] = one[B.row_ptr[300]:B.row_ptr[301]].flip(0)
    for col, bad in ((dB.col, torch.clamp(dB.col + 1, max=899)), (dB.col, one), (dA.col, 599 - dA.col)):
        good = col.clone()
        col.copy_(bad)
        with pytest.raises(gm.GmError) as ei:
            gm.spgemm_execute(plan)
        assert ei.value.status == -10
        col.copy_(good)
    compare_rows(gm.spgemm_execute(plan), ref, dtype)


def _scattered(rng, R, n_rows, per_row, fill, n_mid, n_cols, k, dtype):
    """Groups of R rows alike, times rows of k columns anywhere."""
    A = _blocks(rng, [R] * (n_rows // R), per_row, fill, n_mid, dtype)
    return A, _csr([rng.choice(n_cols, k, replace=False) for _ in range(n_mid)], n_cols, rng, dtype)


@pytest.mark.parametrize("dtype,R,k,n_cols,panels", [
    (np.float32, 2, 150, 200, False), (np.float32, 3, 100, 300, False), (np.float32, 4, 200, 400, False), (np.float32, 8, 150, 700, False),
    (np.float32, 8, 150, 400, True), (np.float32, 16, 150, 600, True), (np.float32, 32, 150, 1500, True),
    (np.float64, 4, 200, 300, False), (np.float64, 8, 100, 400, False), (np.float64, 8, 200, 400, True), (np.float64, 32, 200, 1500, True)])
def test_panels_where_they_are_the_faster_way(dtype, R, k, n_cols, panels):
    # few rows alike, or short pieces of rows of B: a panel takes longer than its rows one by one (up to twice the call)
    A, B = _scattered(np.random.default_rng(R * n_cols), R, 16000, 100, 0.9 if R < 8 else 0.8, 2000, n_cols, k, dtype)
    C, info, stats = run_gpu(A, B)
    assert info.heavy_tasks == 1 and info.products_heavy >= 1 << 26
    assert stats.panel_rows > 0.9 * A.n_rows if panels else stats.panel_rows == 0
    ref = oracle.spgemm(A, B)
    compare_rows(C, ref, dtype)


@pytest.mark.parametrize("n_rows,R", [(1024, 32), (1025, 41), (2000, 40)])  # all rows looked at, or one in 32
def test_few_heavy_rows_alike(n_rows, R):
    A, B = _scattered(np.random.default_rng(n_rows), R, n_rows, 300, 0.9, 1000, 400, 380, np.float32)
    C, info, stats = check_product(A, B)
    assert info.rows_heavy == n_rows and stats.panel_rows >= n_rows - 1  # (a run ends after 1024 rows)


@pytest.mark.parametrize("dtype,width", [(np.float32, 64), (np.float64, 32)])
@pytest.mark.parametrize("groups", [509, 510, 511, 512, 513])
def test_groups_that_a_panel_may_reach(dtype, width, groups):
    # every panel reaches all groups of columns: up to 511 (the last one's sums lie behind it), and more, which stays with the tasks
    rng = np.random.default_rng(groups)
    n_mid, n_cols = 200, groups * width
    at = [int(i * (groups - 4) / (n_mid - 1)) * width for i in range(n_mid)]
    B = _csr([a + np.nonzero(rng.random(4 * width) < 0.9)[0] for a in at], n_cols, rng, dtype)
    assert np.unique(B.col // width).size == groups
    A = _blocks(rng, [32] * 70, n_mid, 1.0, n_mid, dtype) if dtype == np.float32 else _blocks(rng, [32] * 110, n_mid, 1.0, n_mid, dtype)
    C, info, stats = check_product(A, B)
    assert info.heavy_tasks == 1 and stats.panel_rows == (A.n_rows if groups <= 511 else 0)
