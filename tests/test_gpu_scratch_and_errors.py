"""Refused allocations and error returns: what a call leaves behind, and what it still computes."""
import ctypes
import threading
import time
from types import SimpleNamespace

import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2607_22866_b200 as gm
from paper_2607_22866_b200 import binding
from helpers import random_csr
from parity import compare_rows, make_opts

pytestmark = pytest.mark.gpu


@pytest.fixture
def allocator():
    """The torch allocator behind a predicate: allocator.refuse(bytes) -> True refuses the request.  allocator.held: what is
    handed out and not given back (results too)."""
    lib = binding.load_library()

    class Hook:
        refuse = staticmethod(lambda n: False)
        held = {}  # bytes by address

    def alloc(n, stream, user):
        p = None if Hook.refuse(n) else binding._torch_alloc(n, stream, user)
        if p:
            Hook.held[p] = n
        return p

    def free(p, stream, user):
        Hook.held.pop(p, None)
        binding._torch_free(p, stream, user)

    cbs = binding._ALLOC_FN(alloc), binding._FREE_FN(free)
    lib.gm_set_allocator(*cbs, None)
    yield Hook
    lib.gm_set_allocator(binding._alloc_cb, binding._free_cb, None)


def _after(n):
    """Refuses every request after the first n."""
    seen = []

    def refuse(_):
        seen.append(1)
        return len(seen) > n
    return refuse


@pytest.mark.parametrize("opts", [dict(), dict(stage_elems=1 << 20), dict(tau=256, chunk_width=1024, max_fanout=4), dict(single_stream=1)])
@pytest.mark.parametrize("granted", [0, 1, 2])  # C.row_ptr refused, C.col, C.val
def test_a_refused_c_leaves_nothing_running(allocator, opts, granted):
    # the plan's stream and the execute's differ, and the execute's is busy when the allocation is refused
    A = gen.rmat(12, 16, seed=4, dtype=np.float32)
    dA = gm.DeviceCSR.from_host(A)
    plan_stream, stream = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    plan = gm.spgemm_plan(dA, dA, opts=make_opts(**opts), stream=plan_stream)
    with torch.cuda.stream(stream):
        torch.cuda._sleep(20_000_000)
        allocator.refuse = staticmethod(_after(granted))
        with pytest.raises(gm.GmError) as ei:
            gm.spgemm_execute(plan)
        assert ei.value.status == -5
        assert stream.query() and plan_stream.query()
    plan.destroy()
    allocator.refuse = staticmethod(lambda n: False)
    C, _, _ = gm.spgemm(dA, dA)
    compare_rows(C, oracle.spgemm(A, A), np.float32)


def _light_matrix(dtype):
    """30011 rows of 144 products and some of none, one, a thousand: no heavy row with tau = 1024."""
    A = gen.erdos_renyi_k(30011, 12, seed=5, dtype=dtype)
    rows = np.split(A.col, A.row_ptr[1:-1])
    rng = np.random.default_rng(5)
    for i, k in ((0, 0), (7, 1), (8, 85), (30010, 84), (12345, 20), (12346, 0)):
        rows[i] = np.sort(rng.choice(A.n_rows, k, replace=False)).astype(np.int32)
    rp = np.zeros(A.n_rows + 1, np.int64)
    np.cumsum([len(r) for r in rows], out=rp[1:])
    return gen.CSR(A.n_rows, A.n_cols, rp, np.concatenate(rows).astype(np.int32), rng.uniform(-1, 1, rp[-1]).astype(dtype))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("how", ["more products than asked for", "area refused", "C refused beside it", "C refused beside it, from the host"])
def test_light_rows_without_room_for_their_products(allocator, how, dtype):
    A = _light_matrix(dtype)
    ref = oracle.spgemm(A, A)
    ip = oracle.row_products(A, A)
    area = int(ip.sum()) * (4 + np.dtype(dtype).itemsize)
    assert ip.max() <= 1024 and area > 1 << 25
    opts = make_opts(tau=1024, stage_elems=1 << 20 if how == "more products than asked for" else 0)
    dA = gm.DeviceCSR.from_host(A)
    if how == "area refused":
        allocator.refuse = staticmethod(lambda n: n > area)
    elif how.startswith("C refused"):
        allocator.refuse = staticmethod(lambda n: sum(allocator.held.values()) + n > 3 * area // 2 + (20 << 20))
    if how.endswith("host"):
        rp, col, val = np.empty(A.n_rows + 1, np.int64), np.empty(ref.nnz, np.int32), np.empty(ref.nnz, dtype)
        assert gm.spgemm_host(A, A, rp, col, val, opts=opts) == ref.nnz
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        return
    plan = gm.spgemm_plan(dA, dA, opts=opts)
    hashed = how != "C refused beside it"
    assert plan.info().light_bin_rows[7] == (plan.info().rows_light if hashed else 0)
    for _ in range(2):
        compare_rows(gm.spgemm_execute(plan), ref, dtype)
        info = plan.info()
        assert info.light_bin_rows[7] == info.rows_light == int((ip > 0).sum()) and info.workspace_bytes < area
        assert np.array_equal(plan.row_products().cpu().numpy(), ip)


def test_merged_rows_beside_a_long_one_without_room_for_their_products(allocator):
    A, _, _ = gen.config_inputs(1, shrink=2)  # 5-point stencil
    rows = np.split(A.col, A.row_ptr[1:-1])
    rows[77] = np.arange(0, A.n_cols, A.n_cols // 700, dtype=np.int32)
    rp = np.zeros(A.n_rows + 1, np.int64)
    np.cumsum([len(r) for r in rows], out=rp[1:])
    A = gen.CSR(A.n_rows, A.n_cols, rp, np.concatenate(rows), np.random.default_rng(1).uniform(-1, 1, rp[-1]))
    dA = gm.DeviceCSR.from_host(A)
    C, info, _ = gm.spgemm(dA, dA)
    assert info.rows_heavy > 0 and info.light_bin_rows[0] > 0
    allocator.refuse = staticmethod(lambda n: n > 12 * info.products_total * 3 // 4)
    D, info, _ = gm.spgemm(dA, dA)
    assert info.light_bin_rows[7] == info.rows_light
    ref = oracle.spgemm(A, A)
    compare_rows(C, ref, np.float64)
    compare_rows(D, ref, np.float64)


def test_no_room_for_the_lists_of_the_hash_accumulator(allocator):
    # C refused, and then what hashing the light rows takes: an error, and the plan can still be executed later
    A = _light_matrix(np.float32)
    ref = oracle.spgemm(A, A)
    dA = gm.DeviceCSR.from_host(A)
    plan = gm.spgemm_plan(dA, dA, opts=make_opts(tau=1024))
    for granted in (0, 0, 1, 2):  # C.row_ptr and the lists; the lists again; C.row_ptr; C.val
        allocator.refuse = staticmethod(_after(granted))
        with pytest.raises(gm.GmError) as ei:
            gm.spgemm_execute(plan)
        assert ei.value.status == -5
    allocator.refuse = staticmethod(lambda n: False)
    for _ in range(2):
        compare_rows(gm.spgemm_execute(plan), ref, np.float32)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["light", "heavy"])
@pytest.mark.parametrize("refused", [False, True])
def test_c_takes_little_more_than_its_entries(allocator, kind, dtype, refused):
    # many products per entry: C is allocated before its size is known, with room for every product, and does not keep it;
    # where that room is refused C is allocated when its size is known
    rng = np.random.default_rng(2)
    entry = 4 + np.dtype(dtype).itemsize
    k, hot = (18, 30) if kind == "light" else (25, 300)
    n = (60 << 20) // entry // (k * hot // 5)
    B = random_csr(rng, 500, hot, 0.2, dtype)
    B = gen.CSR(500, 100000, B.row_ptr, B.col * 33, B.val)
    rp = np.arange(n + 1, dtype=np.int64) * k
    col = np.concatenate([np.sort(rng.choice(500, k, replace=False)) for _ in range(n)]).astype(np.int32)
    A = gen.CSR(n, 500, rp, col, rng.uniform(-1, 1, col.size).astype(dtype))
    ip, ref = oracle.row_products(A, B), oracle.spgemm(A, B)
    room = int(ip.sum()) * entry  # (no row has more products than C has columns)
    assert 33 << 20 < room - ref.nnz * entry and room < 64 << 20
    if refused:
        allocator.refuse = staticmethod(lambda n: n == room // entry * 4)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
    C, info, stats = gm.spgemm(dA, dB)
    compare_rows(C, ref, dtype)
    held = C.col.untyped_storage().nbytes() + C.val.untyped_storage().nbytes()
    assert held == stats.c_capacity * entry <= (1 if refused else 2) * ref.nnz * entry + (0 if refused else 32 << 20)


def test_an_execute_does_not_wait_for_another_ones_stream():
    # one thread's stream is busy for half a second before its product: a product on another stream is done long before
    A = gen.rmat(12, 16, seed=4, dtype=np.float32)
    dA = gm.DeviceCSR.from_host(A)
    plans, streams = [gm.spgemm_plan(dA, dA) for _ in range(2)], [torch.cuda.Stream() for _ in range(2)]
    assert plans[0].info().rows_light > 0 and plans[0].info().rows_heavy > 0
    results = [gm.spgemm_execute(p, stream=s) for p, s in zip(plans, streams)]
    torch.cuda.synchronize()
    with torch.cuda.stream(streams[0]):
        torch.cuda._sleep(1_000_000_000)
    busy = threading.Thread(target=lambda: results.append(gm.spgemm_execute(plans[0], stream=streams[0])))
    busy.start()
    time.sleep(0.1)
    results.append(gm.spgemm_execute(plans[1], stream=streams[1]))
    assert not streams[0].query()
    busy.join()
    assert len(results) == 4
    ref = oracle.spgemm(A, A)
    for C in results:
        compare_rows(C, ref, np.float32)


@pytest.mark.parametrize("execute_on", ["default", "other", "none"])
def test_a_plan_outlives_its_stream(execute_on):
    # kernels that fill the plan's tables may still run when planning returns; the stream they run on is destroyed then
    A = gen.rmat(15, 16, seed=4, dtype=np.float32)
    dA = gm.DeviceCSR.from_host(A)
    gm.spgemm_plan(dA, dA).destroy()
    torch.cuda.synchronize()
    rt, handle = torch.cuda.cudart(), ctypes.c_void_p()
    assert int(rt.cudaStreamCreate(ctypes.addressof(handle))) == 0
    plan = gm.spgemm_plan(dA, dA, stream=SimpleNamespace(cuda_stream=handle.value))
    assert int(rt.cudaStreamDestroy(handle.value)) == 0
    if execute_on != "none":
        stream = torch.cuda.Stream() if execute_on == "other" else torch.cuda.current_stream()
        with torch.cuda.stream(stream):
            for _ in range(2):
                compare_rows(gm.spgemm_execute(plan), oracle.spgemm(A, A, 0, 500), np.float32)
    plan.destroy()
    C, _, _ = gm.spgemm(dA, dA)
    compare_rows(C, oracle.spgemm(A, A, 0, 500), np.float32)


@pytest.mark.parametrize("opts", [dict(), dict(level0_multisplit=2)])  # tasks, chunks
def test_budgets_of_shared_memory_in_several_threads(opts):
    # the kernels' limits of dynamic shared memory belong to the process: one thread's small budget must not cut another's
    # (which takes a launch right between the two, hence the many short calls)
    rng = np.random.default_rng(9)
    A, B = random_csr(rng, 64, 500, 0.5, np.float32), random_csr(rng, 500, 20000, 0.01, np.float32)
    dA, dB = gm.DeviceCSR.from_host(A), gm.DeviceCSR.from_host(B)
    ref, failed = oracle.spgemm(A, B), []

    def work(smem):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                plan = gm.spgemm_plan(dA, dB, smem, make_opts(**opts))
                for i in range(1000):
                    C = gm.spgemm_execute(plan)
                    if i % 250 == 0:
                        compare_rows(C, ref, np.float32)
        except Exception as e:  # (a thread's exception does not reach the test)
            failed.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(smem,)) for smem in (232448, 101376, 232448, 65536)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
