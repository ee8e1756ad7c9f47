"""Refused allocations and error returns: what a call leaves behind, and what it still computes."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2607_22866_b200 as gm
from paper_2607_22866_b200 import binding
from parity import compare_rows, make_opts

pytestmark = pytest.mark.gpu


@pytest.fixture
def allocator():
    """The torch allocator behind a predicate: allocator.refuse(bytes) -> True refuses the request."""
    lib = binding.load_library()

    class Hook:
        refuse = staticmethod(lambda n: False)

    def alloc(n, stream, user):
        return None if Hook.refuse(n) else binding._torch_alloc(n, stream, user)

    cb = binding._ALLOC_FN(alloc)
    lib.gm_set_allocator(cb, binding._free_cb, None)
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
