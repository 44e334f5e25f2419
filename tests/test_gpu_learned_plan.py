"""A plan for learned sizing does no work that only the symbolic pass reads (the
histogram of A's column lengths), and a symbolic pass run on it all the same finds
its hub columns."""
import ctypes

import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity

pytestmark = pytest.mark.gpu


def test_learned_plans_leave_the_hub_histogram_out():
    R = synth.rmat_symmetric(13, 16, seed=1)
    assert max(R.colptr[1:] - R.colptr[:-1]) >= 1024        # hub columns
    dR = g.to_device(R, ptr_dtype=torch.int32, idx_dtype=torch.int32)
    lib, launches, plans = g.load_library(), {}, {}
    for sizing in (g.SPG_SIZING_EXACT, g.SPG_SIZING_LEARNED):
        alloc = g._TorchAllocator(dR.colptr.device)
        opts = g.make_options(4, 256, sizing=sizing, allocator=alloc)
        c, h = dR.as_c(), ctypes.c_void_p()
        g._check(lib.spgemm_plan(ctypes.byref(c), ctypes.byref(c), ctypes.byref(opts), ctypes.byref(h)))
        plans[sizing] = g.Plan(h, dR, dR, opts, alloc)
        launches[sizing] = g.spgemm_plan_stats(plans[sizing])["kernel_launches"]
    assert launches[g.SPG_SIZING_LEARNED] == launches[g.SPG_SIZING_EXACT] - 1
    ref = oracle.spgemm(R, R)
    for plan in plans.values():
        assert_full_parity(g.spgemm_numeric(plan), ref, "with hubs")
        g.spgemm_plan_destroy(plan)
