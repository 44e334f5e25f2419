"""A symbolic pass that runs out of workspace leaves its plan as it was: called
again with room, it and the numeric pass give the whole product."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity

pytestmark = pytest.mark.gpu

CHUNK = 4 << 20      # small workspace buffers are carved from chunks of this size


class Allocator(g._TorchAllocator):
    """Counts the chunks asked for; refuses the one numbered `refuse` once."""
    refuse, last = None, None

    def __init__(self, device):
        super().__init__(device)
        self.chunks = 0
        Allocator.last = self

    def _alloc(self, nbytes, ctx, stream):
        if nbytes == CHUNK:
            self.chunks += 1
            if self.chunks == Allocator.refuse:
                Allocator.refuse = None
                return None
        return super()._alloc(nbytes, ctx, stream)


def inputs(k, n=30000, m=2000, used=3000):
    """A: m x k, its first `used` columns hold 3 rows; B: one entry per column."""
    rng = np.random.default_rng(5)
    rows = np.sort(np.stack([rng.choice(m, 3, replace=False) for _ in range(used)]), 1).ravel()
    A = synth._csc_from_sorted(m, k, np.repeat(np.arange(used), 3), rows, rng.uniform(-1, 1, rows.size))
    B = synth._csc_from_sorted(k, n, np.arange(n), rng.integers(0, used, n), rng.uniform(-1, 1, n))
    return A, B


def test_symbolic_again_after_it_ran_out_of_workspace(monkeypatch):
    monkeypatch.setattr(g, "_TorchAllocator", Allocator)

    def chunks(k):
        plan = g.spgemm_plan(*(g.to_device(M) for M in inputs(k)), 1, 1024)
        in_plan = Allocator.last.chunks
        g.spgemm_symbolic(plan)
        total = Allocator.last.chunks
        g.spgemm_plan_destroy(plan)
        return in_plan, total

    # the bitmaps over A's columns grow with k: the smallest k whose workspace no
    # longer fits one chunk asks for the second at the end of the symbolic pass
    lo, hi = 30_000, 4_000_000
    assert chunks(lo) == (1, 1) and chunks(hi)[1] == 2
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if chunks(mid)[1] > 1 else (mid, hi)
    assert chunks(hi) == (1, 2)
    A, B = inputs(hi)
    plan = g.spgemm_plan(g.to_device(A), g.to_device(B), 1, 1024)
    Allocator.refuse = 2
    with pytest.raises(g.SpgError) as e:
        g.spgemm_symbolic(plan)
    assert e.value.status == g.SPG_OUT_OF_MEMORY
    g.spgemm_symbolic(plan)
    C = g.spgemm_numeric(plan)
    torch.cuda.synchronize()
    g.spgemm_plan_destroy(plan)
    assert_full_parity(C, oracle.spgemm(A, B), "after a second symbolic pass")
