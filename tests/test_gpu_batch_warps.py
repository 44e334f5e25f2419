"""Batches whose instances fall into each table class (bounds up to 256, 512 and
1024 entries a column), at 4 and at 8 asked warps per CTA, against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import check_values

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", ["f64", "i64", "i32"])
@pytest.mark.parametrize("warps", [4, 8])
@pytest.mark.parametrize("degrees", [(8, 30), (16, 30), (30, 34), None])
def test_asked_warps_in_every_class(degrees, warps, values):
    pairs = []
    for i, (a, b) in enumerate([degrees] * 3 if degrees else [(8, 30), (16, 30), (30, 34)]):
        pairs.append((synth.uniform_columns(2500 + 37 * i, a, seed=i, values=values),
                      synth.uniform_columns(2500 + 37 * i, b, seed=10 + i, values=values)))
    batch = g.spgemm_batch_create(*([g.to_device(p[q]) for p in pairs] for q in (0, 1)), warps_per_cta=warps)
    g.spgemm_batch_execute(batch)
    assert g.spgemm_batch_status(batch) == g.SPG_OK
    for i, (A, B) in enumerate(pairs):
        cp, ri, v = (t.cpu().numpy() for t in g.spgemm_batch_result(batch, i))
        ref = oracle.spgemm(A, B)
        assert np.array_equal(cp, ref["colptr"]) and np.array_equal(ri, ref["rowidx"]), i
        check_values(v, ref["vals"], ref["absum"], f"instance {i}")
    g.spgemm_batch_destroy(batch)
