"""The warp tables of the light columns at every size of their range (1 to 1024
products a column, with and without repeated rows, rows of 10 to 22 bits): the
plan's path, the batched launch and the one-launch multiply against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity, check_values, run_gpu

pytestmark = pytest.mark.gpu


def pair(m, most, values, seed):
    """A: m x 400, 8 rows per column; B: one column for every count of entries
    up to `most` / 8 (so 8, 16, ... `most` products), and an empty one."""
    rng = np.random.default_rng(seed)
    k, q = 400, np.arange(0, most // 8 + 1)
    rows = np.sort(np.stack([rng.choice(m, 8, replace=False) for _ in range(k)]), 1).ravel()
    draw = (lambda n: rng.uniform(-1, 1, n)) if values == "f64" else (lambda n: rng.integers(-2**62, 2**62, n))
    A = synth._csc_from_sorted(m, k, np.repeat(np.arange(k), 8), rows, draw(rows.size))
    br = np.concatenate([np.sort(rng.choice(k, n, replace=False)) for n in q] + [np.zeros(0, np.int64)])
    B = synth._csc_from_sorted(k, q.size, np.repeat(np.arange(q.size), q), br.astype(np.int64), draw(br.size))
    return A, B


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("m", [900, 5000, 200_000, 3_000_000])
def test_every_table_size(m, values):
    A, B = pair(m, 1024, values, 21)
    ref = oracle.spgemm(A, B)
    assert_full_parity(run_gpu(A, B, 2, 64), ref, f"plan m={m} {values}")
    dA, dB = g.to_device(A, ptr_dtype=torch.int32), g.to_device(B, ptr_dtype=torch.int32)
    batch = g.spgemm_batch_create([dA, dA], [dB, dB])
    g.spgemm_batch_execute(batch)
    assert g.spgemm_batch_status(batch) == g.SPG_OK
    cp, ri, v = (t.cpu().numpy() for t in g.spgemm_batch_result(batch, 1))
    assert np.array_equal(cp, ref["colptr"]) and np.array_equal(ri, ref["rowidx"])
    check_values(v, ref["vals"], ref["absum"], f"batch m={m} {values}")
    g.spgemm_batch_destroy(batch)


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("most,table_log", [(128, 8), (512, 10)])
def test_one_launch_tables(most, table_log, values):
    A, B = pair(100_000, most, values, 22)
    sp = g.SmallProduct(*(g.to_device(M, ptr_dtype=torch.int32) for M in (A, B)), P=3, b=64, table_log=table_log)
    assert_full_parity(sp.run().C(), oracle.spgemm(A, B), f"one launch {table_log} {values}")


def test_repeated_rows_and_a_learned_overflow():
    """Products of few rows many times over, and a learned capacity that overflows the table."""
    rng = np.random.default_rng(23)
    A, B = pair(40, 1024, "f64", 24)          # 40 rows: every table slot is hit again and again
    assert_full_parity(run_gpu(A, B, 1, 64), oracle.spgemm(A, B), "40 rows")
    A, B = pair(50_000, 1024, "f64", 25)
    model = g.spgemm_model_create(1)
    g.spgemm_model_set_params(model, np.zeros(g.SPG_MODEL_NPARAMS, np.float32))   # predicts 1 entry
    C, st = g.spgemm_1d_multiply(g.to_device(A), g.to_device(B), sizing=g.SPG_SIZING_LEARNED, model=model)
    assert st == g.SPG_OVERFLOW_RECOMPUTED
    assert_full_parity(C, oracle.spgemm(A, B), "learned overflow")
