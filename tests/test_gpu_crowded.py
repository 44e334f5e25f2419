"""Products that come few to a batch of B's entries or many to a row: the windows
of a batch shared by number instead of claimed.  Doubles within the result
contract's 1e-12 * sum |a b|, integers exactly."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity, run_gpu
from test_gpu_heavy_walk import columns

pytestmark = pytest.mark.gpu


def one_row_each(m, k, n, per, values, rng, share=0.0):
    """A: one row per column (row 0 for `share` of them); B: `per` entries per column."""
    rows = np.where(rng.random(k) < share, 0, rng.integers(0, m, k))
    draw = (lambda s: rng.uniform(-1, 1, s)) if values == "f64" else (lambda s: rng.integers(-2**62, 2**62, s))
    A = synth._csc_from_sorted(m, k, np.arange(k), rows, draw(k))
    br = np.concatenate([np.sort(rng.choice(k, per, replace=False)) for _ in range(n)])
    return A, synth._csc_from_sorted(k, n, np.repeat(np.arange(n), per), br, draw(br.size))


def heavy_ms(A, B, **kw):
    """Time of the heavy numeric kernel, the shortest of five passes."""
    dA, dB = (g.to_device(M, ptr_dtype=torch.int32, idx_dtype=torch.int32) for M in (A, B))
    plan = g.spgemm_plan(dA, dB, 4, 1024, **kw)
    g.spgemm_symbolic(plan)
    C = g.spgemm_numeric(plan)
    ms = []
    for _ in range(5):
        g.spgemm_numeric_refresh(plan, C)
        ms.append(g.spgemm_plan_stats(plan)["ms_num_heavy"])
    g.spgemm_plan_destroy(plan)
    return min(ms)


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("products", [31, 32, 33, 255, 256, 257, 288, 1023, 1024, 1025, 1056])
@pytest.mark.parametrize("long_seg", [0, 300])
def test_batches_of_few_windows(products, long_seg, values):
    """Batches of 1, 8, 9, 32, 33 and 34 windows, with and without a long segment."""
    rng = np.random.default_rng(products)
    short = -(-products // 120)             # segments short enough for 120 of them
    lens = [short] * (products // short) + ([products % short] if products % short else [])
    lens += [long_seg] if long_seg else []
    A = columns(lens, 3000, rng, values)
    B = columns([len(lens), len(lens) // 2 + 1], len(lens), rng, values)
    for R in (1024, 4096):
        assert_full_parity(run_gpu(A, B, 1, 64, light_max=32, slab_rows=R), oracle.spgemm(A, B),
                           f"{products} products, {long_seg}, {values}, R={R}")


def test_few_products_a_batch_do_not_wait():
    """Ten slabs visit every entry of B ten times, with a tenth of the products
    each: sharing the windows by number, 2.4 times the time of one slab (3.0 and
    more when every batch waits for claims)."""
    rng = np.random.default_rng(3)
    one = one_row_each(4000, 200000, 300, 100000, "i64", rng)
    ten = one_row_each(40000, 200000, 300, 100000, "i64", rng, share=0.9)
    assert heavy_ms(*ten) < 2.7 * heavy_ms(*one)
