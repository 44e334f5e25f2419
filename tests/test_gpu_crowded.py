"""Products that come few to a batch of B's entries or many to a row: the windows
of a batch shared by number instead of claimed, and the walks that combine a
warp's products of one row before they add them.  Doubles within the result
contract's 1e-12 * sum |a b|, integers exactly."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity, check_values, mask_from_pattern, run_gpu
from test_gpu_heavy_walk import columns

pytestmark = pytest.mark.gpu


def one_row_each(m, k, n, per, values, rng, share=0.0):
    """A: one row per column (row 0 for `share` of them); B: `per` entries per column."""
    rows = np.where(rng.random(k) < share, 0, rng.integers(0, m, k))
    draw = (lambda s: rng.uniform(-1, 1, s)) if values == "f64" else (lambda s: rng.integers(-2**62, 2**62, s))
    A = synth._csc_from_sorted(m, k, np.arange(k), rows, draw(k))
    br = np.concatenate([np.sort(rng.choice(k, per, replace=False)) for _ in range(n)])
    return A, synth._csc_from_sorted(k, n, np.repeat(np.arange(n), per), br, draw(br.size))


def kernel_ms(A, B, group="ms_num_heavy", **kw):
    """Time of the heavy (or light) numeric kernels, the shortest of five passes."""
    dA, dB = (g.to_device(M, ptr_dtype=torch.int32, idx_dtype=torch.int32) for M in (A, B))
    plan = g.spgemm_plan(dA, dB, 4, 1024, **kw)
    g.spgemm_symbolic(plan)
    C = g.spgemm_numeric(plan)
    ms = []
    for _ in range(5):
        g.spgemm_numeric_refresh(plan, C)
        ms.append(g.spgemm_plan_stats(plan)[group])
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
    assert kernel_ms(*ten) < 2.7 * kernel_ms(*one)


def star(m, k, n, per, values, rng):
    """A's columns: nothing, row 0 alone, row 0 and a few others, or 40 and more
    rows; B takes them in any order, so that a window's owners have gaps."""
    kind = rng.integers(0, 12, k)
    cols, rows = [], []
    for c in range(k):
        d = 0 if kind[c] < 2 else 1 if kind[c] < 9 else int(rng.integers(2, 5)) if kind[c] < 11 else int(rng.integers(40, 300))
        r = np.unique(np.concatenate([[0], rng.choice(m, d - 1, replace=False)])) if d else np.zeros(0, np.int64)
        cols.append(np.full(r.size, c))
        rows.append(r)
    cols, rows = np.concatenate(cols), np.concatenate(rows).astype(np.int64)
    draw = (lambda s: rng.uniform(-1, 1, s)) if values == "f64" else (lambda s: rng.integers(-2**62, 2**62, s))
    A = synth._csc_from_sorted(m, k, cols, rows, draw(rows.size))
    br = np.concatenate([np.sort(rng.choice(k, p, replace=False)) for p in per])
    return A, synth._csc_from_sorted(k, n, np.repeat(np.arange(n), per), br, draw(br.size))


PER = [33, 255, 256, 257, 300, 512, 513, 600, 2049, 2305, 3000]


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("share", [0.3, 0.6, 1.0, "star"])
@pytest.mark.parametrize("m", [3000, 30000])
def test_heavy_columns_with_a_crowded_row(m, share, values):
    """One base slab and several, under a mask, and sized by the learned model;
    columns of one batch (256 entries), of several, and of more than eight."""
    rng = np.random.default_rng(31)
    k, n = 3500, len(PER)
    if share == "star":
        A, B = star(m, k, n, PER, values, rng)
    else:
        A, _ = one_row_each(m, k, 1, 1, values, rng, share)
        B = columns(PER, k, rng, values)
    ref = oracle.spgemm(A, B)
    for R in (1024, 4096):
        assert_full_parity(run_gpu(A, B, 2, 64, light_max=32, slab_rows=R), ref, f"m={m} {share} {values} R={R}")
    M = columns([m // 2] * n, m, rng, "i64")
    for complement in (False, True):
        plan = g.spgemm_plan(g.to_device(A), g.to_device(B), 2, 64, light_max=32, mask=mask_from_pattern(M),
                             mask_complement=complement)
        C = g.spgemm_numeric(plan)
        torch.cuda.synchronize()
        g.spgemm_plan_destroy(plan)
        assert_full_parity(C, oracle.spgemm_masked(A, B, M, complement), f"masked {m} {share} {values}")
    model = g.spgemm_model_create(1)
    C, _ = g.spgemm_1d_multiply(g.to_device(A), g.to_device(B), 2, 64, light_max=32, slab_rows=1024,
                                sizing=g.SPG_SIZING_LEARNED, model=model)
    assert_full_parity(C, ref, f"learned {m} {share} {values}")


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("m,d", [(1, 1), (4, 1), (4, 4), (32, 3), (32, 8), (500, 2)])
def test_light_columns_with_crowded_rows(m, d, values):
    rng = np.random.default_rng(32)
    A = columns([d if c % 5 else 0 for c in range(3500)], m, rng, values)
    B = columns([1, 31, 32] + PER, 3500, rng, values)
    ref = oracle.spgemm(A, B)
    dA, dB = (g.to_device(M, ptr_dtype=torch.int32, idx_dtype=torch.int32) for M in (A, B))
    assert_full_parity(run_gpu(A, B, 2, 64), ref, f"plan m={m} d={d} {values}")
    model = g.spgemm_model_create(1)
    C, _ = g.spgemm_1d_multiply(dA, dB, 2, 64, sizing=g.SPG_SIZING_LEARNED, model=model)
    assert_full_parity(C, ref, f"learned m={m} d={d} {values}")
    batch = g.spgemm_batch_create([dA], [dB])
    g.spgemm_batch_execute(batch)
    assert g.spgemm_batch_status(batch) == g.SPG_OK
    cp, ri, v = (t.cpu().numpy() for t in g.spgemm_batch_result(batch, 0))
    assert np.array_equal(cp, ref["colptr"]) and np.array_equal(ri, ref["rowidx"])
    check_values(v, ref["vals"], ref["absum"], f"batch m={m} d={d} {values}")
    g.spgemm_batch_destroy(batch)
    for table_log in (8, 10) if m <= 128 else (10,):
        sp = g.SmallProduct(dA, dB, P=3, b=64, table_log=table_log)
        assert_full_parity(sp.run().C(), ref, f"one launch m={m} d={d} {values}")


def test_crowded_doubles_keep_up_with_integers():
    """99% of a heavy column's products on one row, and a light column's on four
    rows: combined, 1.5 and 1.8 times the integers' time (16 and 4.3 times with
    an exchange for every product)."""
    rng = np.random.default_rng(33)
    ms = {v: kernel_ms(*one_row_each(4000, 200000, 300, 100000, v, np.random.default_rng(34), share=0.99))
          for v in ("f64", "i64")}
    assert ms["f64"] < 4 * ms["i64"], ms
    for v in ("f64", "i64"):
        A = columns([4] * 20000, 4, rng, v)
        ms[v] = kernel_ms(A, columns([2000] * 2000, 20000, rng, v), "ms_num_light")
    assert ms["f64"] < 3 * ms["i64"], ms
