"""The heavy columns' product walk and accumulator at their edges: segment
lengths around the length classes (31 | 32, 255 | 256), columns of B around the
staging batch (256 entries) and with more middle-length segments than the
windows hold, items whose rows all have a slot (dense) and items addressed by
rank (sparse), many products of one row at once, NaN and infinities.  Doubles
within the result contract's 1e-12 * sum |a b|, integers exactly."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity, run_gpu

pytestmark = pytest.mark.gpu


def columns(lens, m, rng, values, window=None):
    """m-row matrix whose column c holds lens[c] distinct rows (drawn below `window`)."""
    w = m if window is None else window
    cols = np.repeat(np.arange(len(lens)), lens)
    rows = np.concatenate([np.sort(rng.choice(w, n, replace=False)) for n in lens])
    vals = rng.uniform(-1, 1, rows.size) if values == "f64" else rng.integers(-2**62, 2**62, rows.size)
    return synth._csc_from_sorted(m, len(lens), cols, rows, vals)


SHAPES = {
    # name: (segment lengths of A's columns, entries of every column of B, rows of A)
    "short_31": ([31] * 300, [255, 256, 257, 300], 20000),
    "mid_32_255": ([32, 255] * 130, [256, 260, 129], 60000),
    "mids_past_the_windows": ([200] * 256 + [5] * 64 + [700] * 8, [328, 300, 256], 70000),
    "long_256_3000": ([256, 257, 3000, 1] * 60, [240, 64, 63], 100000),
    "one_each": ([1, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 1000], [12, 11, 5], 30000),
    "dense_item": ([31, 32, 500, 1000] * 70, [280, 256, 9], 1024),
    "dense_item_ragged": ([7, 300, 64] * 90, [270, 13], 3001),
    "dense_slabs": ([3000, 255, 31] * 60, [180, 150], 20000),
}


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_walk_edges_match_oracle(shape, values):
    lens, nb, m = SHAPES[shape]
    rng = np.random.default_rng(11)
    A = columns(lens, m, rng, values)
    B = columns(nb, len(lens), rng, values)
    for R in (1024, 4096, 8192, 16384):
        C = run_gpu(A, B, 2, 64, light_max=32, slab_rows=R)
        assert_full_parity(C, oracle.spgemm(A, B), f"{shape} {values} R={R}")


@pytest.mark.parametrize("m,window", [(5000, 40), (90000, 90000)])
def test_many_products_of_one_row(m, window):
    """Every column of A holds the same few rows (all warps add to the same
    slots), in a dense and in a rank-addressed item."""
    rng = np.random.default_rng(12)
    if window < m:
        A = columns([33] * 900, m, rng, "f64", window=window)
    else:
        rows = np.sort(rng.choice(m, 40, replace=False))
        A = synth._csc_from_sorted(m, 900, np.repeat(np.arange(900), 40), np.tile(rows, 900),
                                   rng.uniform(-1, 1, 36000))
    B = columns([900, 899, 257], 900, rng, "f64")
    assert_full_parity(run_gpu(A, B, 1, 64, light_max=32, slab_rows=1024), oracle.spgemm(A, B), "one row")


def test_nan_and_infinities_stay_where_they_belong():
    rng = np.random.default_rng(13)
    A = columns([40, 300, 31] * 40, 6000, rng, "f64")
    B = columns([120, 100], 120, rng, "f64")
    A.vals[::97] = np.inf
    A.vals[5::101] = np.nan
    # a signalling NaN among the inputs
    A.vals.view(np.uint64)[7::103] = 0x7FF4A5C300000000
    C = run_gpu(A, B, 1, 64, light_max=32, slab_rows=1024)
    cp, ri, v = C.to_host()
    dense = np.zeros((6000, 120))
    dense[A.rowidx, np.repeat(np.arange(120), np.diff(A.colptr))] = A.vals
    for j in range(2):
        want = np.zeros(6000)
        ks, bv = B.col(j)
        with np.errstate(invalid="ignore"):
            for k, x in zip(ks, bv):
                r, a = A.col(int(k))
                want[r] += a * x
        got = v[cp[j]:cp[j + 1]]
        want = want[ri[cp[j]:cp[j + 1]]]
        assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
        fine = np.isfinite(want)
        mag = sum(np.abs(np.where(np.isfinite(dense[:, k]), dense[:, k], 0.0) * x) for k, x in zip(ks, bv))
        assert np.all(np.abs(got[fine] - want[fine]) <= 1e-12 * mag[ri[cp[j]:cp[j + 1]]][fine])
        assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])


@pytest.mark.parametrize("n,s", [(9000, 3), (700, 40)])
def test_betweenness_on_long_and_short_frontiers(n, s):
    """Frontier columns of several pieces (256 entries a warp) and shorter than one."""
    from oracle import bc as obc
    rng = np.random.default_rng(14)
    r, c = rng.integers(0, n, 6 * n), rng.integers(0, n, 6 * n)
    keep = r != c
    cols, rows = synth._sort_dedup(np.concatenate([c[keep], r[keep]]), np.concatenate([r[keep], c[keep]]), n)
    A = synth._csc_from_sorted(n, n, cols, rows, np.ones(cols.size))
    src = rng.choice(n, s, replace=False).astype(np.int32)
    bc, _, _ = g.spgemm_bc_batch(g.to_device(A), torch.from_numpy(src).cuda(), P=2, b=64)
    want = obc.brandes(A, src)
    want = want[0] if isinstance(want, tuple) else want
    got = bc.cpu().numpy()
    assert np.all(np.abs(got - want) <= 1e-9 * np.maximum(1.0, np.abs(want)))


@pytest.mark.parametrize("values", ["f64", "i64"])
@pytest.mark.parametrize("m,R", [(90_000, 1024), (90_000, 4096), (90_000, 8192), (30_000, 16384)])
def test_wide_masked_items(m, R, values):
    """Few products per entry and slab under a mask: items of 10,240 entries and
    512 threads; columns of several items, segments around 127 | 128 entries
    and more than a batch (512) of entries."""
    from test_gpu_mask import mask_from_pattern
    rng = np.random.default_rng(15)
    lens = [4] * 5000 + [31, 32, 127, 128, 129] * 4
    A = columns(lens, m, rng, values)
    B = columns([5020, 5000, 513, 512, 511], len(lens), rng, values)
    M = columns([m // 2, m // 3, m // 2, 100, m], m, rng, "i64")
    for complement in (False, True):
        mask = mask_from_pattern(M)
        plan = g.spgemm_plan(g.to_device(A), g.to_device(B), 2, 64, light_max=32, slab_rows=R, mask=mask,
                             mask_complement=complement)
        g.spgemm_symbolic(plan)
        C = g.spgemm_numeric(plan)
        torch.cuda.synchronize()
        g.spgemm_plan_destroy(plan)
        assert_full_parity(C, oracle.spgemm_masked(A, B, M, complement), f"wide m={m} R={R} {values} {complement}")
