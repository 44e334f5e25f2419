"""The planning kernels at the sizes where their launches change: scans by one
CTA, by two and by three launches, column bins in longer chunks, D~ lists sized
by their bound or by a read-back, block bounds in shared or global memory, lane
groups per column, and input validation of unaligned row ids."""
import numpy as np
import pytest
import torch

import oracle
import paper_2408_14558_gb300 as g
import synth
from parity import assert_full_parity, run_gpu

pytestmark = pytest.mark.gpu


def banded(m, n, per, rng, values="f64"):
    """m x n, column j holds rows j % m, j % m + 1, ... (per entries, wrapped ones dropped)."""
    cols = np.repeat(np.arange(n, dtype=np.int64), per)
    rows = cols % m + np.tile(np.arange(per), n)
    ok = rows < m
    cols, rows = cols[ok], rows[ok]
    vals = rng.uniform(-1, 1, rows.size) if values == "f64" else rng.integers(-5, 6, rows.size)
    return synth._csc_from_sorted(m, n, cols, rows, vals)


@pytest.mark.parametrize("n", [1, 2047, 2049, 8192, 32768, 32769, 40000])
@pytest.mark.parametrize("per", [1, 9, 64, 65])
def test_scan_and_group_edges(n, per):
    rng = np.random.default_rng(n + per)
    A, B = banded(n, n, 3, rng), banded(n, n, per, rng)
    for P in (1, 7):
        assert_full_parity(run_gpu(A, B, P, 64), oracle.spgemm(A, B), f"n={n} per={per} P={P}")


@pytest.mark.parametrize("P", [512, 513])
def test_many_blocks(P):
    rng = np.random.default_rng(3)
    A, B = banded(6000, 6000, 4, rng), banded(6000, 5000, 5, rng)
    dA, dB = (g.to_device(M, ptr_dtype=torch.int32, idx_dtype=torch.int32) for M in (A, B))
    plan = g.spgemm_plan(dA, dB, P, 64)
    blk = g.spgemm_plan_blocks(plan)
    g.spgemm_symbolic(plan)
    C = g.spgemm_numeric(plan)
    assert_full_parity(C, oracle.spgemm(A, B), f"P={P}")
    want = oracle.block_volumes(A, B, blk["bounds"], 64)
    for q in ("flops", "gathered", "remote"):
        assert np.array_equal(blk[q], want[q]), q
    g.spgemm_plan_destroy(plan)


@pytest.mark.parametrize("n,P", [(1 << 20, 1), ((1 << 20) + 1, 1), (1 << 20, 300), (4_200_000, 2)])
def test_large_scans_and_bins(n, P):
    """nnz(B) on both sides of 2^20; P * ceil(k / 32) beyond the two-launch scan;
    more columns than 2048 chunks of 2048."""
    rng = np.random.default_rng(4)
    A, B = banded(n, n, 1, rng, "i64"), banded(n, n, 1, rng, "i64")
    assert_full_parity(run_gpu(A, B, P, 4096), oracle.spgemm(A, B), f"n={n} P={P}")


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("at", [0, 1, 2, 3, 5, 250, 254, 255])
def test_validation_finds_a_bad_row_at_every_alignment(offset, at):
    rng = np.random.default_rng(5)
    A = synth.uniform_columns(64, 4, seed=1)
    buf = torch.zeros(256 + 4, dtype=torch.int32, device="cuda")
    row = buf[offset:offset + 256]
    row.copy_(torch.from_numpy(A.rowidx))
    M = g.DeviceCSC(64, 64, torch.from_numpy(A.colptr.astype(np.int32)).cuda(), row,
                    torch.from_numpy(A.vals).cuda())
    assert_full_parity(g.multiply(M, M, 2, 16), oracle.spgemm(A, A), "aligned or not")
    for bad in (-1, 64, int(A.rowidx[at - 1]) if at % 4 else 1000):   # below, above, repeated in its column
        keep = int(row[at])
        row[at] = bad
        with pytest.raises(g.SpgError) as e:
            g.multiply(M, M, 2, 16)
        assert e.value.status == g.SPG_INVALID_INPUT
        with pytest.raises(g.SpgError) as e:
            g.multiply(M, M, 2, 16, split=g.SPG_SPLIT_FLOPS)
        assert e.value.status == g.SPG_INVALID_INPUT
        row[at] = keep
    assert_full_parity(g.multiply(M, M, 2, 16), oracle.spgemm(A, A), "restored")


@pytest.mark.parametrize("lens", [[1], [1] * 31 + [2], [2] + [1] * 31, [1, 1, 40], [32], [1, 2]])
@pytest.mark.parametrize("P", [1, 5])
def test_gather_of_scattered_short_columns(lens, P):
    """A~'s columns of one entry or little more, picked from A with gaps: a
    32-entry step meets up to 32 columns, wherever the 32 that the lanes hold end."""
    rng = np.random.default_rng(len(lens) + P)
    n = 6000
    cols = np.repeat(np.arange(n), np.resize(lens, n))
    rows = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in np.resize(lens, n)])
    A = synth._csc_from_sorted(n, n, cols, rows, rng.uniform(-1, 1, rows.size))
    for per in (3, 40):   # B's columns need some of A's only
        picks = np.concatenate([np.sort(rng.choice(n, per, replace=False)) for _ in range(60)])
        B = synth._csc_from_sorted(n, 60, np.repeat(np.arange(60), per), picks, rng.uniform(-1, 1, picks.size))
        assert_full_parity(run_gpu(A, B, P, 64), oracle.spgemm(A, B), f"per={per}")


@pytest.mark.parametrize("lens", [[520] * 30, [700, 0, 4000, 1, 513] * 4])
def test_long_columns_of_B(lens):
    """A mean above 512 entries per column of B: one CTA per column in the statistics."""
    rng = np.random.default_rng(6)
    A = banded(5000, 5000, 3, rng)
    cols = np.repeat(np.arange(len(lens)), lens)
    rows = np.concatenate([np.sort(rng.choice(5000, k, replace=False)) for k in lens])
    B = synth._csc_from_sorted(5000, len(lens), cols, rows, rng.uniform(-1, 1, rows.size))
    assert_full_parity(run_gpu(A, B, 3, 64), oracle.spgemm(A, B), "long columns of B")


def test_plans_of_several_threads_and_streams():
    """Plans take their page-locked words and events from a pool: four threads,
    each on its own stream, make, keep and destroy plans (more at a time than
    the pool keeps, and one of more blocks than its words hold)."""
    import threading
    rng = np.random.default_rng(7)
    A = banded(3000, 3000, 4, rng)
    ref = oracle.spgemm(A, A)
    bad = []

    def work(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                dA = g.to_device(A, ptr_dtype=torch.int32, idx_dtype=torch.int32)
                plans = [g.spgemm_plan(dA, dA, 1 + i, 64) for _ in range(8)]
                for plan in plans:
                    g.spgemm_symbolic(plan)
                Cs = [g.spgemm_numeric(plan) for plan in plans] + [g.multiply(dA, dA, 1500, 64)]
                s.synchronize()
                assert all(g.spgemm_plan_stats(p)["ms_numeric"] > 0 for p in plans)
                fresh = g.spgemm_plan(dA, dA, 1, 64)
                assert g.spgemm_plan_stats(fresh)["ms_numeric"] == 0
                for C in Cs:
                    assert_full_parity(C, ref, f"thread {i}")
                for plan in plans + [fresh]:
                    g.spgemm_plan_destroy(plan)
        except BaseException as e:   # noqa: BLE001
            bad.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
