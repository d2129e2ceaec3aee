"""Rows in which many products fall on one column, in the kernels that sort a
row's products instead of hashing them.  Integer sums and minima are exact;
sums of f32 are held to the bound of the order they are formed in."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu
N = 300001


def H():
    from paper_1109_3739_gb300 import hspgemm
    return hspgemm


def rows_of_runs(rows, dt, seed, n=N):
    """A, B and for each list of run lengths one row of A * B with that many products on each of its columns: the
    j-th entry of A meets a row of B with the columns of more than j products."""
    order = np.argsort(I.draws(seed, 3, 0, n), kind="stable")
    pieces, arows, nb = [], [], 0
    for i, runs in enumerate(rows):
        runs = np.asarray(runs)
        cols = order[(37 * i) % 1000:][:len(runs)]
        for j in range(int(runs.max())):
            pieces.append(np.sort(cols[runs > j]))
        arows.append(np.arange(nb, len(pieces)))
        nb = len(pieces)
    bptr = np.concatenate([[0], np.cumsum([len(p) for p in pieces])])
    aptr = np.concatenate([[0], np.cumsum([len(r) for r in arows])])
    B = csr(nb, n, bptr, np.concatenate(pieces), I.random_values(int(bptr[-1]), dt, seed, kind="signed"), dt)
    A = csr(len(rows), nb, aptr, np.concatenate(arows), I.random_values(int(aptr[-1]), dt, seed + 1, kind="signed"), dt)
    return A, B


def every_way(sr, A, B, check):
    """check(C, what) of the product by every entry point that sorts rows."""
    h = H()
    dA, dB = h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)
    check(h.spgemm(sr, dA, dB).to_host(), "spgemm")
    P = h.Plan(sr, dA, dB)
    P.C.val.zero_()
    P.execute()
    P.status()
    check(P.C.to_host(), "plan")
    check(h.spgemm_batched(sr, [dA], [dB])[0].to_host(), "batched")
    Q = h.BatchPlan(sr, [dA], [dB])
    Q.execute()
    check(Q.result()[0].to_host(), "batch plan")


def padded(runs, f):
    """The runs, and columns of one product up to f products."""
    return list(runs) + [1] * (f - sum(runs))


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32"), ("min_plus", "i32")])
@pytest.mark.parametrize("f", [64, 65, 128, 200, 256, 511, 512, 1000, 1024])
def test_sorted_rows(f, sr, dt):
    """Runs on both sides of the walked length, of a round and of two, alone and side by side, at every offset."""
    half = f // 2
    rows = [padded([r], f) for r in (1, 2, 3, 4, 5, 6, 31, 32, 33, 63, 64, 65, half, half + 1) if r <= half + 1]
    for r in (3, 4, 5, 6, 9, 17, 33):  # as many runs as the share of repeated columns allows
        rows += [padded([r] * (half // (r - 1) * (r - 1) // r), f)] if half > r else []
    rows += [padded([2, 3, 4, 5, 6, 7] * (f // 64), f)] * 4 + [padded([3, 33, 5, 4], f)] * 4 if f >= 128 else []
    A, B = rows_of_runs(rows, dt, 61)
    ref = oracle.spgemm(sr, A, B)
    every_way(sr, A, B, lambda C, what: assert_bitexact(C, ref, f"{what} {f}"))


@pytest.mark.parametrize("f", [128, 256, 512, 1024])
def test_sums_of_a_long_run_stay_accurate(f):
    """One large product and many that are each less than half a unit in its last place: added one after another
    they vanish, and the sum is off by their whole sum.  A run is added up as a tree over each 32 of its elements
    and then round by round, so its error is at most (5 + rounds + 1) roundings of the sum."""
    lengths = [5, 9, 33, f // 4, f // 2, f // 2 + 1]
    A, B = rows_of_runs([padded([r], f) for r in lengths], "f32", 62)
    A.val[:] = 1.0
    B.val[:] = np.float32(0.75 * 2.0 ** -24)
    for q in A.rowptr[:-1]:
        k = A.col[q]
        B.val[B.rowptr[k]:B.rowptr[k + 1]] = 1.0
    exact = [1.0 + (r - 1) * 0.75 * 2.0 ** -24 for r in lengths]

    def check(C, what):
        for i, r in enumerate(lengths):
            v = C.val[C.rowptr[i]:C.rowptr[i + 1]].astype(np.float64)
            assert len(v) == f - r + 1
            bound = (5 + (r + 31) // 32 + 1 + 1) * 2.0 ** -24 * exact[i]
            assert abs(v.max() - exact[i]) <= bound, (what, f, r, v.max() - exact[i], bound)
            assert np.count_nonzero(v == 1.0) >= f - r

    every_way("plus_times", A, B, check)


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32"), ("or_and", "bool")])
def test_block_rows_with_a_repeated_column(sr, dt):
    """Rows of 1100 to 3600 outputs with 31 to 34 products, an eighth of the outputs and a few columns of each:
    sorted as they are up to 32 products a column, handed to the table beyond; and all of a row's columns but one
    in one bucket of its sort."""
    rows = []
    for c in (1100, 1820, 2300, 3600):
        rows += [[r] + [1] * (c - 1) for r in (2, 31, 32, 33, 34, c // 9)]
        rows += [[r] * (c // 10 // r) + [1] * (c - c // 10 // r) for r in (16, 32, 33)] + [[20, 2, 33] + [1] * (c - 3)]
    A, B = rows_of_runs(rows, dt, 63)
    h = H()
    for n, far in ((N, 0), (1 << 24, (1 << 24) - N)):  # (far: the greatest column moved away from the others)
        B2 = csr(B.m, n, B.rowptr, np.where(B.col == B.col.max(), B.col + far, B.col), B.val, dt)
        ref = oracle.spgemm(sr, A, B2)
        dA, dB = h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B2)
        assert_bitexact(h.spgemm(sr, dA, dB).to_host(), ref, f"spgemm {n}")
        P = h.Plan(sr, dA, dB)
        P.execute()
        P.status()
        assert_bitexact(P.C.to_host(), ref, f"plan {n}")
