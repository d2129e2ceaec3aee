"""SpAsgn's merge at the sizes where it can go wrong: words of 32 entries,
tiles of 2048, rows of more than 1024 entries (taken by a whole block), tiles
with more entries of B than of A, and index vectors that do or do not keep
the order of B's rows.  Values are copied, or added once, so every comparison
is bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr, rand_sparse

pytestmark = pytest.mark.gpu


def H():
    from paper_1109_3739_gb300 import hspgemm
    return hspgemm


def one_row(nnz, n, row, m, dtype):
    """m x n matrix whose entries (every second column) all lie in one row."""
    rowptr = np.zeros(m + 1, np.int64)
    rowptr[row + 1:] = nnz
    return csr(m, n, rowptr, 2 * np.arange(nnz), I.random_values(nnz, dtype, 3, kind="signed"), dtype)


def check(A, Iv, Jv, B, what):
    h = H()
    for acc in (False, True):
        if acc and A.dtype == "bool":
            continue
        got = h.spasgn(h.DeviceCSR.from_host(A), Iv, Jv, h.DeviceCSR.from_host(B), accumulate=acc).to_host()
        assert_bitexact(got, oracle.spasgn(A, Iv, Jv, B, accumulate=acc, sr="plus_times"), f"{what} accumulate={acc}")


@pytest.mark.parametrize("nnz", [1, 31, 32, 33, 1024, 1025, 2047, 2048, 2049, 4096, 70001])
@pytest.mark.parametrize("touched", [True, False])
def test_row_lengths(nnz, touched):
    n = 2 * nnz + 5
    A = one_row(nnz, n, 2, 5, "i64")
    Iv = np.array([0, 2 if touched else 3, 4], np.int32)
    Jv = np.unique(np.array([0, 1, n // 2, n - 1, min(n - 1, 64)])).astype(np.int32)
    check(A, Iv, Jv, rand_sparse(3, len(Jv), 0.8, 9, "i64"), f"row of {nnz}")


@pytest.mark.parametrize("dt", ["f64", "f32", "i32", "bool"])
@pytest.mark.parametrize("order", ["increasing", "rows reversed", "all reversed"])
def test_dense_block(dt, order):
    """A block with far more entries than A; J decreasing puts B's rows out of order."""
    A = rand_sparse(150, 140, 0.02, 21, dt)
    Iv, Jv = np.arange(10, 110, dtype=np.int32), np.arange(20, 120, dtype=np.int32)
    if order != "increasing":
        Iv = Iv[::-1].copy()
    if order == "all reversed":
        Jv = Jv[::-1].copy()
    check(A, Iv, Jv, rand_sparse(100, 100, 0.6, 22, dt), f"{dt} {order}")


def test_whole_matrix():
    """I and J hold every row and column: only B remains (or A + B)."""
    A, B = rand_sparse(70, 90, 0.3, 31, "f64"), rand_sparse(70, 90, 0.2, 32, "f64")
    check(A, np.arange(70, dtype=np.int32), np.arange(90, dtype=np.int32), B, "whole")


def test_column_of_b_out_of_range():
    """An entry of B outside its J is reported, as by the products."""
    h = H()
    A = h.DeviceCSR.from_host(rand_sparse(20, 20, 0.3, 41, "f64"))
    B = csr(2, 3, [0, 1, 2], [0, 3], np.ones(2), "f64")
    with pytest.raises(h.HsError) as e:
        h.spasgn(A, np.array([1, 2], np.int32), np.array([3, 4, 5], np.int32), h.DeviceCSR.from_host(B))
    assert e.value.code == -8
