"""SpRef's row sort at the edges of its tiers (8 entries: eight lanes; 64: a
warp; 2048: a block; beyond: a bitmap of B's columns, in chunks of 2^20), its
gather at the edges of words and tiles, and the symbolic and numeric warp rows
at the edges of their sorts.  Values are copied bit for bit; sums of small
integers are exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu


def H():
    from paper_1109_3739_gb300 import hspgemm
    return hspgemm


def rows_of_length(lengths, n, dtype, seed):
    """A matrix with rows of the given lengths, columns drawn without replacement."""
    cols = [np.sort(I.random_unique_sequence(n, c, seed + i)) for i, c in enumerate(lengths)]
    rowptr = np.concatenate([[0], np.cumsum(lengths)])
    col = np.concatenate(cols) if cols else np.zeros(0, np.int32)
    return csr(len(lengths), n, rowptr, col, I.random_values(len(col), dtype, seed, kind="signed"), dtype)


def check(A, Iv, Jv, what):
    h = H()
    got = h.spref(h.DeviceCSR.from_host(A), Iv, Jv).to_host()
    assert_bitexact(got, oracle.spref(A, Iv, Jv), what)


@pytest.mark.parametrize("dt", ["f64", "f32", "bool"])
@pytest.mark.parametrize("order", ["random", "increasing", "one repeated"])
def test_row_tiers(dt, order):
    lengths = [0, 1, 7, 8, 9, 31, 32, 33, 64, 65, 255, 256, 257, 511, 2047, 2048, 2049, 5000, 0, 3]
    n = 6000
    A = rows_of_length(lengths, n, dt, 5)
    Jv = I.random_unique_sequence(n, n, 6)
    if order == "increasing":
        Jv = np.sort(Jv)[::1]
    elif order == "one repeated":
        Jv = np.concatenate([Jv, Jv[:1]])
    Iv = np.concatenate([I.random_unique_sequence(len(lengths), len(lengths), 7), [17, 17, 4]]).astype(np.int32)
    check(A, Iv, Jv.astype(np.int32), f"{dt} {order}")


@pytest.mark.parametrize("total", [1, 31, 32, 33, 2047, 2048, 2049, 4097])
def test_gather_edges(total):
    """One long row among empty ones; half of the columns asked for."""
    A = rows_of_length([0] * 40 + [total] + [0] * 3000, 2 * total + 3, "i64", 11)
    Jv = I.random_unique_sequence(A.n, (A.n + 1) // 2, 12)
    check(A, np.arange(A.m, dtype=np.int32), Jv, f"{total}")
    check(A, np.array([40, 0, 40], np.int32), np.sort(Jv), f"{total} increasing")


def test_more_columns_than_the_bitmap():
    n = (1 << 20) + 4097
    A = rows_of_length([3000, 2500, 40], n, "i32", 21)
    check(A, np.array([2, 0, 1], np.int32), I.random_unique_sequence(n, n, 22), "wide")


@pytest.mark.parametrize("f", [33, 63, 64, 65, 128, 129, 256, 512, 513, 1024])
@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32"), ("or_and", "bool")])
def test_sorted_rows(f, sr, dt):
    """Rows of f products, a few of which share a column (runs across lanes and rounds of 32)."""
    n = 4 * f
    k = max(1, f // 16)
    lengths = [f // k + (1 if i < f % k else 0) for i in range(k)]
    B = rows_of_length(lengths, n, dt, 31)
    B.col[:] = np.concatenate([np.sort(np.unique(np.concatenate([[2 * f, 2 * f + 1], b])))[:len(b)]
                               for b in np.split(B.col, np.cumsum(lengths)[:-1])]).astype(np.int32)
    m = 37
    A = csr(m, k, np.arange(m + 1) * k, np.tile(np.arange(k), m), I.random_values(m * k, dt, 33, kind="signed"), dt)
    h = H()
    got = h.spgemm(sr, h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)).to_host()
    assert_bitexact(got, oracle.spgemm(sr, A, B), f"{sr} {f}")
