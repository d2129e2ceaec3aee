"""Tiny rows on both sides of the two lines that decide whether several share a
warp: their number, and their products on average.  Exact comparisons."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32"), ("or_and", "bool")])
@pytest.mark.parametrize("rows,entries,per", [(65535, 2, 4), (65536, 2, 4), (65536, 4, 4), (65536, 17, 1), (70001, 3, 5),
                                              (70001, 8, 4), (65537, 40, 0)])
def test_tiny_rows(rows, entries, per, sr, dt):
    """`entries` entries of A a row, each with `per` products (0: every other one with one)."""
    from paper_1109_3739_gb300 import hspgemm as h
    k, n = 5003, 777
    col = (np.arange(rows)[:, None] * 31 + np.arange(entries) * 7) % k
    A = csr(rows, k, np.arange(rows + 1) * entries, np.sort(col, axis=1).reshape(-1),
            I.random_values(rows * entries, dt, 88, kind="signed"), dt)
    lens = np.full(k, per) if per else np.arange(k) % 2
    bcol = np.concatenate([np.sort(I.random_unique_sequence(n, int(c), 89 + i)) for i, c in enumerate(lens) if c])
    bptr = np.concatenate([[0], np.cumsum(lens)])
    B = csr(k, n, bptr, bcol, I.random_values(int(bptr[-1]), dt, 90, kind="signed"), dt)
    got = h.spgemm(sr, h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)).to_host()
    assert_bitexact(got, oracle.spgemm(sr, A, B), f"{rows} rows of {entries} x {per}")
