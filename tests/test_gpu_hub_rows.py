"""Rows of thousands of entries of A and few products an entry, by how many of
them a product has: few enough to be moved to the kernel of 1024 threads, too
many of them, and so many that only the longest are.  Exact comparisons."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu


def operands(lengths, n, dt, k=20011):
    """Rows of the given lengths over k columns; B's rows hold an entry each."""
    offs = np.concatenate([[0], np.cumsum(lengths)])
    col = np.concatenate([(97 * i + np.arange(c)) % k for i, c in enumerate(lengths)])
    row = np.repeat(np.arange(len(lengths)), lengths)
    order = np.lexsort((col, row))
    A = csr(len(lengths), k, offs, col[order], I.random_values(len(col), dt, 81, kind="signed"), dt)
    bcol = (I.draws(82, 1, 0, k) % np.uint64(n)).astype(np.int32)
    B = csr(k, n, np.arange(k + 1), bcol, I.random_values(k, dt, 83, kind="signed"), dt)
    return A, B


SHAPES = {"few": [5000] * 3 + [17000], "at the limit": [4097] * 304, "too many": [4097] * 310,
          "the longest": [4097] * 300 + [17000] * 20, "none": [16500] * 310}


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("sr,dt,n", [("plus_times", "i64", 256), ("min_plus", "f32", 1500), ("or_and", "bool", 1000)])
def test_products_with_hub_rows(shape, sr, dt, n):
    from paper_1109_3739_gb300 import hspgemm as h
    lengths = [x for i, c in enumerate(SHAPES[shape]) for x in (c, (3 * i) % 200)]
    A, B = operands(lengths, n, dt)
    ref = oracle.spgemm(sr, A, B)
    dB = h.DeviceCSR.from_host(B)
    for dcsr in (False, True):
        dA = h.DeviceCSR.from_host(A, dcsr=dcsr)
        assert_bitexact(h.spgemm(sr, dA, dB).to_host(), ref, f"{shape} dcsr={dcsr}")
    assert_bitexact(h.spgemm_noalloc(sr, h.DeviceCSR.from_host(A), dB, len(ref.col)).to_host(), ref, f"{shape} noalloc")
