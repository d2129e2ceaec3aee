"""The no-allocation entry point at the limit of its fixed scratch."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu


def test_as_many_rows_as_the_fixed_scratch_holds():
    """16 bytes a row, the scan's partial sums and 1 KB: the counters are not taken from the rows' room."""
    m, k = 2096544, 8
    A = csr(m, k, np.arange(m + 1), np.arange(m) % k, np.arange(m) % 13, "i64")
    A.val = A.val.astype(np.int64)
    B = I.er_matrix(k, k, 2, seed=76, dtype="i64")
    from paper_1109_3739_gb300 import hspgemm as h
    want = oracle.spgemm("plus_times", A, B)
    got = h.spgemm_noalloc("plus_times", h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B), len(want.col))
    assert_bitexact(got.to_host(), want, "noalloc")
