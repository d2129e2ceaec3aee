"""Units of rows with thousands of entries of A, their B segments laid out by a
warp where there are many such rows and by blocks where there are few.  Exact
comparisons."""
from __future__ import annotations

import os

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32")])
@pytest.mark.parametrize("lengths", [[1100] * 1600, [1100] * 1600 + [9000, 20000], [1023, 1024, 1025, 3000] * 3],
                         ids=["many", "many and two longer", "few"])
def test_units_of_long_rows(lengths, sr, dt):
    from paper_1109_3739_gb300 import hspgemm as h
    n, k, per = 150001, 30011, 4  # four products an entry: outputs of more than a table, in parts of the columns
    m = len(lengths)
    aptr = np.concatenate([[0], np.cumsum(lengths)])
    col = np.concatenate([(251 * i + np.arange(c)) % k for i, c in enumerate(lengths)])
    order = np.lexsort((col, np.repeat(np.arange(m), lengths)))
    A = csr(m, k, aptr, col[order], I.random_values(len(col), dt, 85, kind="signed"), dt)
    bcol = (I.draws(86, 1, 0, k * per) % np.uint64(n // per)).astype(np.int64).reshape(k, per) + np.arange(per) * (n // per)
    B = csr(k, n, np.arange(k + 1) * per, bcol.reshape(-1), I.random_values(k * per, dt, 87, kind="signed"), dt)
    ref = oracle.spgemm(sr, A, B, nthreads=os.cpu_count() or 1)
    assert np.diff(ref.rowptr).min() > 3900
    dA, dB = h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)
    assert_bitexact(h.spgemm(sr, dA, dB).to_host(), ref, "spgemm")
    P = h.Plan(sr, dA, dB)
    P.C.val.zero_()
    P.execute()
    P.status()
    assert_bitexact(P.C.to_host(), ref, "plan")
