"""SpRef with a J of 2^24 columns: many rows of more than 2048 entries, which
the radix sort takes there, and a few of them, which stay with the bitmap over
seventeen stretches of columns.  Values are copied bit for bit."""
from __future__ import annotations

import functools

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact, csr

pytestmark = pytest.mark.gpu
N = (1 << 24) + 3


@functools.lru_cache(maxsize=None)
def order():
    return np.argsort(I.draws(91, 1, 0, N), kind="stable").astype(np.int32)


def long_rows(count, dt):
    """`count` rows of 2049 to 2600 entries among short and empty ones."""
    lengths = np.zeros(3 * count + 50, np.int64)
    lengths[1::3][:count] = 2049 + np.arange(count) % 552
    lengths[0::3] = np.arange(len(lengths[0::3])) % 70
    rowptr = np.concatenate([[0], np.cumsum(lengths)])
    col = np.concatenate([np.sort(order()[(977 * i) % 100000:][:c]) for i, c in enumerate(lengths)])
    return csr(len(lengths), N, rowptr, col, I.random_values(len(col), dt, 92, kind="signed"), dt)


@pytest.mark.parametrize("count,dt", [(400, "f64"), (400, "i32"), (400, "bool"), (2, "f32")])
def test_long_rows_of_a_wide_matrix(count, dt):
    from paper_1109_3739_gb300 import hspgemm as h
    A = long_rows(count, dt)
    Iv = np.concatenate([I.random_unique_sequence(A.m, A.m, 93), [1, 1]]).astype(np.int32)
    d = h.DeviceCSR.from_host(A)
    for Jv in (order(), order()[: N // 3]):
        ref = oracle.spref(A, Iv, Jv)
        assert_bitexact(h.spref(d, Iv, Jv).to_host(), ref, f"{count} {dt}")
        assert_bitexact(h.spref(d, Iv, Jv, validate=True).to_host(), ref, f"{count} {dt}, checked")


def test_long_rows_of_a_wide_matrix_when_allocations_fail():
    """Every allocation of the radix route in turn: HS_ENOMEM with nothing left, or the bitmaps take over."""
    import ctypes

    import torch
    from paper_1109_3739_gb300 import hspgemm as h
    from tests.test_gpu_failure import _host, _sweep
    A = long_rows(400, "i32")
    d, Jv = h.DeviceCSR.from_host(A), order()
    Iv = np.arange(A.m, dtype=np.int32)[::-1].copy()
    dI, dJ, a, ref = torch.from_numpy(Iv).cuda(), torch.from_numpy(Jv).cuda(), d.desc(), oracle.spref(A, Iv, Jv)

    def run(al):
        c = h.hs_mat()
        st = h.library().hs_spref(ctypes.byref(a), dI.data_ptr(), len(Iv), dJ.data_ptr(), len(Jv), ctypes.byref(c),
                                  ctypes.byref(al.struct), None, 0)
        return st, c

    allocations, nomem, taken_over = _sweep(h, run, lambda c, al: assert_bitexact(_host(h, c, al), ref, "after a failure"))
    assert allocations >= 12 and nomem >= 3 and taken_over >= 5
