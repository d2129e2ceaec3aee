"""The symbolic pass's sets at the widths where a bitmap of B's columns stops
fitting the hash table's room (32 columns a slot: 2^15, 2^16 and 2^18 columns
for rows of up to 512, 1024 and 4096 products), and rows of few products taken
several at a time.  Sums of small integers: every comparison is exact."""
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


def product(A, B, what, sr="plus_times"):
    h = H()
    got = h.spgemm(sr, h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)).to_host()
    assert_bitexact(got, oracle.spgemm(sr, A, B), what)


def wide_b(n, k, per_row, seed, dtype="i64"):
    """k rows of `per_row` columns, the first and last column among them, some shared."""
    cols = []
    for i in range(k):
        c = I.random_sequence(n, per_row, seed + i)
        c[:4] = [0, n - 1, n // 2, min(31 + i, n - 1)]
        cols.append(np.unique(c))
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])])
    col = np.concatenate(cols)
    return csr(k, n, rowptr, col, I.random_values(len(col), dtype, seed, kind="signed"), dtype)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 32767, 32768, 32769, 65536, 65537, 262144, 262145])
def test_widths(n):
    k = 40
    B = wide_b(n, k, 100, 3)
    # rows of 1, 5, 9 and 40 entries: about 100, 500, 900 and 4000 products
    cols = [np.arange(e) % k if e == k else np.sort(I.random_unique_sequence(k, e, 50 + e)) for e in (1, 5, 9, 40) * 9]
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])])
    A = csr(len(cols), k, rowptr, np.concatenate(cols), I.random_values(rowptr[-1], "i64", 7, kind="signed"), "i64")
    product(A, B, f"{n} columns")
    h = H()
    C, offs = h.spgemm_batched("plus_times", [h.DeviceCSR.from_host(A)] * 2, [h.DeviceCSR.from_host(B)] * 2)
    P = h.BatchPlan("plus_times", [h.DeviceCSR.from_host(A)] * 2, [h.DeviceCSR.from_host(B)] * 2)
    P.execute()
    D, _ = P.result()
    ref = oracle.spgemm("plus_times", A, B)
    for got in (C, D):
        one = h.csr_rows(got, int(offs[1]), int(offs[2])).to_host()
        assert_bitexact(one, ref, f"{n} columns, batched")


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32"), ("or_and", "bool")])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_tiny_rows_together(sr, dt, seed):
    """Rows of 0 to 32 products in every mixture: empty entries, one long B row, shared columns, more than 32
    entries of A for a few products."""
    n, k, m = 50, 400, 3000
    u = I.draws(seed, 40, 0, k)
    blen = np.where(u % 7 == 0, 0, (u >> np.uint64(8)) % 5).astype(np.int64)
    blen[:3] = [32, 31, 17]
    cols = [np.sort(I.random_unique_sequence(n, int(c), 60 + i)) for i, c in enumerate(blen)]
    B = csr(k, n, np.concatenate([[0], np.cumsum(blen)]), np.concatenate(cols),
            I.random_values(int(blen.sum()), dt, seed, kind="signed"), dt)
    rows, empty = [], np.nonzero(blen == 0)[0]
    for i in range(m):
        w = I.draws(seed, 41, 64 * i, 64)
        pick = np.unique((w[: 1 + int(w[60] % (20 if i % 17 == 0 else 5))] % np.uint64(k)).astype(np.int64))
        pick = pick[np.cumsum(blen[pick]) <= 32]
        if i % 97 == 0:
            pick = np.unique(np.concatenate([pick, empty]))  # more than 32 entries, most of them idle
        rows.append(pick if i % 11 else pick[:0])
    assert np.mean([blen[r].sum() for r in rows if blen[r].sum()]) < 8
    for copies in (1, 40):  # a short list of such rows (one to a warp) and a long one (several to a warp)
        long = rows * copies
        rowptr = np.concatenate([[0], np.cumsum([len(r) for r in long])])
        vals = I.random_values(int(rowptr[-1]), dt, seed + 9, kind="signed")
        product(csr(m * copies, k, rowptr, np.concatenate(long), vals, dt), B, f"tiny {sr} x{copies}", sr)
