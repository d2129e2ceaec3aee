"""The kernels that take rows by their size, at the edges of their ranges: rows
sorted instead of hashed, bitmaps of all columns, and rows whose bitmap is
handed from the symbolic to the numeric pass.  Integer sums, minima and
structures: every comparison is exact."""
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


def operands(n, rows, dt, seed):
    """A and B, a row of A * B for each list of spans (first, last): an entry of A and a row of B for each span,
    which holds that stretch of one random order of the columns.  A row's products all differ in column, except
    where its spans overlap."""
    order = np.argsort(I.draws(seed, 3, 0, n), kind="stable")
    pieces, arows = [], []
    for spans in rows:
        take = []
        for a, b in spans:
            take.append(len(pieces))
            pieces.append(np.sort(order[a:b]))
        arows.append(np.array(take, np.int64))
    bptr = np.concatenate([[0], np.cumsum([len(p) for p in pieces])])
    aptr = np.concatenate([[0], np.cumsum([len(t) for t in arows])])
    B = csr(len(pieces), n, bptr, np.concatenate(pieces), I.random_values(int(bptr[-1]), dt, seed, kind="signed"), dt)
    A = csr(len(arows), len(pieces), aptr, np.concatenate(arows), I.random_values(int(aptr[-1]), dt, seed + 1, kind="signed"),
            dt)
    return A, B


def product(A, B, what, sr):
    h = H()
    ref = oracle.spgemm(sr, A, B)
    dA, dB = h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)
    assert_bitexact(h.spgemm(sr, dA, dB).to_host(), ref, what)
    P = h.Plan(sr, dA, dB)
    if P.C.val is not None:
        P.C.val.zero_()
    P.execute()
    assert_bitexact(P.C.to_host(), ref, f"{what}, plan")


def split(f, parts, start=0):
    cuts = np.linspace(0, f, parts + 1).astype(int) + start
    return [(int(a), int(b)) for a, b in zip(cuts[:-1], cuts[1:])]


KINDS = [("plus_times", "i64"), ("min_plus", "f32"), ("or_and", "bool")]


@pytest.mark.parametrize("sr,dt", KINDS)
def test_rows_counted_by_a_sort(sr, dt):
    """33 to 512 products over too many columns for a bitmap: up to 64 are sorted, more are hashed."""
    rows = []
    for f in (33, 63, 64, 65, 128, 512):
        for dup in (0, 1, f // 2, f - 1):
            base = split(f - dup, min(3, f - dup))
            rows.append(base + ([(0, min(dup, f - dup))] if dup else []) + ([(0, 1)] * (dup - min(dup, f - dup))))
    product(*operands(300001, rows, dt, 5), f"sorted count {sr}", sr)


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1])
def test_structure_by_bitmap(n):
    """Structure-only rows of 500 to 9000 outputs; over 4096 they are not staged."""
    rows = [split(c, p) + [(0, min(c, d))] for c in (500, 1025, 2049, 4095, 4096, 4097, 9000) for p, d in ((3, 1), (300, 400))]
    product(*operands(n, rows, "bool", 6), f"{n} columns", "or_and")


@pytest.mark.parametrize("n", [(1 << 19) - 1, 1 << 19, (1 << 19) + 1])
def test_many_rows_of_the_symbolic_bitmap(n):
    """Enough rows of more than 4096 products for two CTAs an SM, where half a bitmap holds B's columns."""
    A, B = operands(n, [split(4100 + 40 * i, 3 + i, 17 * i) + [(17 * i, 17 * i + 9)] for i in range(7)], "i64", 7)
    many = 100  # the seven rows over and over
    A = csr(7 * many, B.m, np.concatenate([[0], np.cumsum(np.tile(np.diff(A.rowptr), many))]),
            np.tile(A.col, many), np.tile(A.val, many), "i64")
    product(A, B, f"{n} columns", "plus_times")


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "f32"), ("or_and", "bool")])
@pytest.mark.parametrize("n", [70001, (1 << 17) + 4097, 300001])
def test_rows_that_leave_their_bitmap(n, sr, dt):
    """Rows of the units on both sides of an output for every second word of the bitmap, some with fewer products
    than the bitmap has words, and parts of one and of many segments."""
    half = (n + 63) // 64
    words = (n + 31) // 32
    cs = sorted({max(4097, half - 1), max(4097, half), max(4097, half + 1), max(4097, words), 6000, 20011, n // 2, n})
    rows = [split(c, 5) + [(1, 40)] * 3 for c in cs]
    product(*operands(n, rows, dt, 8), f"{n} columns {sr}", sr)


@pytest.mark.parametrize("sr,dt", [("plus_times", "i64"), ("min_plus", "i32"), ("min_plus", "f32"), ("or_and", "bool")])
def test_rows_sorted_as_they_are(sr, dt):
    """1025 to 4096 outputs with few repeated columns, on both sides of the share and of the capacity, the repeats
    spread over the row or all of one column, in one round of entries and in several."""
    rows = []
    for c in (1025, 1820, 2047, 2048, 2049, 3640, 4000, 4095):
        for dup in (0, 1, c // 8 - 1, c // 8, c // 8 + 1, 2048 - c, 2049 - c, 4096 - c, 4097 - c):
            if not 0 <= dup <= c or c + dup > 4097:
                continue
            rows.append(split(c, 3) + ([(0, dup)] if dup else []))
            if dup and dup < 600:
                rows.append(split(c, 290) + [(7, 8)] * dup)
    product(*operands(600001, rows, dt, 9), f"few repeats {sr} {dt}", sr)


@pytest.mark.parametrize("sr,dt", KINDS)
def test_hub_rows_beside_short_ones(sr, dt):
    """Rows of thousands of entries of A (few outputs, and units whose segments are laid out by blocks), B rows of
    thousands of entries, short rows of every bin, in one product and in a captured replay of its plan."""
    import torch
    n = 100003
    rows = [split(4500, 4500) + [(0, 3)] * 600, split(9000, 1500) + [(5, 2600)], split(20000, 3) + [(0, 2049)] * 4,
            split(4096, 4096), split(4097, 4097)]
    for f in (0, 1, 20, 32, 33, 100, 200, 400, 700, 1500, 3000, 4500, 9000):
        rows += [split(f, min(f, 4)) + ([(0, f // 2)] if f > 1 else [])] * 3 if f else [[]]
    A, B = operands(n, rows, dt, 10)
    product(A, B, f"hubs {sr}", sr)
    if dt == "bool":
        return
    h = H()
    P = h.Plan(sr, h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B))
    P.execute()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        P.execute()
    P.C.val.zero_()
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert_bitexact(P.C.to_host(), oracle.spgemm(sr, A, B), f"hubs {sr}, captured")


def test_millions_of_empty_rows():
    """More rows than one pass of the scan's tiles, almost all empty, with long gaps inside a tile of entries."""
    m, k, n = 8_500_001, 64, 1000
    at = np.unique(np.concatenate([np.arange(0, 40), [20000, 20001, 60000, 4_000_000], m - 1 - np.arange(3),
                                   (I.draws(4, 9, 0, 500) % np.uint64(m)).astype(np.int64)]))
    lens = 1 + np.arange(len(at)) % 40
    rowptr = np.zeros(m + 1, np.int64)
    rowptr[at + 1] = lens
    rowptr = np.cumsum(rowptr)
    cols = np.concatenate([np.sort(I.random_unique_sequence(k, int(c), 70 + i)) for i, c in enumerate(lens)])
    A = csr(m, k, rowptr, cols, I.random_values(len(cols), "i64", 11, kind="signed"), "i64")
    B = csr(k, n, np.arange(k + 1) * 5, np.concatenate([np.sort(I.random_unique_sequence(n, 5, 80 + i)) for i in range(k)]),
            I.random_values(5 * k, "i64", 12, kind="signed"), "i64")
    product(A, B, "empty rows", "plus_times")


@pytest.mark.parametrize("c,dup", [(1500, 0), (1500, 100), (3500, 0), (3500, 300)])
def test_sorted_rows_treat_special_values_as_the_table_does(c, dup):
    """(min,+) with infinities and NaNs: a row that is sorted as it is against the same row in the table (the
    unsorted output keeps it)."""
    h = H()
    A, B = operands(600001, [split(c, 3) + ([(0, dup)] if dup else [])] * 3, "f32", 13)
    B.val[::7], B.val[1::11], B.val[2::13], B.val[3::17] = np.nan, np.inf, -np.inf, -0.0
    A.val[1] = np.inf
    dA, dB = h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)
    got = h.spgemm("min_plus", dA, dB).to_host()
    raw = h.spgemm("min_plus", dA, dB, sorted_rows=False).to_host()
    assert np.array_equal(got.rowptr, raw.rowptr)
    for a, b in zip(got.rowptr[:-1], got.rowptr[1:]):
        order = np.argsort(raw.col[a:b])
        assert np.array_equal(got.col[a:b], raw.col[a:b][order])
        assert np.array_equal(got.val[a:b], raw.val[a:b][order], equal_nan=True)


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("c,dup", [(1500, 0), (1500, 100), (3500, 0), (3500, 300)])
def test_sorted_rows_add_to_the_identity_as_the_table_does(c, dup, dt):
    """(+,x) with products of -0: a sum starts from 0 in a row that is sorted as it is, as in the table (the unsorted
    output keeps it), so a lone -0 becomes +0 on both ways, bit for bit."""
    h = H()
    A, B = operands(600001, [split(c, 3) + ([(0, dup)] if dup else [])] * 3, dt, 14)
    A.val[:] = 1
    B.val[::2], B.val[1::7] = -0.0, np.nan
    dA, dB = h.DeviceCSR.from_host(A), h.DeviceCSR.from_host(B)
    got = h.spgemm("plus_times", dA, dB).to_host()
    raw = h.spgemm("plus_times", dA, dB, sorted_rows=False).to_host()
    assert np.array_equal(got.rowptr, raw.rowptr)
    zeros = 0
    for a, b in zip(got.rowptr[:-1], got.rowptr[1:]):
        order = np.argsort(raw.col[a:b])
        x, y = got.val[a:b], raw.val[a:b][order]
        assert np.array_equal(got.col[a:b], raw.col[a:b][order])
        nan = np.isnan(x)
        assert np.array_equal(nan, np.isnan(y))
        # (sums of several terms are formed in an unspecified order: at most 2 here, so the same either way)
        assert np.array_equal(np.signbit(x[~nan]), np.signbit(y[~nan])) and np.array_equal(x[~nan], y[~nan])
        zeros += np.count_nonzero(x[~nan] == 0)
        assert not np.signbit(x[~nan][x[~nan] == 0]).any()
    assert zeros > c // 4
