"""Plans whose bins run on streams beside the caller's: captured by a thread
that has executed nothing before, executed on another stream while a capture
is open, on two streams of one thread, and on streams of either priority.
Integer sums: every comparison is exact."""
from __future__ import annotations

import threading

import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact

pytestmark = pytest.mark.gpu


def H():
    from paper_1109_3739_gb300 import hspgemm
    return hspgemm


class Case:
    """A product with rows in every kind of bin, as a plan with an output of its own."""

    def __init__(self, seed, stream=None):
        import torch
        h = H()
        self.A = I.rmat_matrix(14, 8, seed=seed, dtype="i64", kind="signed")
        d = h.DeviceCSR.from_host(self.A)
        torch.cuda.synchronize()
        self.plan, self.val = h.Plan("plus_times", d, d, stream=stream), d.val
        self.out = torch.zeros_like(self.plan.C.val)
        torch.cuda.synchronize()

    def execute(self, stream=None):
        self.plan.execute(self.val, self.val, self.out, stream=stream)

    def check(self, what):
        import torch
        torch.cuda.synchronize()
        self.plan.status()
        c = self.plan.C
        got = H().DeviceCSR(c.m, c.n, c.rowptr, c.col, self.out, c.dtype).to_host()
        assert_bitexact(got, oracle.spgemm("plus_times", self.A, self.A), what)
        self.out.zero_()
        torch.cuda.synchronize()


def test_capture_is_the_threads_first_execution():
    import torch
    a = Case(51)
    g = torch.cuda.CUDAGraph()
    failed = []

    def capture():
        try:
            with torch.cuda.graph(g, stream=torch.cuda.Stream()):
                a.execute()
        except Exception as e:  # (reported by the test's own thread)
            failed.append(e)

    t = threading.Thread(target=capture)
    t.start()
    t.join()
    assert not failed, failed
    for _ in range(2):
        g.replay()
        a.check("captured by a fresh thread")


def test_execution_beside_an_open_capture():
    """An eager execution on another stream neither joins nor breaks a capture, of another plan or of the same."""
    import torch
    a, b = Case(52), Case(53)
    g, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="relaxed"):
        a.execute()
        b.execute(stream=other)
        a.execute(stream=other)
        a.execute()
    b.check("eager execution of another plan")
    a.check("eager execution of the captured plan")
    g.replay()
    a.check("the capture")
    a.execute(stream=other)
    a.check("eager execution after the capture")


@pytest.mark.parametrize("priorities", [(0, 0), (-1, 0), (-1, -1)])
def test_two_plans_on_two_streams(priorities):
    import torch
    streams = [torch.cuda.Stream(priority=p) for p in priorities]
    cases = [Case(54 + i, s) for i, s in enumerate(streams)]
    for _ in range(5):
        for c, s in zip(cases, streams):
            c.execute(s)
    for c in cases:
        c.check("two streams")
    for c, s in zip(cases, reversed(streams)):
        c.execute(s)
    for c in cases:
        c.check("each other's stream")


def test_products_on_more_streams_than_side_streams():
    import torch
    h = H()
    A = I.rmat_matrix(13, 8, seed=56, dtype="i64", kind="signed")
    ref = oracle.spgemm("plus_times", A, A)
    d = h.DeviceCSR.from_host(A)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(priority=-(i % 2)) for i in range(12)]
    got = []
    for s in streams * 2:
        with torch.cuda.stream(s):
            got.append(h.spgemm("plus_times", d, d))
    torch.cuda.synchronize()
    for c in got:
        assert_bitexact(c.to_host(), ref, "one of many streams")
