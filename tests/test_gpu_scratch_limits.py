"""A small operation is served by an allocator that hands out small blocks only."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import oracle
from paper_1109_3739_gb300 import inputs as I
from tests.helpers import assert_bitexact

pytestmark = pytest.mark.gpu
LIMIT = 300 << 10  # bytes: more than any array of the operations below


def H():
    from paper_1109_3739_gb300 import hspgemm
    return hspgemm


class SmallBlocks:
    """Allocator callbacks (torch memory) that refuse every block of more than LIMIT bytes."""

    def __init__(self, h):
        import torch
        self.base = h._TorchAlloc(torch.device("cuda"))
        self._a = h.ALLOC_FN(lambda n, st, ctx: None if n > LIMIT else self.base._alloc(n, st, ctx))
        self.struct = h.hs_allocator(self._a, self.base._f, None)


def result(h, c, al):
    import torch
    live, n = al.base.live, int(c.nnz)
    d = h.DeviceCSR(c.m, c.n, live[c.ptr].view(torch.int64)[:c.m + 1], live[c.idx].view(torch.int32)[:n],
                    live[c.val].view(torch.int64)[:n], "i64").to_host()
    h.library().hs_mat_free(ctypes.byref(c), ctypes.byref(al.struct), None)
    torch.cuda.synchronize()
    assert not al.base.live
    return d


@pytest.mark.parametrize("op", ["spgemm", "spref", "spref, repeated", "spasgn", "sparse"])
def test_small_operations_need_small_blocks_only(op):
    import torch
    h = H()
    L = h.library()
    al, c = SmallBlocks(h), h.hs_mat()
    A = I.er_matrix(1000, 1000, 4, seed=71, dtype="i64")
    dA = h.DeviceCSR.from_host(A)
    a, ref, al_ = dA.desc(), ctypes.byref, ctypes.byref(al.struct)
    Iv, Jv = I.random_unique_sequence(1000, 300, 72), I.random_unique_sequence(1000, 400, 73)
    if op == "spref, repeated":
        Jv = np.concatenate([Jv, Jv[:1]])
    dI, dJ = torch.from_numpy(Iv.astype(np.int32)).cuda(), torch.from_numpy(Jv.astype(np.int32)).cuda()
    if op == "spgemm":
        st = L.hs_spgemm(h.SEMIRING["plus_times"], ref(a), ref(a), ref(c), al_, None, 0)
        want = oracle.spgemm("plus_times", A, A)
    elif op.startswith("spref"):
        st = L.hs_spref(ref(a), dI.data_ptr(), len(Iv), dJ.data_ptr(), len(Jv), ref(c), al_, None, 0)
        want = oracle.spref(A, Iv, Jv)
    elif op == "spasgn":
        B = I.er_matrix(300, 400, 3, seed=74, dtype="i64")
        dB = h.DeviceCSR.from_host(B)
        b = dB.desc()
        st = L.hs_spasgn(ref(a), dI.data_ptr(), 300, dJ.data_ptr(), 400, ref(b), 0, 0, ref(c), al_, None, 0)
        want = oracle.spasgn(A, Iv, Jv, B)
    else:
        ti, tj, tv = I.rmat_tuples(10, 8, seed=75, dtype="i64", kind="signed")
        di, dj, dv = (torch.from_numpy(x).cuda() for x in (ti, tj, tv))
        st = L.hs_sparse(di.data_ptr(), dj.data_ptr(), dv.data_ptr(), len(ti), 1024, 1024, h.DTYPE["i64"],
                         h.SEMIRING["plus_times"], ref(c), al_, None, 0)
        want = oracle.sparse(ti, tj, tv, 1024, 1024, "plus_times", dtype="i64")
    torch.cuda.synchronize()
    assert st == 0, h.STATUS[st]
    assert_bitexact(result(h, c, al), want, op)
