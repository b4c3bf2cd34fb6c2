"""Ties of the batched interpolative decompositions.  The pivot is the remaining
column of largest norm, norms summed anew after every step, the lowest index
among equals: after a pivot along e_0 the columns [x, v] and [y, v] are equal
bit for bit and the lower one is next, whatever x and y.  Norms carried from
step to step by subtraction ((x^2 + |v|^2) - x^2) differ in their last bits."""
import numpy as np
import pytest
import torch

from oracle import idqr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,entry", [(2, "alloc"), (7, "alloc"), (40, "alloc"), (7, "noalloc"), (40, "noalloc")])
def test_equal_columns_go_by_index(m, entry):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_2666_gb300 import hif
    rng = np.random.default_rng(m)
    count, n = 200, 4
    mats = np.zeros((count, n, m))                       # column-major m x n each
    mats[:, 0, 0] = 100.0
    mats[:, 1:, 0] = rng.permuted(np.tile([3.0, 2.0, 1.0], (count, 1)), axis=1)
    mats[:, 1:, 1:] = rng.standard_normal((count, 1, m - 1))
    i32 = lambda v: torch.as_tensor(np.full(count, v, dtype=np.int32) if np.isscalar(v) else v)
    i64 = lambda step: torch.arange(count, dtype=torch.int64) * step
    args = [torch.as_tensor(mats.reshape(-1)), i64(m * n), i32(m), i32(n), torch.full((count,), 1e-10, dtype=torch.float64),
            torch.zeros(count, dtype=torch.int32), torch.zeros(count * n, dtype=torch.int32), i64(n),
            torch.zeros(count * n * n, dtype=torch.float64), i64(n * n)]
    if entry == "alloc":
        args = [a.numpy() for a in args]
        hif.hif_id_batched(*args)
    else:
        args = [a.cuda() for a in args]
        assert hif.hif_id_batched_noalloc(*args) == hif.HIF_OK
        args = [a.cpu().numpy() for a in args]
    k, perm = args[5], args[6].reshape(count, n)
    for i in range(count):
        sk, rd, _ = idqr.interp_decomp(mats[i].T, 1e-10)
        assert list(sk) == [0, 1] and k[i] == 2
        assert list(perm[i]) == list(sk) + list(rd)
