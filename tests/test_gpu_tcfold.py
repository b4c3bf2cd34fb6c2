"""Tensor-core direct sum at the edges of its tiles: 2^k right-hand sides and
32 / 2^k target lines per tile, sizes around multiples of the lines and of the
128-wide chunks, and coherent sources whose mirror pairs have the largest
digits.  Same bound as the other sizes (1e-13 of a column's largest entry:
the sum is exact up to digits below 2^-55 and its FP64 combination)."""
import numpy as np
import pytest
import torch

import hif_inputs as hi
from oracle import kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,nrhs,coherent", [
    (4, 2, 1, False), (31, 2, 1, False), (33, 2, 1, True), (65, 2, 2, False), (97, 2, 4, True), (129, 2, 5, False),
    (128, 2, 12, False), (9, 3, 1, True), (17, 3, 3, False)])
def test_folded_sum_matches_oracle(n, dim, nrhs, coherent):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, dim, smooth_seed=5 + n)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), pb.kernel_id, 1e-2,
                          proxy_dirs=pb.proxy if dim == 3 else None, precision="fp32")
    op = kernels.Operator(pb.points, pb.weights, pb.a, pb.b, pb.c, pb.kernel_id)
    x = hi.gaussian_rhs(pb.N, nrhs, 60 + n)
    if coherent:
        x = np.asfortranarray(np.where(np.abs(x) < 10.0, 0.4999 * (-1.0) ** np.arange(nrhs), x))
    for trans in (False, True):
        y = fac.matvec(T(x), trans=trans).cpu().numpy()
        ref = op.matvec(x, trans=trans)
        assert np.all(np.abs(y - ref).max(axis=0) <= 1e-13 * np.abs(ref).max(axis=0))
    fac.close()
