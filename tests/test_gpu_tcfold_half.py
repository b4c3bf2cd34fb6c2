"""Tensor-core direct sum whose digits are too large for one accumulator drain per
slot: constant sources with every digit 127 on full chunks of 128, alone and
beside Gaussian columns (the drain is chosen for the launch).  The column sums
stay exact, so the bounds are those of the other sizes: 1e-13 of a column's
largest entry, and for KD digit classes N (KD + 1) 2^(2 - 8 KD) max|T| max|v|,
all that the dropped digits can add up to."""
import numpy as np
import pytest
import torch

import hif_inputs as hi
from oracle import kernels

pytestmark = pytest.mark.gpu


def largest_chunk_sum(v, n):
    """max over lines and chunks of 128 of sum |digit|, digits 0..6."""
    u = np.ldexp(v, -(int(np.floor(np.log2(np.abs(v).max()))) + 2)).reshape(n, n)
    tot = np.zeros_like(u)
    for _ in range(7):
        d = np.rint(256.0 * u)
        u = 256.0 * u - d
        tot += np.abs(d)
    return max(tot[:, c:c + 128].sum(axis=1).max() for c in range(0, n, 128))


@pytest.mark.parametrize("n,nrhs,classes", [(128, 1, 8), (128, 8, 8), (256, 1, 8), (256, 3, 8), (160, 8, 8), (128, 1, 6),
                                            (256, 8, 5)])
def test_saturated_digits_match_oracle(n, nrhs, classes):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, 2)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), 0, 1e-2, precision="fp32")
    op = kernels.Operator(pb.points, pb.weights, pb.a, pb.b, pb.c, 0)
    x = np.asfortranarray(hi.gaussian_rhs(pb.N, nrhs, 60 + n)).reshape(pb.N, nrhs, order="F")
    x[:, 0] = sum(127.0 * 256.0 ** -(k + 1) for k in range(7)) / pb.weights
    assert largest_chunk_sum(pb.weights * pb.c * x[:, 0], n) > 65536
    rows = np.random.default_rng(n).choice(pb.N, 96, replace=False)
    A = op.entries(rows, np.arange(pb.N))
    ref = A @ x                                          # A is symmetric: b = c = 1
    for trans in (False, True):
        y = fac.matvec(T(x), trans=trans, classes=classes).cpu().numpy()[rows]
        if classes == 8:
            bound = 1e-13 * np.abs(ref).max(axis=0)
        else:
            v = np.abs(pb.weights[:, None] * x).max(axis=0)
            A[np.arange(96), rows] -= 1.0                # a = 1 is not in the table
            G = np.abs(A).max() / pb.weights[0]
            bound = pb.N * (classes + 1) * 2.0 ** (2 - 8 * classes) * G * v + 1e-13 * np.abs(ref).max(axis=0)
        assert np.all(np.abs(y - ref).max(axis=0) <= bound)
    fac.close()
