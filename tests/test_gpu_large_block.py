"""One block of 6,241 rows in 64 bits: its first two LU panels are too long for a
cluster's shared memory and take the one-CTA panel kernel, the others the
cluster one.  The factored operator is A itself: apply against the direct sum,
solve against the right-hand side, to N 2^-53 times a growth of a few hundred."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


def test_block_above_the_cluster_panels():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(79, 2, smooth_seed=7)
    c = 1.0 + 0.5 * hi.smooth_field(pb.points, 99)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(c), 0, 1e-6, occupancy=pb.N + 1)
    assert fac.stats()["top_size"] == pb.N == 6241
    x = T(hi.gaussian_rhs(pb.N, 3, 5))
    tol = pb.N * 2.0 ** -53 * 300
    for f, g, trans in ((fac.apply, fac.solve, False), (fac.apply_transpose, fac.solve_transpose, True)):
        y = fac.matvec(x, trans=trans)
        assert float((f(x) - y).norm()) <= tol * float(y.norm())
        assert float((fac.matvec(g(x), trans=trans) - x).norm()) <= tol * float(x.norm())
    fac.close()
