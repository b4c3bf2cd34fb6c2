"""The rows per fold chunk of a 32-bit factorization, fixed or picked by timing:
another order of the folds' sums, so other roundings of F, and the same refined
solution to what its residual of 1e-10 leaves open."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 100])
def test_autotuned_folds_refine_to_the_same_solution(n):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, 2, smooth_seed=1002)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    f = T(hi.gaussian_rhs(pb.N, 2, 9))
    out = []
    for autotune in (False, True):
        fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), 0, 1e-6, precision="fp32",
                              autotune=autotune)
        u, its, rel = fac.solve_refined(f, tol=1e-10)
        assert rel <= 1e-10 and its <= 4
        out.append(u)
        fac.close()
    # a second-kind operator, condition below 10: two residuals of 1e-10
    assert float((out[0] - out[1]).norm()) <= 2e-9 * float(out[0].norm())
