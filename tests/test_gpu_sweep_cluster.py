"""The sweeps with a box on one CTA and on clusters of CTAs: every operation
(LU and LDL boxes, FP64 and FP32), right-hand sides around the 1, 2, 4 and 8
that a CTA holds.  The order of the sums does not depend on the number of
right-hand sides, so a block equals its columns; 1e-13 (1e-5 in FP32) leaves
room for rounding only.  F F^{-1} = I as in the other sweep tests."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu
OPS = ("solve", "solve_transpose", "apply", "apply_transpose")


@pytest.mark.parametrize("n,general,precision", [(17, False, "fp64"), (40, True, "fp64"), (72, False, "fp64"),
                                                 (72, True, "fp32")])
def test_sweeps_block_equals_columns(n, general, precision):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, 2, smooth_seed=3 + n)
    c = 1.0 + 0.5 * hi.smooth_field(pb.points, 99) if general else pb.c
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(c), 0, 1e-6, precision=precision)
    tol = 1e-13 if precision == "fp64" else 1e-5
    x = T(hi.gaussian_rhs(pb.N, 17, n))
    for op in OPS:
        f = getattr(fac, op)
        cols = torch.stack([f(x[:, q].contiguous()) for q in range(17)], dim=1)
        for nrhs in (2, 3, 4, 5, 8, 9, 17):
            y = f(x[:, :nrhs].t().contiguous().t())
            assert float((y - cols[:, :nrhs]).abs().max()) <= tol * float(cols.abs().max())
    eye = fac.apply(fac.solve(x)) - x
    eyet = fac.apply_transpose(fac.solve_transpose(x)) - x
    assert max(float(eye.abs().max()), float(eyet.abs().max())) <= (1e-11 if precision == "fp64" else 1e-3)
    fac.close()
