"""More right-hand sides than the second dimension of a grid has CTAs for
(65,535 groups of up to 8): solved in several launches, column by column the
same to the bit."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["solve", "apply_transpose"])
def test_more_right_hand_sides_than_a_grid_takes(op):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(8, 2, smooth_seed=3)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), 0, 1e-6, precision="fp32")
    nrhs = 8 * 65535 + 9
    x = T(hi.gaussian_rhs(pb.N, 16, 1))[:, torch.arange(nrhs, device="cuda:0") % 16].t().contiguous().t()
    y = getattr(fac, op)(x)
    few = getattr(fac, op)(x[:, :16].t().contiguous().t())
    for q in range(16):
        assert torch.equal(y[:, q::16], few[:, q:q + 1].expand(-1, y[:, q::16].shape[1]))
    fac.close()
