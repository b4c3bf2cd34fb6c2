"""A block of right-hand sides against its columns: the order of every sum of a
sweep depends on the box and the launch shape of its sublevel only, so the
columns agree to the bit whatever the number that a CTA holds (1, 2, 4, 8)."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,general,precision", [
    (17, 2, False, "fp64"), (40, 2, True, "fp64"), (72, 2, False, "fp64"), (72, 2, True, "fp32"), (72, 2, False, "fp32"),
    (12, 3, True, "fp64")])
def test_block_equals_columns_to_the_bit(n, dim, general, precision):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, dim, smooth_seed=3 + n)
    c = 1.0 + 0.5 * hi.smooth_field(pb.points, 99) if general else pb.c
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(c), pb.kernel_id, 1e-6,
                          proxy_dirs=pb.proxy if dim == 3 else None, precision=precision)
    x = T(hi.gaussian_rhs(pb.N, 17, n))
    for op in ("solve", "solve_transpose", "apply", "apply_transpose"):
        f = getattr(fac, op)
        cols = torch.stack([f(x[:, q].contiguous()) for q in range(17)], dim=1)
        for nrhs in (2, 3, 4, 5, 8, 9, 17):
            assert torch.equal(f(x[:, :nrhs].t().contiguous().t()), cols[:, :nrhs]), (op, nrhs)
    fac.close()
