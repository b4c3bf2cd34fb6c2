"""LDL blocks in the shared memory of a cluster: the remaining block is reduced
symmetrically, entry by entry as in the one-CTA kernel."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,precision", [(12, "fp64"), (16, "fp64"), (20, "fp64"), (20, "fp32")])
def test_symmetric_block_is_the_one_cta_block_to_the_bit(monkeypatch, n, precision):
    # one box of n^2 rows, LDL: same pivots, and every entry reduced by
    # (c_i c_q) / d in the same order, so that L and D agree exactly; apply
    # multiplies by them alone
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, 2, smooth_seed=70 + n)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    x = T(hi.gaussian_rhs(pb.N, 2, n))
    out = []
    for line in ("0", "100000"):
        monkeypatch.setenv("HIF_ELIM_MID", line)
        fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), 0, 1e-6, occupancy=512,
                              precision=precision)
        st = fac.stats()
        assert st["top_size"] == pb.N and st["ldl_boxes"] == 1 and st["ldl_fallbacks"] == 0
        out.append(fac.apply(x))
        fac.close()
    assert torch.equal(*out)
