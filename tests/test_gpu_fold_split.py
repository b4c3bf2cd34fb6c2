"""Folds of a box's proxy matrix by one CTA and by clusters of 2, 4 and 8 whose
R factors are folded together: R is that of the same matrix up to rounding and
row signs, so the skeleton sets are the same and the operators agree to 1e-10,
the bound of the other comparisons of two ways to the same R."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,general,precision", [(16, 2, False, "fp64"), (50, 2, True, "fp64"),
                                                     (64, 2, False, "fp64"), (64, 2, False, "fp32"),
                                                     (12, 3, True, "fp64")])
def test_split_folds_match(monkeypatch, n, dim, general, precision):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, dim, smooth_seed=21 + n)
    c = 1.0 + 0.5 * hi.smooth_field(pb.points, 97) if general else pb.c
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    x = T(hi.gaussian_rhs(pb.N, 2, n))
    ref = None
    for split in ("1", "2", "4", "8"):
        monkeypatch.setenv("HIF_FOLD_SPLIT", split)
        fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(c), pb.kernel_id, 1e-6,
                              proxy_dirs=pb.proxy if dim == 3 else None, precision=precision)
        if precision == "fp32":
            u, _, rel = fac.solve_refined(x, tol=1e-10)
            assert rel <= 1e-10
            got = ([], [u])
        else:
            subs = fac.stats()["sublevels"]
            got = ([fac.eliminated_dofs(s) for s in range(subs + 1)], [fac.solve(x), fac.apply(x)])
        fac.close()
        if ref is None:
            ref = got
            continue
        for p, q in zip(got[0], ref[0]):
            assert np.array_equal(p, q)
        for p, q in zip(got[1], ref[1]):
            assert float((p - q).abs().max()) <= (1e-10 if precision == "fp64" else 1e-8) * float(q.abs().max())
