"""Eliminations in the shared memory of a cluster of CTAs against the one-CTA
kernel: HIF_ELIM_MID moves the line between the two.  Same pivots and the same
arithmetic up to the order of the sums, so the factored operators agree to
1e-12 as the existing comparisons of elimination paths do (FP32: 1e-4)."""
import numpy as np
import pytest
import torch

import hif_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,general,precision,alpha", [
    (17, 2, False, "fp64", None), (33, 2, True, "fp64", None), (64, 2, False, "fp64", None),
    (64, 2, True, "fp32", None), (12, 3, False, "fp64", None), (40, 2, False, "fp64", "1e9")])
def test_cluster_elimination_matches_one_cta(monkeypatch, n, dim, general, precision, alpha):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, dim, smooth_seed=11 + n)
    c = 1.0 + 0.5 * hi.smooth_field(pb.points, 98) if general else pb.c
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    if alpha:                                   # every LDL box falls back to LU
        monkeypatch.setenv("HIF_LDL_TEST_ALPHA", alpha)
    x = T(hi.gaussian_rhs(pb.N, 3, n))
    out, stats = [], []
    for line in ("0", "100000"):
        monkeypatch.setenv("HIF_ELIM_MID", line)
        fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(c), pb.kernel_id, 1e-6,
                              proxy_dirs=pb.proxy if dim == 3 else None, precision=precision)
        out.append([getattr(fac, op)(x) for op in ("solve", "apply", "solve_transpose", "apply_transpose")])
        stats.append(fac.stats())
        fac.close()
    for key in ("ldl_boxes", "ldl_fallbacks", "factor_bytes", "top_size"):
        assert stats[0][key] == stats[1][key]
    assert (stats[0]["ldl_fallbacks"] > 0) == bool(alpha)
    tol = 1e-12 if precision == "fp64" else 1e-4
    for p, q in zip(*out):
        assert float((p - q).abs().max()) <= tol * float(q.abs().max())


@pytest.mark.parametrize("n,dim,precision", [(64, 2, "fp64"), (40, 2, "fp32"), (12, 3, "fp64")])
def test_panel_elimination_matches_cluster(monkeypatch, n, dim, precision):
    # LU blocks above HIF_ELIM_CLUSTER_R rows by panels of 32 columns: blocks of
    # one panel and of several, ragged last panels, the top block
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(n, dim, smooth_seed=41 + n)
    c = 1.0 + 0.5 * hi.smooth_field(pb.points, 96)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    x = T(hi.gaussian_rhs(pb.N, 3, n))
    monkeypatch.setenv("HIF_ELIM_MID", "0")
    monkeypatch.setenv("HIF_BIG_ELIM", "24")
    out = []
    for line in ("100000", "33", "8"):
        monkeypatch.setenv("HIF_ELIM_CLUSTER_R", line)
        fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(c), pb.kernel_id, 1e-6,
                              proxy_dirs=pb.proxy if dim == 3 else None, precision=precision)
        out.append([getattr(fac, op)(x) for op in ("solve", "apply", "solve_transpose", "apply_transpose")])
        fac.close()
    tol = 1e-12 if precision == "fp64" else 1e-4
    for other in out[1:]:
        for p, q in zip(other, out[0]):
            assert float((p - q).abs().max()) <= tol * float(q.abs().max())


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("seed", [1004, 1007, 1010])
def test_fp32_solve_then_apply_returns_the_vector(symmetric, seed):
    """F (F^{-1} f) = f up to the rounding of the FP32 factors alone.  Solve
    and apply pass ~16 (sub)levels each; with one unit of rounding (2^-24 of
    the vector) per level and pass the sum is at most 32 of them.  Triangular
    inverses that amplify their own rounding miss this."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    pb = hi.volume_problem(512, 2, smooth_seed=seed, rhs_seed=1003, nrhs=2)
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device="cuda:0")
    f = T(pb.f.T).t()
    fac = P.Factorization(T(pb.points), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), pb.kernel_id, 1e-6,
                          precision="fp32", symmetric=symmetric, autotune=False)
    err = float((fac.apply(fac.solve(f)) - f).norm() / f.norm())
    fac.close()
    assert err <= 32 * 2.0 ** -24
