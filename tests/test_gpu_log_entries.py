"""Direct sums off the grid.  The table-driven logarithm through a two-point
sum: y_0 = G(r) w, one rounding each for a few products around a logarithm
good to 1 ulp, so 8 ulp of the value (or of its r = e value near r = 1, where
the squared distance itself carries the error).  Scattered points in several
shares of the sources, and the Helmholtz sum on grids, in any order of the
points, and for points that only nearly form a grid."""
import numpy as np
import pytest
import torch

import hif_inputs as hi
from oracle import helmholtz, kernels

pytestmark = pytest.mark.gpu
T = lambda v, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(v), dtype=dt, device="cuda:0")


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    return P


@pytest.mark.parametrize("scale", [1e-75, 1e-9, 1.0, 3.7, 1e30])
def test_pair_sums_match_numpy(P, scale):
    # pairs far apart in one handle: sources other than point 0 are switched on one by one
    rng = np.random.default_rng(3)
    N = 300
    x = rng.uniform(-1.0, 1.0, (N, 2)) * scale
    x[0] = 0.0
    x[1] = [scale, 0.0]                                   # r = scale exactly
    x[2] = [scale * (1 + 2.0 ** -40), 0.0]
    w, one = np.full(N, scale * scale * 1e-4), np.ones(N)
    fac = P.Factorization(T(x), T(w), T(one), T(one), T(one), 0, 0.5, occupancy=512)
    got = fac.matvec(torch.eye(N, dtype=torch.float64, device="cuda:0")).cpu().numpy()
    fac.close()
    d = x[:, None, :].astype(np.longdouble) - x[None, :, :]
    with np.errstate(divide="ignore"):
        ref = -np.log((d * d).sum(axis=2)) / (4 * np.longdouble(np.pi)) * w[0]
    off = ~np.eye(N, dtype=bool)
    err = np.abs(got - ref)[off] / np.maximum(np.abs(ref[off]), w[0] / (4 * np.pi))
    assert float(err.max()) <= 8 * 2.0 ** -53


@pytest.mark.parametrize("n,dim,nrhs", [(20, 2, 1), (57, 2, 2), (70, 2, 5), (13, 3, 9)])
def test_scattered_sums_match_oracle(P, n, dim, nrhs):
    pb = hi.volume_problem(n, dim, smooth_seed=4)
    rng = np.random.default_rng(n)
    x = pb.points + rng.uniform(-0.2, 0.2, pb.points.shape) / n
    c = 1.0 + 0.5 * hi.smooth_field(x, 31)
    fac = P.Factorization(T(x), T(pb.weights), T(pb.a), T(pb.b), T(c), pb.kernel_id, 1e-2, precision="fp32",
                          proxy_dirs=pb.proxy if dim == 3 else None)
    op = kernels.Operator(x, pb.weights, pb.a, pb.b, c, pb.kernel_id)
    f = hi.gaussian_rhs(pb.N, nrhs, 8)
    for trans in (False, True):
        y = fac.matvec(T(f), trans=trans).cpu().numpy()
        ref = op.matvec(f, trans=trans)
        assert np.all(np.abs(y - ref).max(axis=0) <= 1e-13 * np.abs(ref).max(axis=0))
    fac.close()


@pytest.mark.parametrize("n,nrhs,kind", [(9, 1, "grid"), (33, 3, "grid"), (24, 5, "shuffled"), (24, 2, "moved")])
def test_helmholtz_sums_match_oracle(P, n, nrhs, kind):
    pb = hi.helmholtz_problem(n, n / 32.0, nrhs=nrhs)
    x = pb.points.copy()
    rng = np.random.default_rng(n)
    if kind == "shuffled":
        x = x[rng.permutation(pb.N)]
    elif kind == "moved":                                 # within the grid test's 1e-6 but not on the grid
        x = x + rng.uniform(-1e-8, 1e-8, x.shape)
    fac = P.Factorization(T(x), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), 2, 1e-2, wavenumber=pb.k)
    op = helmholtz.HelmholtzOperator(x, pb.weights, pb.a, pb.b, pb.c, pb.k)
    f = T(pb.f, torch.complex128)
    for trans in (False, True):
        y = fac.matvec(f, trans=trans).cpu().numpy()
        ref = op.matvec(pb.f, adjoint=trans)
        assert np.abs(y - ref).max() <= 1e-12 * np.abs(ref).max()
    fac.close()
