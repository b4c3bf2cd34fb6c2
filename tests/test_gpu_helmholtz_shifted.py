"""The Helmholtz direct sum on grids away from the origin: their coordinates carry
the rounding of the shift, and the sum is over the points as given.  1e-13 of the
largest entry, as the other direct sums (1e-12 is the bound of the unshifted
test against the same operator)."""
import numpy as np
import pytest
import torch

import hif_inputs as hi
from oracle import helmholtz as hz

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(24, 0.0), (24, 1.0), (24, 100.0), (33, 1e4), (32, 1e4), (24, 1e6)])
def test_sum_is_over_the_given_points(n, shift):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1307_2666_gb300 as P
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda:0")
    pb = hi.helmholtz_problem(n, 2.0, nrhs=2)
    pts = pb.points + shift * np.array([1.0, -0.7])
    A = hz.HelmholtzOperator(pts, pb.weights, pb.a, pb.b, pb.c, pb.k).dense()
    fac = P.Factorization(T(pts), T(pb.weights), T(pb.a), T(pb.b), T(pb.c), 2, 1e-3, wavenumber=pb.k)
    for trans, M in ((False, A), (True, A.conj().T)):
        ref = M @ pb.f
        y = fac.matvec(T(pb.f), trans=trans).cpu().numpy()
        assert np.abs(y - ref).max() <= 1e-13 * np.abs(ref).max()
    fac.close()
