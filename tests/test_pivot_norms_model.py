"""The pivot rule of the large 64-bit groups (big_step_kernel, big_update_kernel)
as a model on the CPU: squares of the column norms carried from step to step,
summed anew below kNormKeep of the last sum, and the columns within kNormTie of
the largest summed before a pivot or the rank is decided.  Every decision has
to be the one that sums over all columns give, ties to the lowest index."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1307_2666_gb300", "csrc")


def constant(name):
    src = open(os.path.join(CSRC, "k_large.cu")).read()
    return float(re.search(rf"constexpr double {name} = ([0-9.e+-]+);", src).group(1))


def square(col):
    return float(np.add.reduce(col * col))


def pivots(A, tol, keep, tie):
    """Returns the pivots taken, and at how many steps they are not those of sums."""
    R = np.array(A, dtype=np.float64)
    m, n = R.shape
    perm = np.arange(n)
    nrm = np.array([square(R[:, l]) for l in range(n)])
    last, fresh = nrm.copy(), np.ones(n, dtype=bool)
    nu0, wrong, order = None, 0, []
    for j in range(min(m, n)):
        top = nrm[j:].max()
        close = j + np.nonzero(nrm[j:] >= (1.0 - tie) * top)[0]
        th2 = 0.0 if j == 0 else (tol * nu0) ** 2
        if not fresh[close].all() and (close.size > 1 or abs(top - th2) <= tie * th2):
            for l in close[~fresh[close]]:
                nrm[l] = last[l] = square(R[j:, l])
                fresh[l] = True
        first = lambda v: j + min(np.nonzero(v == v.max())[0], key=lambda l: perm[j + l])
        p = first(nrm[j:])
        exact = np.array([square(R[j:, l]) for l in range(j, n)])
        e = first(exact)
        bn, be = np.sqrt(nrm[p]), np.sqrt(exact.max())
        nu0 = bn if j == 0 else nu0
        stop, estop = bn <= tol * nu0 or bn == 0.0, be <= tol * nu0 or be == 0.0
        wrong += (stop != estop) or (not stop and p != e)
        if stop:
            break
        order.append(int(perm[p]))
        for v in (perm, nrm, last, fresh):
            v[[j, p]] = v[[p, j]]
        R[:, [j, p]] = R[:, [p, j]]
        x = R[j:, j].copy()
        ss = x[1:] @ x[1:]
        if ss != 0.0:
            beta = -np.copysign(np.sqrt(x[0] * x[0] + ss), x[0])
            v = x / (x[0] - beta)
            v[0] = 1.0
            R[j:, j + 1:] -= np.outer(v, (beta - x[0]) / beta * (v @ R[j:, j + 1:]))
            R[j, j], R[j + 1:, j] = beta, 0.0
        s = np.maximum(nrm[j + 1:] - R[j, j + 1:] ** 2, 0.0)
        for q, l in enumerate(range(j + 1, n)):
            if s[q] >= keep * last[l]:
                nrm[l], fresh[l] = s[q], False
            else:
                nrm[l] = last[l] = square(R[j + 1:, l])
                fresh[l] = True
    return order, wrong


def tied(rng, m, n):
    """A column along e_0, then pairs that are equal below the first row."""
    A = np.zeros((m, n))
    A[0, 0] = 1e3
    half = (n - 1) // 2
    A[1:, 1:1 + half] = rng.standard_normal((m - 1, half))
    A[1:, 1 + half:1 + 2 * half] = A[1:, 1:1 + half]
    A[0, 1:] = rng.uniform(0.5, 2.0, n - 1)
    return A


def test_ties_are_decided_on_sums():
    keep, tie = constant("kNormKeep"), constant("kNormTie")
    missed = 0
    for seed in range(20):
        A = tied(np.random.default_rng(seed), 60, 21)
        assert pivots(A, 1e-9, keep, tie)[1] == 0
        missed += pivots(A, 1e-9, keep, -1.0)[1]      # no column close: carried squares alone
    assert missed > 0


@pytest.mark.parametrize("m,n,decay", [(300, 120, 0.0), (300, 120, 0.02), (600, 200, 0.1), (200, 150, 0.3)])
def test_pivots_and_rank_are_those_of_sums(m, n, decay):
    keep, tie = constant("kNormKeep"), constant("kNormTie")
    rng = np.random.default_rng(m + n)
    U, _ = np.linalg.qr(rng.standard_normal((m, n)))
    V, _ = np.linalg.qr(rng.standard_normal((n, n)))
    A = (U * 10.0 ** (-decay * np.arange(n))) @ V.T
    order, wrong = pivots(A, 1e-9, keep, tie)
    assert wrong == 0 and len(order) > 10


def test_margin_covers_the_worst_carried_error():
    # 1,000 steps, 10,000 rows: subtractions and reflections as bounded beside
    # the constants, relative to a square at the keep line
    keep, tie = constant("kNormKeep"), constant("kNormTie")
    u = 2.0 ** -53
    assert 2 * (1000 * u / keep + 1000 * 2 * 10000 * u / keep) <= tie
