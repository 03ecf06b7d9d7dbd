"""The factor half of the preconditioner fit over its range of sizes: cluster
orthogonalisation (uneven row shares, fewer rows than CTAs), the Jacobi sweeps'
antidiagonals (even, odd, rank 1 and 2), rank-deficient covariances.

Against oracle.precond on the same moments.  The covariances have eigenvalues
spaced by a factor 0.9, so a subspace of rank <= 32 has a condition number below
1e2 and a relative gap of 0.1: FP64 rounding (n 2^-53 < 1e-13) reaches U U^T
multiplied by at most 1e3 in each of <= 7 products, well under 1e-9.
"""
import numpy as np
import pytest

import oracle.precond as opc
from paper_2104_07097_gb300 import mhar
from paper_2104_07097_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-9


def moments(n, kept, seed, scale):
    """(s1, s2, count) with covariance M diag(0.9^k) M^T of rank `kept`."""
    rng = np.random.default_rng(seed)
    M = np.linalg.qr(rng.standard_normal((n, n)))[0][:, :kept]
    sigma = scale * (M * 0.9 ** np.arange(kept)) @ M.T
    count = 1000
    s1 = rng.standard_normal(n) * np.sqrt(scale)
    s2 = 0.5 * (sigma + sigma.T) * (count - 1) + np.outer(s1, s1) / count
    return s1, s2, count


def fitted(n, s1, s2, count, rank, power):
    p = wl.cube(n)
    with mhar.Sampler(p.A, p.b, p.x0, 16, precision="fp64", seed=5) as smp:
        smp.fit_from_moments(s1, s2, count, rank, power)
        return smp.preconditioner()


@pytest.mark.parametrize("n,rank,power", [(1, 1, 0), (2, 2, 1), (7, 3, 2), (9, 9, 0), (20, 2, 6),
                                          (65, 32, 2), (130, 31, 3), (300, 0, 2), (500, 32, 4)])
def test_fit_from_moments_sizes(n, rank, power):
    s1, s2, count = moments(n, min(n, 60), n, 3e-5)
    delta, U = fitted(n, s1, s2, count, rank, power)
    sigma = (s2 - np.outer(s1, s1) / count) / (count - 1.0)
    dw, Uw = opc.fit(sigma, rank, power, seed=5)
    if rank > 0:
        top = np.abs(Uw @ Uw.T).max()
        np.testing.assert_allclose(U @ U.T, Uw @ Uw.T, rtol=0, atol=TOL * top)
        assert np.all(np.diff((U * U).sum(0)) <= TOL * top)   # largest eigenvalue first
        G = U.T @ U                                           # columns orthogonal
        assert np.abs(G - np.diag(np.diag(G))).max() <= TOL * np.abs(G).max()
    sd = np.sqrt(np.diag(sigma))
    assert np.abs(delta ** 2 - dw ** 2).max() <= TOL * (sd ** 2).max()


@pytest.mark.parametrize("n,kept,rank", [(20, 6, 20), (12, 11, 12), (100, 3, 32)])
def test_fit_rank_deficient(n, kept, rank):
    """More columns than the covariance has directions: U U^T is the covariance."""
    s1, s2, count = moments(n, kept, n, 1.0)
    delta, U = fitted(n, s1, s2, count, rank, 4)
    sigma = (s2 - np.outer(s1, s1) / count) / (count - 1.0)
    assert np.isfinite(U).all() and np.isfinite(delta).all()
    np.testing.assert_allclose(U @ U.T, sigma, rtol=0, atol=TOL * np.abs(sigma).max())
