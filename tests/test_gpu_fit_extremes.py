"""Moments at the ends of the FP64 range."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar
from paper_2104_07097_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def moments(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((1000, n)) @ rng.standard_normal((n, n))
    return X.sum(0), X.T @ X, 1000


@pytest.mark.parametrize("n,rank", [(5, 1), (20, 7), (64, 32)])
def test_overflowing_covariance(n, rank):
    """Finite moments whose covariance (the first coordinate's, then all) is not: refused,
    with eigenvalues that are not numbers on the way; the sampler goes on as before."""
    p = wl.cube(n)
    s1, s2, count = moments(n, n)
    with mhar.Sampler(p.A, p.b, p.x0, 16, precision="fp64", seed=5) as smp, \
            mhar.Sampler(p.A, p.b, p.x0, 16, precision="fp64", seed=5) as ref:
        for first in (1, n):
            big = s1.copy()
            big[:first] = 1e156
            with pytest.raises(mhar.MharError) as e:
                smp.fit_from_moments(big, s2, count, rank, 2)
            assert e.value.code == mhar.E_NONFINITE
        assert np.array_equal(smp.run(3, thin=1), ref.run(3, thin=1))
        for s in (smp, ref):
            s.fit_from_moments(s1, s2, count, rank, 2)
        for a, b in zip(smp.preconditioner(), ref.preconditioner()):
            assert np.array_equal(a, b)
        assert np.array_equal(smp.run(3, thin=1), ref.run(3, thin=1))


@pytest.mark.parametrize("half", [-300, 300])
@pytest.mark.parametrize("n,rank", [(5, 1), (20, 7), (64, 32)])
def test_covariance_of_any_scale(n, rank, half):
    """Every step of the fit scales exactly with a power of two: moments of points times
    2^half, whose squared covariances leave FP64's range, give (delta, U) times 2^half."""
    p = wl.cube(n)
    s1, s2, count = moments(n, n)
    out = []
    for k in (0, half):
        with mhar.Sampler(p.A, p.b, p.x0, 16, precision="fp64", seed=5) as smp:
            smp.fit_from_moments(s1 * 2.0 ** k, s2 * 2.0 ** (2 * k), count, rank, 2)
            delta, U = smp.preconditioner()
            out.append((delta * 2.0 ** -k, U * 2.0 ** -k))
    (d0, U0), (d1, U1) = out
    assert np.abs(U0).max() > 0.0
    assert np.array_equal(d0, d1) and np.array_equal(U0, U1)
