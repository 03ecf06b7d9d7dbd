"""mhar_check (FP64 feasibility) against numpy, at the edges of its FP32 screen.

The check evaluates in FP64 only the rows its screen leaves; the reference is the
plain FP64 maximum.  Both sum n products, so they agree to 2 n u sum |a_i x_i| plus
the rounding of the difference (u = 2^-53)."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def reference(A, b, X):
    v = X @ A.T - b
    k, i = np.unravel_index(np.nanargmax(v), v.shape)
    tol = 2.0 ** -52 * ((A.shape[1] + 2) * (np.abs(X[k]) @ np.abs(A[i])) + np.abs(b[i]))
    return v[k, i], tol


# m on and beside the 128-row tiles, more row tiles than 2 n entries hold (m > 256 n),
# one walker and ragged 64-walker tiles.
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,m,z", [(1, 2, 1), (1, 700, 65), (2, 1100, 3), (17, 127, 64),
                                   (33, 128, 131), (100, 129, 63), (40, 1000, 200), (1, 5000, 900),
                                   (64, 129, 520)])
def test_check_against_numpy(precision, n, m, z):
    rng = np.random.default_rng(n + m + z)
    A = rng.standard_normal((m, n))
    b = rng.uniform(0.5, 1.5, m)
    X = rng.standard_normal((z, n))
    with mhar.Sampler(A, b, np.zeros(n), z, precision=precision) as s:
        s.set_state(X, 0)
        X, _ = s.state()              # as the mode holds them
        got = s.check().max_violation
    want, tol = reference(A, b, X)
    assert abs(got - want) <= tol


# The screen's own limits: products beyond the FP32 range, values far below it, all
# values equal, a maximum that cancels to the last bits.
@pytest.mark.parametrize("kind", ["huge", "tiny", "ties", "cancel"])
def test_check_screen_limits(kind):
    rng = np.random.default_rng(5)
    n, m, z = 20, 300, 800
    A, b = rng.standard_normal((m, n)), np.ones(m)
    X = 0.1 * rng.standard_normal((z, n))
    if kind == "huge":
        A, X = A * 1e30, X * 1e30
    elif kind == "tiny":
        A, X, b = A * 1e-25, X * 1e-25, b * 1e-50
    elif kind == "ties":
        A, X = np.tile(A[:1], (m, 1)), np.tile(X[:1], (z, 1))
    else:
        b = (A @ X[7]) * (1 + 1e-14) + 1e-12 * np.arange(1, m + 1)
        b = np.where(b > 0, b, 50.0)
    with mhar.Sampler(A, b, np.zeros(n), z, precision="fp64") as s:
        s.set_state(X, 0)
        got = s.check().max_violation
    want, tol = reference(A, b, X)
    assert abs(got - want) <= tol
