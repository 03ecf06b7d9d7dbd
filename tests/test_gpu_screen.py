"""The screened chord of the FP64 / FP32 modes against the direct kernels, bit for bit.

A redundant all-zero row 0 . x <= 2^60 lies outside the screen's range, so the same
body with it takes the direct kernels; both must give the same samples and chords."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def both(p, z, precision, steps=6, pre=None, seed=4, X0=None):
    out = []
    for direct in (False, True):
        A, b = p.A, p.b
        if direct:
            A, b = np.vstack([A, np.zeros((1, p.n))]), np.append(b, 2.0 ** 60)
        with mhar.Sampler(A, b, p.x0, z, AE=p.AE, bE=p.bE, precision=precision, seed=seed) as s:
            screened = not direct and (precision == "fp64" or p.n >= 64 or p.m * z >= 2 ** 21)
            assert s.kernel_name() == ("screen_kernel" if screened else "chord_simt_kernel")
            if pre is not None:
                s.set_preconditioner(*pre)
            if X0 is not None:
                s.set_state(X0, 0)
            got = s.run(steps, thin=1)
            out.append((got, s.chord(), s.stats().stalls))
    (a, ca, sa), (d, cd, sd) = out
    assert np.array_equal(a, d)
    for u, v in zip(ca, cd):
        assert np.array_equal(u, v)
    assert sa == sd


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,m,z", [(1, 640, 4000), (3, 700, 3030), (16, 897, 3700), (64, 1000, 640),
                                   (65, 1025, 641), (129, 1100, 620), (200, 5000, 130)])
def test_shapes(precision, n, m, z):
    both(wl.random_polytope(n, m, seed=n, check_bounded=n > 3), z, precision)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["duplicates", "simplex", "illcond", "cube", "tiny", "stiff"])
def test_bodies(precision, kind):
    rng = np.random.default_rng(3)
    pre = None
    if kind == "duplicates":           # every bound ties with another row's
        p = wl.random_polytope(30, 350, seed=1)
        p.A, p.b = np.tile(p.A, (2, 1)), np.tile(p.b, 2)
    elif kind == "simplex":            # sparse rows, slacks of very different size, m_E = 1
        p = wl.simplex_cuts(60, 700, seed=2)
    elif kind == "illcond":
        p = wl.ill_conditioned(40, 800, seed=3)
        extent = 1.0 / np.abs(p.A).max(axis=0)
        pre = (extent, 0.3 * extent[:, None] * rng.standard_normal((40, 5)))
    elif kind == "cube":
        p = wl.cube(400)
    else:                              # points / directions outside 2^-50 .. 2^50
        p = wl.random_polytope(20, 700, seed=4)
        if kind == "tiny":
            p.b = p.b * 1e-17
        else:
            pre = (np.full(20, 1e-18), None)
    both(p, 3001, precision, pre=pre)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_walkers_on_facets(precision):
    """Points on (or, by rounding, just outside) a facet: zero slacks on both sides."""
    p = wl.cube(24)
    p.A, p.b = np.tile(p.A, (16, 1)), np.tile(p.b, 16)
    rng = np.random.default_rng(6)
    X0 = rng.uniform(-0.9, 0.9, (2800, 24))
    X0[::3, 5] = 1.0
    X0[1::3, 7] = -1.0 - 1e-9
    both(p, 2800, precision, X0=X0)
