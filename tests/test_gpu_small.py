"""Small bodies in one launch (small_kernel) against the per-iteration kernels.

All-zero rows 0 . x <= 2^60 change nothing but the route: with them a body lies outside
the range of the fast paths and takes the direct kernels, whose FP64 bits the one-launch
kernel must give."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def both(p, z, pre=None, X0=None, steps=(5, 1, 3), seed=9, walker0=0):
    out = []
    for direct in (False, True):
        A, b = p.A, p.b
        if direct:
            extra = max(1, 1025 // p.n + 1 - p.m)
            A, b = np.vstack([A, np.zeros((extra, p.n))]), np.append(b, np.full(extra, 2.0 ** 60))
        with mhar.Sampler(A, b, p.x0, z, precision="fp64", seed=seed, walker0=walker0) as s:
            name = s.kernel_name()
            assert name.startswith("chord_") if direct else name == "small_kernel"
            if pre is not None:
                s.set_preconditioner(*pre)
            if X0 is not None:
                s.set_state(X0, 3)
            got = [s.run(k, thin=1) for k in steps]     # launches of several lengths
            out.append((np.concatenate(got), s.chord(), s.stats().stalls, s.state()))
    (a, ca, sa, xa), (d, cd, sd, xd) = out
    assert np.array_equal(a, d)
    for u, v in zip(ca, cd):
        assert np.array_equal(u, v)
    assert sa == sd and xa[1] == xd[1] and np.array_equal(xa[0], xd[0])


# One walker per CTA up to the most a CTA takes, ragged last CTAs, both chord forms
# (m n up to 1024 direct, above screened), n and m on and beside 4, 32 and 128.
@pytest.mark.parametrize("n,m,z", [(1, 2, 1), (1, 33, 700), (2, 7, 3), (10, 20, 100), (5, 60, 9001),
                                   (8, 128, 2500), (8, 129, 1301), (37, 300, 301), (64, 130, 650),
                                   (100, 390, 20), (31, 520, 61), (24, 1900, 128)])
def test_shapes(n, m, z):
    p = wl.cube(n) if m < 4 * n else wl.random_polytope(n, m, seed=n, check_bounded=n > 1 and m < 300)
    if n == 1:
        p.A[0], p.A[1] = 1.0, -1.0
    both(p, z, walker0=5)


@pytest.mark.parametrize("rank", [0, 1, 5, 32])
@pytest.mark.parametrize("n,m,z", [(6, 60, 40), (40, 400, 70)])
def test_preconditioned(n, m, z, rank):
    p = wl.ill_conditioned(n, m, seed=3, smin=1e-2)
    extent = 1.0 / np.abs(p.A).max(axis=0)
    U = 0.3 * extent[:, None] * np.random.default_rng(1).standard_normal((n, rank))
    both(p, z, pre=(extent, U if rank else None))


@pytest.mark.parametrize("kind", ["duplicates", "facets", "tiny", "stiff", "huge"])
def test_bodies(kind):
    p = wl.random_polytope(20, 160, seed=4)
    pre = X0 = None
    if kind == "duplicates":
        p.A, p.b = np.tile(p.A, (2, 1)), np.tile(p.b, 2)
    elif kind == "facets":              # on and, by rounding, just outside a facet
        p = wl.cube(20)
        p.A, p.b = np.tile(p.A, (4, 1)), np.tile(p.b, 4)
        X0 = np.random.default_rng(6).uniform(-0.9, 0.9, (90, 20))
        X0[::3, 5] = 1.0
        X0[1::3, 7] = -1.0 - 1e-9
    elif kind == "tiny":                # points below the range the screen covers
        p.b = p.b * 1e-17
    elif kind == "stiff":               # directions below it
        pre = (np.full(20, 1e-18), None)
    else:                               # points and directions above it
        p.A, p.b, pre = p.A * 1e-8, p.b * 1e7, (np.full(20, 1e20), None)
    both(p, 90, pre=pre, X0=X0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_walkers_per_cta(precision):
    """A walker's chain does not depend on how many share its CTA."""
    p = wl.random_polytope(7, 60, seed=2)
    with mhar.Sampler(p.A, p.b, p.x0, 5000, precision=precision, seed=3) as s:
        assert s.kernel_name() == "small_kernel"
        many = s.run(7, thin=7)[0]
    for lo, hi in ((0, 1), (1200, 1500), (4990, 5000)):
        with mhar.Sampler(p.A, p.b, p.x0, hi - lo, precision=precision, seed=3, walker0=lo) as s:
            assert np.array_equal(s.run(7, thin=7)[0], many[lo:hi])


@pytest.mark.parametrize("audit", [0, 3, 5])
@pytest.mark.parametrize("device_out", [False, True])
def test_samples(audit, device_out):
    """Samples written by the iteration kernel: thinning across launches and calls,
    a part of the walkers, audits between (their scratch is the staging buffer)."""
    import torch
    p = wl.random_polytope(12, 600, seed=8)    # audits of this size screen
    kw = dict(precision="fp64", seed=2, emit_walkers=700, out_on_device=device_out)
    z, n = 950, p.n
    with mhar.Sampler(p.A, p.b, p.x0, z, precision="fp64", seed=2) as s:
        assert s.kernel_name() == "small_kernel"
        every = s.run(1100, thin=1)
    with mhar.Sampler(p.A, p.b, p.x0, z, audit_every=audit, **kw) as s:
        done = 0
        for steps, thin in ((7, 3), (2, 2), (11, 11), (1045, 20), (1, 5)):
            want = every[done:done + steps][thin - 1::thin][:steps // thin, :700]
            out = torch.zeros(max(1, steps // thin), 700, n, dtype=torch.float64,
                              device="cuda") if device_out else None
            got = s.run(steps, thin=thin, out=out)
            if steps // thin:
                got = got.cpu().numpy() if device_out else got
                assert np.array_equal(got, want)
            done += steps
        assert np.array_equal(s.state()[0], every[done - 1])
        if audit:
            assert s.check().run_max_violation <= 1e-12
