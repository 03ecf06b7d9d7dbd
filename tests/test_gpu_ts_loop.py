"""The tensor-memory-operand kernel running many iterations a launch, against the
shared-memory-operand kernels (one iteration a launch): the same operands, the same
order of every sum, so the same bits whatever the cut into launches and clusters."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def sampler(p, z, smem, **kw):
    return mhar.Sampler(p.A, p.b, p.x0, z, precision="mixed_rs", seed=9, smem_operands=smem, **kw)


# One and two K chunks, last chunks of 1 .. 4 K steps, one row tile to more than the
# CTAs of a cluster times the slots, clusters of 8 down to 1, ragged strips.
@pytest.mark.parametrize("n,m,z", [(1, 3, 1), (5, 60, 130), (16, 129, 1000), (40, 400, 4096),
                                   (60, 1300, 260), (64, 900, 127), (65, 700, 3000),
                                   (100, 2000, 500), (111, 1100, 9900), (128, 1300, 19600)])
def test_launch_lengths(n, m, z):
    p = wl.cube(n) if m < 4 * n else wl.random_polytope(n, m, seed=n, check_bounded=False)
    if n == 1:
        p.A[0], p.A[1] = 1.0, -1.0
    steps = (5, 1, 2, 7)
    out = []
    for smem in (False, True):
        with sampler(p, z, smem, walker0=3) as s:
            assert (s.kernel_name() == "recompute_ts_kernel") != smem
            got = [s.run(k, thin=1) for k in steps]
            out.append((np.concatenate(got), s.chord(), s.stats().stalls, s.state()))
    (a, ca, sa, xa), (d, cd, sd, xd) = out
    assert np.array_equal(a, d)
    for u, v in zip(ca, cd):
        assert np.array_equal(u, v)
    assert sa == sd and xa[1] == xd[1] == sum(steps) and np.array_equal(xa[0], xd[0])


@pytest.mark.parametrize("rank", [0, 1, 7, 32])
@pytest.mark.parametrize("n,m,z", [(6, 60, 40), (40, 400, 700), (100, 1100, 4500)])
def test_preconditioned(n, m, z, rank):
    p = wl.ill_conditioned(n, m, seed=3, smin=1e-2)
    extent = 1.0 / np.abs(p.A).max(axis=0)
    U = 0.3 * extent[:, None] * np.random.default_rng(1).standard_normal((n, rank))
    out = []
    for smem in (False, True):
        with sampler(p, z, smem) as s:
            first = s.run(3, thin=3)             # then a change between launches
            s.set_preconditioner(extent, U if rank else None)
            out.append(np.concatenate([first, s.run(6, thin=1), s.run(4, thin=2)]))
    assert np.array_equal(*out)


@pytest.mark.parametrize("audit", [0, 3, 5])
@pytest.mark.parametrize("device_out", [False, True])
def test_samples(audit, device_out):
    """Samples written by the kernel: thinning across launches and calls, a part of
    the walkers, audits between (their scratch is the staging buffer)."""
    import torch
    p = wl.random_polytope(12, 600, seed=8)
    z, n = 950, p.n
    with sampler(p, z, False) as s:
        every = s.run(600, thin=1)
    with sampler(p, z, False, emit_walkers=700, out_on_device=device_out, audit_every=audit) as s:
        done = 0
        for steps, thin in ((7, 3), (2, 2), (11, 11), (545, 20), (1, 5)):
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
            assert s.check().run_max_violation <= 0.0
