"""The stored-slack kernel running many iterations a launch: the same walk for every cut into
launches, the samples that it writes,
and the oracle's steps over the range of shapes."""
import numpy as np
import pytest

from oracle import mixed
from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


# One K chunk, two (resident operands), three and more (streamed), last chunks of 1 .. 4
# steps, one row tile to more than a CTA's, clusters up to 16, ragged strips.
@pytest.mark.parametrize("n,m,z", [(1, 3, 1), (5, 60, 130), (16, 129, 1000), (40, 400, 4096),
                                   (64, 900, 127), (65, 700, 3000), (100, 2000, 300),
                                   (129, 1300, 140), (200, 2600, 70), (30, 8000, 65)])
def test_launch_lengths(n, m, z):
    p = wl.cube(n) if m < 4 * n else wl.random_polytope(n, m, seed=n, check_bounded=False)
    if n == 1:
        p.A[0], p.A[1] = 1.0, -1.0
    out = []
    for steps in ((9,), (1,) * 9, (2, 5, 2)):
        with mhar.Sampler(p.A, p.b, p.x0, z, precision="mixed", seed=9, walker0=3, refresh_k=4) as s:
            got = np.concatenate([s.run(k, thin=1) for k in steps])
            out.append((got, s.chord(), s.stats().stalls, s.state()))
    for got, chord, stalls, state in out[1:]:
        assert np.array_equal(got, out[0][0]) and stalls == out[0][2]
        assert all(np.array_equal(u, v) for u, v in zip(chord, out[0][1]))
        assert state[1] == 9 and np.array_equal(state[0], out[0][3][0])
    # The oracle's step from the points before each of the first two iterations (the
    # tolerance of the mode's parity tests).
    X = np.tile(p.x0, (z, 1))
    with mhar.Sampler(p.A, p.b, p.x0, z, precision="mixed", seed=9, walker0=3) as s:
        for j in range(2):
            ref = mixed.mixed_run(p.A, p.b, X, 1, "mixed", seed=9, step0=j, walker0=3, trace=True)
            s.set_state(X, j)
            X = s.run(1, thin=1)[0]
            assert np.abs(X - ref["samples"][0]).max() <= 1e-4


@pytest.mark.parametrize("audit", [0, 3])
@pytest.mark.parametrize("device_out", [False, True])
def test_samples(audit, device_out):
    """Thinning across launches, refreshes and calls, a part of the walkers, audits between."""
    import torch
    p = wl.random_polytope(12, 600, seed=8)
    kw = dict(precision="mixed", seed=2, refresh_k=50)
    with mhar.Sampler(p.A, p.b, p.x0, 950, **kw) as s:
        every = s.run(600, thin=1)
    with mhar.Sampler(p.A, p.b, p.x0, 950, emit_walkers=700, out_on_device=device_out,
                      audit_every=audit, **kw) as s:
        done = 0
        for steps, thin in ((7, 3), (2, 2), (11, 11), (545, 20), (1, 5)):
            want = every[done:done + steps][thin - 1::thin][:steps // thin, :700]
            out = torch.zeros(max(1, steps // thin), 700, p.n, dtype=torch.float64,
                              device="cuda") if device_out else None
            got = s.run(steps, thin=thin, out=out)
            if steps // thin:
                got = got.cpu().numpy() if device_out else got
                assert np.array_equal(got, want)
            done += steps
        assert np.array_equal(s.state()[0], every[done - 1])


def test_preconditioner_between():
    """Loop launches, then single iterations under a preconditioner (the other pair's turn)."""
    p = wl.ill_conditioned(20, 200, seed=3, smin=1e-2)
    delta = 1.0 / np.abs(p.A).max(axis=0)
    out = []
    for first in (3, 4):
        with mhar.Sampler(p.A, p.b, p.x0, 100, precision="mixed", seed=9) as s:
            s.run(first)
            s.set_preconditioner(delta, None)
            s.set_state(np.tile(p.x0, (100, 1)), 11)
            out.append(s.run(5, thin=1))
    assert np.array_equal(*out)
