"""Screened contexts that would be slower than the direct kernels (walkers outside the range
that the screen covers, very many rows that tie) go over to those, and back: always the bits
of the direct kernels (which an all-zero row 0 . x <= 2^60 keeps a context on)."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


class Pair:
    """The same chain with the screen and without."""

    def __init__(self, p, z, precision, direct, **kw):
        rows = np.vstack([p.A, np.zeros((1, p.n))]), np.append(p.b, 2.0 ** 60)
        kw = dict(AE=p.AE, bE=p.bE, precision=precision, seed=4, **kw)
        self.s = mhar.Sampler(p.A, p.b, p.x0, z, **kw)
        self.d = mhar.Sampler(*rows, p.x0, z, **kw)
        assert self.s.kernel_name() == "screen_kernel" and self.d.kernel_name() == direct

    def run(self, steps, thin=0):
        a, d = self.s.run(steps, thin), self.d.run(steps, thin)
        assert thin == 0 or np.array_equal(a, d)
        for u, v in zip(self.s.chord(), self.d.chord()):
            assert np.array_equal(u, v)
        (x, t), (y, u) = self.s.state(), self.d.state()
        assert t == u and np.array_equal(x, y)
        return self.s.kernel_name()

    def both(self, call, *args):
        getattr(self.s, call)(*args)
        getattr(self.d, call)(*args)


CASES = [("fp64", "chord_simt_kernel", False), ("fp32", "chord_simt_kernel", False),
         ("fp64", "chord_warp_kernel", True)]


def make(precision, direct, eq, scale=1.0, **kw):
    p = wl.simplex_cuts(30, 200, seed=2) if eq else wl.random_polytope(20, 700, seed=4)
    p.b, p.x0 = p.b * scale, p.x0 * scale
    if eq:
        p.bE = p.bE * scale
    return Pair(p, 130 if eq else 3001, precision, direct, **kw)


@pytest.mark.parametrize("graph_chunk", [0, 16])
@pytest.mark.parametrize("precision,direct,eq", CASES)
def test_tiny_body(precision, direct, eq, graph_chunk):
    """Points of size 1e-17: the direct kernels after the first call, one screened iteration
    after 4, 20, 84 .. of theirs, across calls of every length."""
    q = make(precision, direct, eq, scale=1e-17)
    q.run(3, 1)
    assert q.s.kernel_name() == direct
    for steps, thin in ((2, 1), (2, 2), (1, 1), (1, 0), (40, 7), (60, 20)):
        q.run(steps, thin)
    # 3 screened, then 4 + 1 + 16 + 1 + 64 + 1 + 256: within the last stretch.
    assert q.s.kernel_name() == direct
    q.run(300)
    assert q.s.kernel_name() == direct


@pytest.mark.parametrize("precision,direct,eq", CASES)
def test_long_first_call(precision, direct, eq):
    """The first call looks on the way."""
    q = make(precision, direct, eq, scale=1e-17)
    before = q.s.stats().kernel_launches
    q.run(45, 15)
    assert q.s.kernel_name() == direct
    assert q.s.stats().kernel_launches > before


@pytest.mark.parametrize("precision,direct,eq", CASES)
def test_returns(precision, direct, eq):
    """Directions too short for the screen, then ordinary ones; a state outside the range
    for one iteration only."""
    q = make(precision, direct, eq)
    n = q.s.n
    assert q.run(5, 1) == "screen_kernel"
    q.both("set_preconditioner", np.full(n, 1e-18))
    assert q.run(3, 1) == direct
    q.both("set_preconditioner", np.linspace(0.5, 1.0, n))
    assert q.run(4, 1) == "screen_kernel"
    if eq:
        return
    X = np.full((q.s.z, n), 1e-20)
    q.both("set_state", X, 7)
    assert q.run(1) == direct            # every walker outside, the first iteration
    q.run(4)
    assert q.run(1) == "screen_kernel"   # the trial after four
    assert q.run(30, 6) == "screen_kernel"


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,m,z", [(1, 4000, 3000), (2, 8800, 300)])
def test_rows_that_tie(precision, n, m, z):
    """An interval's ends 2000 times over, 8800 tangents of a circle."""
    p = wl.random_polytope(n, m, seed=5, check_bounded=False)
    q = Pair(p, z, precision, "chord_simt_kernel")
    q.run(3, 1)
    for steps, thin in ((1, 1), (2, 1), (30, 10)):
        q.run(steps, thin)
    if n == 1:                # twice the direct kernels' time and more in FP64 too
        assert q.s.kernel_name() == "chord_simt_kernel"
