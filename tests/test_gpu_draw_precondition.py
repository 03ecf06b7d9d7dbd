"""draw_precondition_kernel at the edges of its tiles (64 walkers x 64 coordinates, quads of
four, blocks of several tiles), against oracle.mixed's step from the same state: the
tolerance is that of the preconditioned walks' parity tests."""
import numpy as np
import pytest

from oracle import mixed
from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,z,rank,smem", [
    ("mixed_rs", 3, 1, 1, True), ("mixed_rs", 64, 64, 32, True), ("mixed_rs", 65, 63, 5, True),
    ("mixed_rs", 130, 65, 0, False), ("mixed_rs", 203, 700, 31, False), ("mixed", 66, 65, 4, False),
    ("fp32", 65, 130, 3, False)])
def test_tiles(prec, n, z, rank, smem):
    p = wl.cube(n)
    rng = np.random.default_rng(n)
    delta, U = rng.uniform(0.5, 1.5, n), 0.4 * rng.standard_normal((n, rank))
    kw = {"smem_operands": True} if smem else {}
    with mhar.Sampler(p.A, p.b, p.x0, z, precision=prec, seed=5, **kw) as s:
        s.set_preconditioner(delta, U if rank else None)
        X = np.tile(p.x0, (z, 1))
        for j in range(3):
            ref = mixed.mixed_run(p.A, p.b, X, 1, prec, seed=5, step0=j, delta=delta, U=U, trace=True)
            s.set_state(X, j)
            X = s.run(1, thin=1)[0]
            assert np.abs(X - ref["samples"][0]).max() <= 1e-4
