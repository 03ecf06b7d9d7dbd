"""FP64 bodies with few tiles that the screened chord takes from the warp-per-walker kernel
(equalities, A past the small-body kernel's shared memory): the bits of the direct kernel,
which an all-zero row 0 . x <= 2^60 (outside the screen's range) brings back."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cuts,z,eq", [(40, 95, 1, True), (64, 64, 33, True), (33, 300, 130, True),
                                         (20, 108, 1500, True), (100, 1400, 21, False),
                                         (65, 1300, 129, False)])
@pytest.mark.parametrize("rank", [-1, 3])
def test_same_bits(n, cuts, z, eq, rank):
    p = wl.simplex_cuts(n, cuts, seed=n) if eq else wl.random_polytope(n, cuts, seed=n,
                                                                      check_bounded=False)
    out = []
    for direct in (False, True):
        A, b = p.A, p.b
        if direct:
            A, b = np.vstack([A, np.zeros((1, n))]), np.append(b, 2.0 ** 60)
        with mhar.Sampler(A, b, p.x0, z, AE=p.AE, bE=p.bE, precision="fp64", seed=9, walker0=2) as s:
            assert s.kernel_name() == ("chord_warp_kernel" if direct else "screen_kernel")
            if rank >= 0:
                U = 0.2 * np.random.default_rng(2).standard_normal((n, rank))
                s.set_preconditioner(np.linspace(0.5, 1.5, n), U)
            out.append((s.run(7, thin=1), s.chord(), s.stats().stalls))
    (a, ca, sa), (d, cd, sd) = out
    assert np.array_equal(a, d) and sa == sd
    assert all(np.array_equal(u, v) for u, v in zip(ca, cd))
