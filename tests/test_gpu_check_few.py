"""The feasibility check of few walkers of a long and wide body: one launch (the screen's two
take longer there), with numpy's value."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar
from test_gpu_check import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed_rs"])
@pytest.mark.parametrize("n,m,z,launches", [(300, 4000, 4, 1), (700, 8192, 4, 1), (300, 8193, 4, 2),
                                            (50, 1600, 40, 1), (130, 1600, 40, 2)])
def test_launches(precision, n, m, z, launches):
    rng = np.random.default_rng(n + m)
    A, b = rng.standard_normal((m, n)), rng.uniform(0.5, 1.5, m)
    per_run = []
    for every in (0, 1):
        with mhar.Sampler(A, b, np.zeros(n), z, precision=precision, audit_every=every) as s:
            s.run(1)
            before = s.stats().kernel_launches
            for _ in range(3):     # one at a time: a loop over iterations ends at an audit
                s.run(1)
            per_run.append(s.stats().kernel_launches - before)
            X, _ = s.state()
            want, tol = reference(A, b, X)
            assert abs(s.check().max_violation - want) <= tol
    assert per_run[1] - per_run[0] == 3 * launches
