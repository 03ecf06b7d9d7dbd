"""A batch's arrival counters that an expired wait left part of the way: the next run starts
from clear ones, in the whole-batch launch and in the buckets' own."""
import ctypes

import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def advanced(buckets, left):
    probs = [(p.A, p.b, p.x0) for p in (wl.random_polytope(n, m, seed=n, check_bounded=False)
                                        for n, m in ((20, 4000), (100, 5000)))]
    b = mhar.Batch(probs, 130, seed=3)
    if buckets:
        for q in sorted(set(b.get_shapes()[2])):
            b.set_bucket_shape(q, 0)
    b.run(2)
    if left:
        fill = mhar.load().mhar_test_batch_arrivals
        fill.argtypes, fill.restype = [ctypes.c_void_p, ctypes.c_int32], ctypes.c_int
        assert fill(b._b, left) == 4          # two bodies of two strips
    b.run(3)
    out = [b.state(q)[0] for q in range(2)]
    b.close()
    return out


@pytest.mark.parametrize("left", [1, 10, 30])        # of up to 32 and 40 units a strip
@pytest.mark.parametrize("buckets", [False, True])
def test_next_run_starts_clear(buckets, left):
    for u, v in zip(advanced(buckets, left), advanced(buckets, 0)):
        assert np.array_equal(u, v)
