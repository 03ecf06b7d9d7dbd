"""A new batch's schedule -- the persistent launch, or clusters for few short strips -- against
the shapes set by hand: the same bits, through every change of shape, and one problem's
status in place."""
import ctypes

import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


# One body of a tile and of many, a few small ones, as many strips as SMs and one more,
# uneven bodies (the persistent launch), one large body cut into more units than SMs.
@pytest.mark.parametrize("sizes,z,persistent", [([(5, 60)], 3, False), ([(36, 500)], 300, False),
                                                ([(20, 300)] * 9, 140, False),
                                                ([(8, 90)] * 152, 100, False),
                                                ([(8, 90)] * 153, 100, True),
                                                ([(20, 100), (200, 4000)], 400, True),
                                                ([(250, 4000)], 700, True)])
def test_default_schedule(sizes, z, persistent):
    probs = [(p.A, p.b, p.x0) for p in (wl.random_polytope(n, m, seed=n + m, check_bounded=False)
                                        for n, m in sizes)]
    count = mhar.load().mhar_test_batch_arrivals
    count.argtypes, count.restype = [ctypes.c_void_p, ctypes.c_int32], ctypes.c_int
    out = []
    for shapes in ((), (0,), (1, 0, 1)):
        b = mhar.Batch(probs, z, seed=11)
        assert b.get_shapes()[0] is False and set(b.get_shapes()[1]) <= {0, -1}
        if not shapes:
            assert (count(b._b, 0) > 0) == persistent
        b.run(1)
        for s in shapes:
            b.set_shape(s)
            b.run(1)
        b.run(6 - 1 - len(shapes))
        out.append([b.state(q)[0] for q in range(0, len(sizes), 17)])
        b.close()
    for got in out[1:]:
        for u, v in zip(got, out[0]):
            assert np.array_equal(u, v)
