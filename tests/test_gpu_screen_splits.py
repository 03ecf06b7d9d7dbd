"""The screened chord with few walkers and many rows, where a CTA takes several row tiles,
against the direct kernels bit for bit; FP32 bodies that the screen would slow down (few
products) take the direct kernel themselves."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def chain(A, b, x0, z, precision, kernel):
    with mhar.Sampler(A, b, x0, z, precision=precision, seed=8) as s:
        assert s.kernel_name() == kernel
        return s.run(5, thin=1), s.chord()


# 17 tiles to 79, one and more strips, a last CTA with fewer tiles.
@pytest.mark.parametrize("n,m,z", [(64, 2100, 65), (20, 4000, 300), (100, 8000, 129), (5, 10001, 7)])
def test_several_tiles_a_cta(n, m, z):
    p = wl.random_polytope(n, m, seed=n, check_bounded=False)
    a, ca = chain(p.A, p.b, p.x0, z, "fp64", "screen_kernel")
    d, cd = chain(np.vstack([p.A, np.zeros((1, n))]), np.append(p.b, 2.0 ** 60), p.x0, z, "fp64",
                  "chord_simt_kernel")
    assert np.array_equal(a, d)
    assert all(np.array_equal(u, v) for u, v in zip(ca, cd))


@pytest.mark.parametrize("n,m,z,screen", [(64, 8000, 65, False), (64, 4000, 65, False),
                                          (96, 8000, 65, False), (64, 4000, 130, False),
                                          (96, 8000, 130, True), (129, 4100, 300, True)])
def test_fp32_with_few_products(n, m, z, screen):
    p = wl.random_polytope(n, m, seed=n, check_bounded=False)
    a, ca = chain(p.A, p.b, p.x0, z, "fp32", "screen_kernel" if screen else "chord_simt_kernel")
    d, cd = chain(np.vstack([p.A, np.zeros((1, n))]), np.append(p.b, 2.0 ** 60), p.x0, z, "fp32",
                  "chord_simt_kernel")
    assert np.array_equal(a, d)
    assert all(np.array_equal(u, v) for u, v in zip(ca, cd))
