"""Small FP64 bodies whose chord ends lie past FP32's range while every row, point and
direction is inside what the FP32 bounds cover: the bits of the direct kernel."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import workloads as wl
from test_gpu_small import both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [23, 26, 40])
def test_ratios_past_fp32(n):
    p = wl.cube(n)
    p.A, p.b, p.x0 = p.A * 2.0 ** -50, p.b * 2.0 ** 50, np.ones(n)
    both(p, 37, pre=(np.full(n, 2.0 ** -40), None), steps=(1,))
