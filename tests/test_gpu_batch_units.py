"""The persistent batched launch with strips cut into units, against one CTA a strip, and
the batch's samples in one launch: the same bits (each chord end is an exact minimum)."""
import numpy as np
import pytest

from paper_2104_07097_gb300 import mhar, workloads as wl

pytestmark = pytest.mark.gpu


def problems(sizes):
    return [(p.A, p.b, p.x0) for p in (wl.random_polytope(n, m, seed=7 * n + m, check_bounded=False)
                                       for n, m in sizes)]


# One tile to many, resident and streamed operands, ragged strips, one long body beside
# many short ones (cut into as many units as it has tiles), more than 128 problems.
@pytest.mark.parametrize("sizes,z", [([(5, 60)], 1), ([(20, 400), (300, 5000)], 130),
                                     ([(64, 1025), (65, 1024), (129, 1600)], 33),
                                     ([(30, 240)] * 20 + [(200, 4000)], 300),
                                     ([(6 + q % 5, 90 + q) for q in range(135)], 40)])
def test_cut_units(sizes, z):
    import torch
    probs = problems(sizes)
    out = []
    for shape in (0, 1):
        with_dev = [torch.zeros(2, z, n, dtype=torch.float64, device="cuda") for n, _ in sizes]
        b = mhar.Batch(probs, z, seed=3, out_on_device=True)
        assert b.get_shapes()[1].count(0) > 0        # the default
        b.set_shape(shape)
        b.run(3)
        b.run(6, thin=3, outs=with_dev)
        out.append([o.cpu().numpy() for o in with_dev])
        out[-1] += [b.state(q)[0] for q in range(len(sizes))]
        b.close()
    for u, v in zip(*out):
        assert np.array_equal(u, v)
    for q in range(len(sizes)):
        assert np.array_equal(out[0][q][1], out[0][len(sizes) + q])


def test_samples_on_the_host():
    sizes = [(10, 100), (40, 500)]
    probs = problems(sizes)
    b = mhar.Batch(probs, 70, seed=3, emit_walkers=31)
    got = b.run(4, thin=2)
    for q, (n, _) in enumerate(sizes):
        assert got[q].shape == (2, 31, n)
        assert np.array_equal(got[q][1], b.state(q)[0][:31])
    b.close()
