"""GPU test of the float64 products on both sides of the rule that sorts their wires (incidences per tile, wires,
CTAs): the operator's rows for every number of vectors are those of one vector at a time, bit for bit in complex128
(each row is summed column by column by one thread in either order)."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw", [60, 127, 128, 2000, 4100])
def test_every_number_of_vectors(nw):
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw, (nw / 0.1) ** (1 / 3), seed=nw, nseg=np.random.default_rng(nw).integers(2, 17, nw).astype(np.int32))
    rng = np.random.default_rng(1)
    x = rng.standard_normal((67, cl.n_unknowns)) + 1j * rng.standard_normal((67, cl.n_unknowns))
    ctx = swm.swm_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, 2.0, swm.SWM_C128)
        one = np.zeros_like(x)
        for r in range(67):
            swm.swm_apply(ctx, x[r:r + 1], one[r:r + 1])
        for n in (2, 6, 7, 12, 13, 31, 32, 33, 64, 67):
            y = np.zeros_like(x[:n])
            swm.swm_apply(ctx, x[:n], y)
            assert np.array_equal(y, one[:n])
    finally:
        swm.swm_destroy(ctx)
