"""GPU test of E = Z M^-1 in complex64 (a lane per column of the transposed blocks) against the complex128
path's (a lane per entry), through the operator: wires of 2 to 16 segments, block counts at the edges of a
warp's share, one block to a warp's 32."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw,side,r_c", [(2, 1.0, 0.0), (61, 6.0, 2.0), (201, 10.0, 0.0), (300, 12.0, 0.0)])
def test_columns_match_entries(nw, side, r_c):
    from paper_2410_03060_gb300 import swm

    rng = np.random.default_rng(nw)
    cl = cloud_uniform_cube(nw, side, seed=nw, nseg=rng.integers(2, 17, nw).astype(np.int32))
    x = rng.standard_normal((3, cl.n_unknowns)) + 1j * rng.standard_normal((3, cl.n_unknowns))
    out = []
    for prec in (swm.SWM_C128, swm.SWM_C64):
        ctx = swm.swm_create(0)
        try:
            swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
            swm.swm_build(ctx, K, r_c, prec)
            y = np.zeros_like(x)
            swm.swm_apply(ctx, x, y)
            out.append(y - x)
        finally:
            swm.swm_destroy(ctx)
    # single-precision entries of Z and M^-1: a few thousand roundings of 6e-8 at most
    assert np.linalg.norm(out[0] - out[1]) <= 2e-4 * np.linalg.norm(out[0])
