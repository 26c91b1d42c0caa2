"""GPU test of the per-kernel GMRES steps (the product of one incidence by wires, dots with partial sums in groups of chunks, the wire-tiled float64
product over the sorted wires) against the persistent solve: row counts that leave the last chunk, piece and
group short, one incidence (more than 64 chunks) and several, from zero and with a restart."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


def _solve(cl, prec, inc, tol, restart, persist, monkeypatch):
    from paper_2410_03060_gb300 import swm

    monkeypatch.setenv("SWM_PERSIST", "1" if persist else "0")
    monkeypatch.setenv("SWM_PRODUCT_FORM", "64")
    ctx = swm.swm_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, 2.0, prec)
        x = np.zeros((len(inc), cl.n_unknowns), dtype=np.complex128)
        assert swm.swm_solve(ctx, inc, tol, restart, 500, x) == swm.SWM_OK
        return x
    finally:
        swm.swm_destroy(ctx)


@pytest.mark.parametrize("prec,tol,bound", [(1, 1e-5, 2e-4), (0, 1e-10, 1e-8)])
@pytest.mark.parametrize("nw,n_inc,restart,nseg", [(3301, 1, 50, None), (61, 1, 50, 16), (33, 1, 50, 2),
                                                   (4203, 9, 4, None), (257, 40, 50, None)])
def test_step_kernels_match_the_persistent_solve(nw, n_inc, restart, nseg, prec, tol, bound, monkeypatch):
    cl = cloud_uniform_cube(nw, 2.2 * nw ** (1 / 3), seed=nw, nseg=nseg)
    rng = np.random.default_rng(n_inc)
    inc = np.stack([rng.uniform(0, 3, n_inc), rng.uniform(0, 6, n_inc), rng.uniform(0, 1, n_inc)], 1)
    a = _solve(cl, prec, inc, tol, restart, False, monkeypatch)
    for r in (0, n_inc - 1):
        b = _solve(cl, prec, inc[r:r + 1], tol, 50, True, monkeypatch)
        # both residuals are at most tol |b|: 20 tol covers the conditioning of these clouds
        assert np.linalg.norm(a[r] - b[0]) <= bound * np.linalg.norm(b[0])
