"""GPU test of the persistent solve with long rows of E read from global memory (a warp per row):
entire coupling of clouds whose E exceeds shared memory, against the same solve with one launch per
kernel, for one and several incidences, both precisions, and from an initial guess."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


def _solve(cl, prec, inc, tol, guess, monkeypatch, persist):
    from paper_2410_03060_gb300 import swm

    monkeypatch.setenv("SWM_PERSIST", "1" if persist else "0")
    ctx = swm.swm_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, 0.0, prec)
        x = np.zeros((len(inc), cl.n_unknowns), dtype=np.complex128)
        if guess is None:
            assert swm.swm_solve(ctx, inc, tol, 50, 500, x) == swm.SWM_OK
        else:
            assert swm.swm_solve_guess(ctx, inc, guess, tol, 50, 500, x) == swm.SWM_OK
        return x
    finally:
        swm.swm_destroy(ctx)


@pytest.mark.parametrize("prec,tol,bound", [(1, 1e-5, 2e-4), (0, 1e-10, 1e-8)])
@pytest.mark.parametrize("nw,n_inc", [(401, 1), (330, 3)])
def test_long_rows_match_the_per_kernel_solve(prec, tol, bound, nw, n_inc, monkeypatch):
    cl = cloud_uniform_cube(nw, 12.0, seed=nw)
    rng = np.random.default_rng(2)
    inc = np.stack([rng.uniform(0, 3, n_inc), rng.uniform(0, 6, n_inc), rng.uniform(0, 1, n_inc)], 1)
    a = _solve(cl, prec, inc, tol, None, monkeypatch, True)
    b = _solve(cl, prec, inc, tol, None, monkeypatch, False)
    # both residuals are at most tol |b|: 20 tol covers the conditioning of these clouds
    assert np.linalg.norm(a - b) <= bound * np.linalg.norm(b)
    g = _solve(cl, prec, inc, tol, 0.9 * b, monkeypatch, True)
    assert np.linalg.norm(g - b) <= bound * np.linalg.norm(b)
