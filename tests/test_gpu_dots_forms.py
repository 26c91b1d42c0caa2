"""GPU test of the per-kernel GMRES dots in the forms that stage u and w: float64, and the half-precision basis
of the bfloat16 solve on both sides of 2^19 rows in all; chunks that are not full, groups of chunks, restarts.
Against the persistent solve of single incidences in complex128."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


def _solve(cl, prec, inc, tol, restart, persist, monkeypatch):
    from paper_2410_03060_gb300 import swm

    monkeypatch.setenv("SWM_PERSIST", "1" if persist else "0")
    ctx = swm.swm_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, 2.0, prec)
        x = np.zeros((len(inc), cl.n_unknowns), dtype=np.complex128)
        assert swm.swm_solve(ctx, inc, tol, restart, 500, x) == swm.SWM_OK
        return x
    finally:
        swm.swm_destroy(ctx)


@pytest.mark.parametrize("prec,tol,bound", [(0, 1e-10, 1e-8), (2, 1e-5, 2e-4)])
@pytest.mark.parametrize("nw,n_inc,restart", [(41, 13, 50), (3301, 1, 4), (700, 140, 50), (700, 150, 5),
                                              (13001, 16, 50)])
def test_dots_match_the_persistent_solve(nw, n_inc, restart, prec, tol, bound, monkeypatch):
    cl = cloud_uniform_cube(nw, 2.2 * nw ** (1 / 3), seed=nw)
    assert (cl.n_unknowns * n_inc >= 1 << 19) == (n_inc in (150, 16))
    rng = np.random.default_rng(n_inc)
    inc = np.stack([rng.uniform(0, 3, n_inc), rng.uniform(0, 6, n_inc), rng.uniform(0, 1, n_inc)], 1)
    a = _solve(cl, prec, inc, tol, restart, False, monkeypatch)
    for r in sorted({0, n_inc // 2, n_inc - 1}):
        b = _solve(cl, 0, inc[r:r + 1], 1e-10, 50, True, monkeypatch)
        # the residual is at most tol |b|: 20 tol covers the conditioning of these clouds, and bfloat16's values
        # are those of complex64 (roundings of 6e-8 in the entries)
        assert np.linalg.norm(a[r] - b[0]) <= bound * np.linalg.norm(b[0])
