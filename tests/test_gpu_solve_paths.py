"""GPU tests of the solve's kernels at the sizes where they change over, with the path that ran asserted from
the profiled launches: the dots of the per-kernel GMRES with several pieces of rows per CTA, a last one that
is not full, and steps that add their sums as pairs and in float32; the persistent solve over long rows
with wires of more rows than a lane takes at once (eight)."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


def _solve(cl, prec, r_c, inc, tol, restart, persist, monkeypatch):
    """The currents; one launch of the persistent kernel and none of the dots, or the other way round."""
    from paper_2410_03060_gb300 import swm

    monkeypatch.setenv("SWM_PERSIST", "1" if persist else "0")
    monkeypatch.delenv("SWM_PRODUCT_FORM", raising=False)
    ctx = swm.swm_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, r_c, prec)
        x = np.zeros((len(inc), cl.n_unknowns), dtype=np.complex128)
        launches = []
        for what in ("gmres", "dots"):
            swm.swm_profile(ctx, what)
            assert swm.swm_solve(ctx, inc, tol, restart, 500, x) == swm.SWM_OK
            launches.append(swm.swm_get_stats(ctx)["prof_launches"])
            swm.swm_profile(ctx, "none")
        assert launches[0] == 1 if persist else launches[1] > 0
        assert (launches[1] == 0) == persist
        return x
    finally:
        swm.swm_destroy(ctx)


def _incidences(n, seed):
    rng = np.random.default_rng(seed)
    return np.stack([rng.uniform(0, 3, n), rng.uniform(0, 6, n), rng.uniform(0, 1, n)], 1)


@pytest.mark.parametrize("prec,tol,bound", [(1, 1e-5, 2e-4), (0, 1e-10, 1e-8)])
@pytest.mark.parametrize("nw,n_inc,restart", [(450, 200, 50), (700, 160, 3), (600, 320, 50)])
def test_dots_over_several_pieces(nw, n_inc, restart, prec, tol, bound, monkeypatch):
    cl = cloud_uniform_cube(nw, 2.2 * nw ** (1 / 3), seed=nw)
    # from 153 incidences on a chunk is a whole vector: pieces of 2,048 rows, the last one short
    assert cl.n_unknowns > 2048 and cl.n_unknowns % 2048 > 0
    inc = _incidences(n_inc, n_inc)
    a = _solve(cl, prec, 2.0, inc, tol, restart, False, monkeypatch)
    for r in (0, 77, n_inc - 1):
        b = _solve(cl, prec, 2.0, inc[r:r + 1], tol, 50, True, monkeypatch)
        # both residuals are at most tol |b|: 20 tol covers the conditioning of these clouds
        assert np.linalg.norm(a[r] - b[0]) <= bound * np.linalg.norm(b[0])


@pytest.mark.parametrize("prec,tol,bound", [(1, 1e-5, 2e-4), (0, 1e-10, 1e-8)])
@pytest.mark.parametrize("nseg", [9, 10, 16])
@pytest.mark.parametrize("nw,n_inc", [(201, 1), (160, 3)])
def test_long_rows_of_wires_of_many_rows(nw, n_inc, nseg, prec, tol, bound, monkeypatch):
    cl = cloud_uniform_cube(nw, 12.0, seed=nw, nseg=nseg)
    inc = _incidences(n_inc, nseg)
    a = _solve(cl, prec, 0.0, inc, tol, 50, True, monkeypatch)
    b = _solve(cl, prec, 0.0, inc, tol, 50, False, monkeypatch)
    assert np.linalg.norm(a - b) <= bound * np.linalg.norm(b)
