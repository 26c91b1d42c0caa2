"""GPU test of product form 76 (E as one record per wire): the BiCGSTAB solve with it gives the same bits
as with form 75 (the sums have the same order), over incidence counts at the edges of its thread layout
(one pair, odd counts, several passes), segment counts up to the largest (two row blocks), wires without
partners and rows longer than a staged piece (columns in several pieces), from zero and from a guess."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inc", [2, 3, 7, 37, 130])
@pytest.mark.parametrize("nw,side,r_c,nseg", [(300, 9.0, 2.0, None), (150, 6.0, 2.0, 16), (90, 3.0, 4.0, None),
                                              (40, 400.0, 1.0, None), (60, 5.0, 1.5, 2)])
def test_records_give_the_same_bits_as_the_sorted_product(nw, side, r_c, nseg, n_inc, monkeypatch):
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw, side, seed=nw, nseg=nseg)
    rng = np.random.default_rng(n_inc)
    inc = np.stack([rng.uniform(0, 3, n_inc), rng.uniform(0, 6, n_inc), rng.uniform(0, 1, n_inc)], 1)
    guess = 1e-3 * (rng.standard_normal((n_inc, cl.n_unknowns)) + 1j * rng.standard_normal((n_inc, cl.n_unknowns)))
    got = {}
    for form in (75, 76):
        monkeypatch.setenv("SWM_PRODUCT_FORM", str(form))
        ctx = swm.swm_create(0)
        try:
            swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
            swm.swm_set_solver(ctx, "bicgstab")
            out = []
            for k in (K, 0.9 * K):  # the second build keeps the pattern and refills the records
                swm.swm_build(ctx, k, r_c, swm.SWM_C64)
                x = np.zeros((n_inc, cl.n_unknowns), dtype=np.complex128)
                swm.swm_solve(ctx, inc, 1e-5, 50, 60, x)
                assert swm.swm_get_stats(ctx)["step_rhs_block"] == form
                out.append(x.copy())
                swm.swm_solve_guess(ctx, inc, guess, 1e-5, 50, 60, x)
                out.append(x.copy())
            got[form] = out
        finally:
            swm.swm_destroy(ctx)
    for a, b in zip(got[75], got[76]):
        assert np.isfinite(a).all()
        assert np.array_equal(a, b)
