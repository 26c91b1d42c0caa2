"""GPU test of BiCGSTAB's timed choice of its product form: the solves after the choice (on the pattern it
was made on, on a new pattern, with another number of incidences in between) give the bits of the same calls
with the reported form forced, so each has the tables its form needs."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


def _solves(cl, n_inc):
    from paper_2410_03060_gb300 import swm

    inc = np.stack([np.linspace(0.1, 3.0, n_inc), np.zeros(n_inc), np.zeros(n_inc)], 1)
    ctx = swm.swm_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_set_solver(ctx, "bicgstab")
        out, forms = [], []
        for r_c, k, sel in ((2.0, K, inc), (2.0, 0.9 * K, inc), (2.4, K, inc[:2]), (2.4, K, inc), (1.5, K, inc)):
            swm.swm_build(ctx, k, r_c, swm.SWM_C64)
            x = np.zeros((len(sel), cl.n_unknowns), dtype=np.complex128)
            swm.swm_solve(ctx, sel, 1e-5, 50, 60, x)
            forms.append(swm.swm_get_stats(ctx)["step_rhs_block"])
            out.append(x)
        return out, forms
    finally:
        swm.swm_destroy(ctx)


@pytest.mark.parametrize("nw,side,n_inc", [(60, 5.0, 3), (300, 9.0, 4), (300, 9.0, 37), (1000, 14.0, 9)])
def test_the_chosen_form_is_ready_on_every_build(nw, side, n_inc, monkeypatch):
    cl = cloud_uniform_cube(nw, side, seed=nw)
    monkeypatch.delenv("SWM_PRODUCT_FORM", raising=False)
    chosen, forms = _solves(cl, n_inc)
    assert forms[0] == forms[1] == forms[3] == forms[4]  # chosen once per shape
    for form in {forms[0], forms[2]}:
        monkeypatch.setenv("SWM_PRODUCT_FORM", str(form))
        forced, got = _solves(cl, n_inc)
        assert set(got) == {form}
        for f, a, b in zip(forms, chosen, forced):
            if f == form:
                assert np.isfinite(a).all() and np.array_equal(a, b)
