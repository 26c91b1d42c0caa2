"""GPU test of the GMRES product of one incidence on both sides of its rule (wires, rows per wire, entries per
row): the per-kernel solve in complex64 against complex128."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw,density,nseg", [(49999, 0.05, 5), (50000, 0.05, 5), (50003, 0.05, 4), (50003, 0.01, 16),
                                             (50003, 0.02, 2), (50003, 1.0, 5)])
def test_complex64_matches_complex128(nw, density, nseg, monkeypatch):
    import torch
    from paper_2410_03060_gb300 import swm

    monkeypatch.setenv("SWM_PERSIST", "0")
    cl = cloud_uniform_cube(nw, (nw / density) ** (1 / 3), seed=nw, nseg=nseg)
    r_c = 2.0 if density < 1.0 else 2.1  # 38.8 partners of four rows: 155 entries a row
    inc = np.array([[0.7, 0.3, 0.2]])
    x = []
    for prec, tol in ((swm.SWM_C128, 1e-9), (swm.SWM_C64, 1e-5)):
        ctx = swm.swm_create(0)
        try:
            swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
            swm.swm_build(ctx, 0.5 * K, r_c, prec)
            x.append(torch.zeros(1, cl.n_unknowns, dtype=torch.complex128, device="cuda"))
            assert swm.swm_solve(ctx, inc, tol, 50, 300, x[-1]) == swm.SWM_OK
        finally:
            swm.swm_destroy(ctx)
    # complex64: a residual of 1e-5 |b|; 20 of it cover the conditioning of these clouds
    assert float((x[0] - x[1]).norm()) <= 2e-4 * float(x[0].norm())
