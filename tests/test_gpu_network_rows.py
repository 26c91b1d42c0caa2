"""GPU test of the warm-start network's message rows: clouds without partners, with more than 16
partners for some wires (rows left absent), and with more than 16 per wire on average (16 rows per
wire), at one and two incidences, against the float64 oracle."""
import numpy as np
import pytest

import oracle as O
import oracle.learned as NL
from gpu_helpers import K
from synth import cloud_uniform_cube
from synth.netinit import init_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inc", [1, 2])
@pytest.mark.parametrize("nw,side,r_c", [(33, 40.0, 1.0), (70, 3.4, 1.5), (40, 2.0, 4.0)])
def test_network_rows_match_oracle(nw, side, r_c, n_inc):
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw, side, seed=nw)
    inc = np.array([[0.4, 0.7, 0.2], [1.9, 3.0, 1.1]])[:n_inc]
    p32 = init_params(3)
    ctx = swm.swm_create(0)
    net = swm.swm_net_create(0)
    try:
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, r_c, swm.SWM_C128)
        swm.swm_net_set_params(net, p32)
        nbr = NL.neighbour_lists(cl, r_c)
        pairs = swm.swm_get_stats(ctx)["nb"] - nw
        assert {33: pairs == 0, 70: 0 < pairs < 16 * nw and (nbr >= 0).sum() < pairs, 40: pairs > 16 * nw}[nw]
        Xe, Xs = NL.features(cl, K, inc, r_c, nbr)
        xi = NL.isolated_currents(cl, K, inc)
        rng = np.random.default_rng(1)
        xt = xi * (1.0 + 0.3 * rng.standard_normal(xi.shape))
        p64 = p32.astype(np.float64)
        lo, go, x0o = NL.loss_and_grad(p64, cl, K, inc, Xe, Xs, xi, xt, nbr)
        x0 = swm.swm_net_predict(net, ctx, inc).T
        # float32 features and layers of at most 256 terms: 1e-5 of the correction's scale
        assert np.linalg.norm(x0 - x0o) <= 1e-5 * np.linalg.norm(x0o)
        lg, gg = swm.swm_net_train_step(net, ctx, inc, xt.T.copy(), 0.0, want_grad=True)
        assert abs(lg - lo) <= 1e-5 * lo
        o = 0
        for i, n in NL.LAYERS:
            a, b = gg[o:o + i * n + n], go[o:o + i * n + n]
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
            o += i * n + n
        with pytest.raises(swm.SwmError):  # zero targets: refused, nothing changes
            swm.swm_net_train_step(net, ctx, inc, np.zeros_like(xt.T).copy(), 1e-3)
        assert np.array_equal(swm.swm_net_get_params(net), p32)
    finally:
        swm.swm_net_destroy(net)
        swm.swm_destroy(ctx)
