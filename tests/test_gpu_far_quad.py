"""GPU test of the float64 far field against extended precision (numpy's long double: 112 bits on Arm, 63 on
x86).  The error is that of the phases k r.c, whose float64 factors are rounded: measured 3.7e-15 of the field
for 200 wires in a cube of 20 wavelengths and 8.2e-15 for 1,500 in one of 40, as with CUDA's sincos."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu
T = np.longdouble


@pytest.mark.skipif(np.finfo(T).nmant < 60, reason="long double is float64 here")
@pytest.mark.parametrize("nw,side,n_obs", [(200, 20.0, 40), (600, 40.0, 12)])
def test_error_is_that_of_the_phases(nw, side, n_obs):
    import torch
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw, side, seed=nw)
    off = np.concatenate([[0], np.cumsum(cl.nseg - 1)]).astype(np.int64)
    rng = np.random.default_rng(0)
    x = rng.standard_normal((1, off[-1])) + 1j * rng.standard_normal((1, off[-1]))
    obs = np.stack([np.arccos(rng.uniform(-1, 1, n_obs)), rng.uniform(0, 2 * np.pi, n_obs)], 1)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (cl.centres, cl.dirs, cl.lengths, cl.nseg, off)]
    comp = torch.zeros(1, n_obs, 2, dtype=torch.complex128, device="cuda")
    swm.swm_far_components(None, *dev, K, torch.from_numpy(x).cuda(), torch.from_numpy(obs).cuda(), comp)
    got = comp.cpu().numpy()[0]

    th, ph = obs.T.astype(T)
    frame = np.stack([np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1),
                      np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), -np.sin(th)], 1),
                      np.stack([-np.sin(ph), np.cos(ph), 0 * ph], 1)])
    c, t, L, n = cl.centres.astype(T), cl.dirs.astype(T), cl.lengths.astype(T), cl.nseg.astype(int)
    D = L / n
    wire = np.repeat(np.arange(nw), n - 1)
    s = -L[wire] / 2 + (np.arange(len(wire)) - off[:-1][wire] + 1) * D[wire]
    err = size = T(0)
    for o in range(n_obs):
        beta = T(K) * (t @ frame[0, o])
        z = beta * D / 2
        amp = D * (np.sin(z) / z) ** 2
        phase = T(K) * (c @ frame[0, o])[wire] + beta[wire] * s
        w = amp[wire] * (np.cos(phase) + 1j * np.sin(phase)) * x[0].astype(np.clongdouble)
        F = (w[:, None] * t[wire]).sum(0)
        for i in (0, 1):
            want = F @ frame[1 + i, o]
            err += abs(got[o, i].astype(np.clongdouble) - want) ** 2
            size += abs(want) ** 2
    # five roundings (the three products of r.c, the direction's cosines twice) of the largest phase at most
    phase = 5 * 2.0 ** -53 * K * np.abs(cl.centres).sum(1).max()
    assert float(np.sqrt(err / size)) <= phase + 2e-15
