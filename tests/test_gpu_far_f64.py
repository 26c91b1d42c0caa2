"""GPU test of the float64 far field at its edges: one to five incidences (one, two or four per
thread, with a remainder), observation counts around a warp and a CTA, wire counts around the staged
block, short segments (series) and segments of several wavelengths (table), far-away clouds, and the
monostatic form, against the float64 oracle."""
import math

import numpy as np
import pytest

import oracle as O
from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw,n_rhs,n_obs", [(1, 1, 1), (31, 2, 33), (33, 3, 127), (65, 4, 129), (7, 5, 128)])
@pytest.mark.parametrize("length,nseg,shift", [((0.3, 0.6), None, 0.0), (6.0, 3, 0.0), ((0.3, 0.6), None, 5000.0)])
def test_far_field_matches_oracle(nw, n_rhs, n_obs, length, nseg, shift):
    import torch
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw, 20.0, seed=nw, length=length, nseg=nseg)
    cl.centres[:] += shift
    m, off = O.numbering(cl.nseg)
    rng = np.random.default_rng(n_obs)
    X = rng.standard_normal((int(off[-1]), n_rhs)) + 1j * rng.standard_normal((int(off[-1]), n_rhs))
    obs = np.stack([np.arccos(rng.uniform(-1, 1, n_obs)), rng.uniform(0, 2 * math.pi, n_obs)], 1)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in (cl.centres, cl.dirs, cl.lengths, cl.nseg, off.astype(np.int64))]
    comp = torch.zeros(n_rhs, n_obs, 2, dtype=torch.complex128, device="cuda")
    sigma = torch.zeros(n_rhs, n_obs, 2, dtype=torch.float64, device="cuda")
    cur = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    o = torch.from_numpy(obs).cuda()
    swm.swm_far_components(None, *dev, K, cur, o, comp)
    swm.swm_far_field(None, *dev, K, cur, o, sigma)
    th, ph = obs[:, 0], obs[:, 1]
    rhat = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
    F = O.far_field(cl, K, X, rhat)  # [obs, 3, rhs]
    e = np.stack([np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), -np.sin(th)], 1),
                  np.stack([-np.sin(ph), np.cos(ph), 0 * ph], 1)], 1)  # [obs, 2, 3]
    ref = np.einsum("osc,oci->ios", e, F)
    # the phase k r.c carries the rounding of its largest term, 2^-52 k |c|, on both sides; the sums
    # of nw m terms of modulus at most D |X| add 1e-14 of their total
    phase = 4 * 2.3e-16 * K * (np.abs(cl.centres).max() * 3 + 10)
    scale = np.abs(X).sum(0).max() * (cl.lengths / cl.nseg).max()
    assert np.abs(comp.cpu().numpy() - ref).max() <= (phase + 1e-14) * scale
    want = np.abs(ref) ** 2 / (4 * math.pi)
    assert np.abs(sigma.cpu().numpy() - want).max() <= (phase + 1e-14) * scale * (np.abs(ref).max() + scale) / 6


@pytest.mark.parametrize("n_inc", [1, 33, 130])
def test_monostatic_rcs_matches_oracle(n_inc):
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(9, 6.0, seed=4)
    inc = np.stack([np.linspace(0.1, 3.0, n_inc), np.linspace(0, 5.0, n_inc), np.full(n_inc, 0.4)], 1)
    ctx = swm.swm_create(0)
    try:
        sigma = np.zeros((n_inc, 2))
        swm.swm_run(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg, K, 2.0, swm.SWM_C128, inc, None, sigma,
                    tol=1e-11)
    finally:
        swm.swm_destroy(ctx)
    X = O.solve_lu(O.assemble(cl, K, 2.0, sparse=False), O.rhs(cl, K, inc))
    ref = O.rcs_monostatic(cl, K, X, inc)
    assert np.abs(sigma - ref).max() <= 1e-9 * ref.max()  # the solve's tolerance times 100
