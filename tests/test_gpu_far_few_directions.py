"""GPU test of the float64 far field with many incidences seen from few directions (a receiver that stays, a
transmitter that moves): threads run over directions and incidences together, one, two or four incidences
each.  Against the same pairs one incidence at a time, and its time against the same number of pairs the
other way round."""
import math

import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


def _device(nw, side):
    import torch

    cl = cloud_uniform_cube(nw, side, seed=nw)
    off = np.concatenate([[0], np.cumsum(cl.nseg - 1)]).astype(np.int64)
    return int(off[-1]), [torch.from_numpy(np.ascontiguousarray(a)).cuda()
                          for a in (cl.centres, cl.dirs, cl.lengths, cl.nseg, off)]


def _case(N, n_rhs, n_obs):
    import torch

    rng = np.random.default_rng(n_rhs * 1000 + n_obs)
    cur = rng.standard_normal((n_rhs, N)) + 1j * rng.standard_normal((n_rhs, N))
    obs = np.stack([np.arccos(rng.uniform(-1, 1, n_obs)), rng.uniform(0, 2 * math.pi, n_obs)], 1)
    return torch.from_numpy(cur).cuda(), torch.from_numpy(obs).cuda()


@pytest.mark.parametrize("n_rhs", [1, 2, 3, 4, 5, 33, 127, 130, 181])
@pytest.mark.parametrize("n_obs", [1, 2, 3, 31, 64])
def test_matches_one_incidence_at_a_time(n_rhs, n_obs):
    import torch
    from paper_2410_03060_gb300 import swm

    N, dev = _device(37, 7.0)
    cur, obs = _case(N, n_rhs, n_obs)
    comp = torch.full((n_rhs, n_obs, 2), math.nan, dtype=torch.complex128, device="cuda")
    swm.swm_far_components(None, *dev, K, cur, obs, comp)
    one = torch.zeros(1, n_obs, 2, dtype=torch.complex128, device="cuda")
    scale = float(dev[2].max())  # per unit of current, over 37 wires of at most five segments
    for r in range(n_rhs):
        swm.swm_far_components(None, *dev, K, cur[r:r + 1].contiguous(), obs, one)
        # the sums of the chunks of wires may be cut elsewhere: their roundings alone
        assert (comp[r] - one[0]).abs().max() <= 2.0 ** -52 * 37 * N * scale
    assert torch.isfinite(comp.abs()).all()


def test_few_directions_take_no_longer_than_few_incidences():
    import torch
    from paper_2410_03060_gb300 import swm

    N, dev = _device(10000, 60.0)
    ms = []
    for n_rhs, n_obs in ((181, 1), (1, 181)):
        cur, obs = _case(N, n_rhs, n_obs)
        sigma = torch.zeros(n_rhs, n_obs, 2, dtype=torch.float64, device="cuda")
        best = math.inf
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            swm.swm_far_field(None, *dev, K, cur, obs, sigma)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms.append(best)
    # as many pairs: a lane per direction alone took about ten times as long
    assert ms[0] <= 3.0 * ms[1]
