"""GPU test of the stateless far field over wires of one segment (no unknowns), which the stateless entry
points take as they come: such wires add nothing, whatever lies beside their place in the currents, so the
results are those of the cloud without them."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rhs", [1, 2, 5])
@pytest.mark.parametrize("nw,empty", [(1, [0]), (9, [0, 3, 4, 8]), (70, [0, 31, 32, 33, 69])])
def test_wires_without_unknowns_add_nothing(nw, empty, n_rhs):
    import torch
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw + 2, 9.0, seed=nw)
    nseg = cl.nseg.astype(np.int32).copy()
    nseg[empty] = 1
    keep = nseg > 1
    off = np.concatenate([[0], np.cumsum(nseg.astype(np.int64) - 1)])
    rng = np.random.default_rng(n_rhs)
    n = int(off[-1])
    X = rng.standard_normal((n_rhs, n)) + 1j * rng.standard_normal((n_rhs, n))
    # entries before and behind the currents that must not be read
    buf = torch.full((n_rhs * n + 2,), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda")
    buf[1:-1] = torch.from_numpy(X.ravel()).cuda()
    cur = buf[1:-1].view(n_rhs, n)
    obs = torch.from_numpy(np.stack([rng.uniform(0, 3, 37), rng.uniform(0, 6, 37)], 1)).cuda()
    out = []
    for sel in (np.ones(nw + 2, bool), keep):
        o = np.concatenate([[0], np.cumsum(nseg[sel].astype(np.int64) - 1)])
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
               for a in (cl.centres[sel], cl.dirs[sel], cl.lengths[sel], nseg[sel], o)]
        comp = torch.zeros(n_rhs, 37, 2, dtype=torch.complex128, device="cuda")
        swm.swm_far_components(None, *dev, K, cur, obs, comp)
        sig = []
        for f in (swm.swm_far_field, swm.swm_far_field_noalloc):
            s = torch.zeros(n_rhs, 37, 2, dtype=torch.float64, device="cuda")
            f(None, *dev, K, cur, obs, s)
            sig.append(s.cpu().numpy())
        out.append([comp.cpu().numpy()] + sig)
    # the chunks of wires differ, so the same terms are added in another order: at most n roundings of
    # 2^-53 of their total on each side
    scale = np.abs(X).sum(1).max() * (cl.lengths / nseg).max()
    bound = 2 * n * 1.2e-16 * scale
    assert np.isfinite(out[0][0]).all()
    assert np.abs(out[0][0] - out[1][0]).max() <= bound
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.abs(a - b).max() <= bound * 2 * scale
