"""GPU test of the copy of E that product form 76 keeps: a call that fits the memory without the copy also
runs, with the same bits, where an allocator grants no more than that (the product then takes form 75, or
gives the copy back when a later buffer needs its memory)."""
import ctypes as C

import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


class _Capped:
    """Torch's allocator behind the context's hooks, refusing what would pass `cap` bytes in all."""

    def __init__(self, swm, ctx, cap):
        import torch

        self.held = self.peak = 0

        def alloc(nbytes, stream, user):
            if self.held + nbytes > cap:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), ctx.device, stream or 0)
            self.held += nbytes
            self.peak = max(self.peak, self.held)
            return p

        def free(ptr, nbytes, stream, user):
            torch.cuda.caching_allocator_delete(ptr)
            self.held -= nbytes

        self.fns = swm.ALLOC_FN(alloc), swm.FREE_FN(free)
        assert swm.load().swm_set_allocator(ctx.handle, self.fns[0], self.fns[1], None) == swm.SWM_OK


def _run(form, cap, monkeypatch):
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(500, 10.0, seed=3)
    inc = np.stack([np.linspace(0.1, 3.0, 9), np.zeros(9), np.zeros(9)], 1)
    obs = np.stack([np.full(181, 1.2), np.linspace(0, 6, 181)], 1)
    monkeypatch.setenv("SWM_PRODUCT_FORM", str(form))
    ctx = swm.swm_create(0, torch_allocator=False)
    try:
        mem = _Capped(swm, ctx, cap)
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_set_solver(ctx, "bicgstab")
        out, forms = [], []
        for k in (K, 0.95 * K):
            swm.swm_build(ctx, k, 2.5, swm.SWM_C64)
            x = np.zeros((9, cl.n_unknowns), dtype=np.complex128)
            swm.swm_solve(ctx, inc, 1e-5, 50, 60, x)
            forms.append(swm.swm_get_stats(ctx)["step_rhs_block"])
            sig = np.zeros((9, len(obs), 2))
            swm.swm_rcs_bistatic(ctx, obs, sig)
            out += [x, sig]
        return out, forms, mem.peak
    finally:
        swm.swm_destroy(ctx)


def test_the_product_copy_never_costs_a_call_its_memory(monkeypatch):
    base, forms, need = _run(75, 1 << 40, monkeypatch)
    assert forms == [75, 75]
    full, forms, peak = _run(76, 1 << 40, monkeypatch)
    assert forms == [76, 76] and peak > need
    for share in (0.0, 0.5, 0.9, 1.0):
        got, forms, _ = _run(76, int(need + share * (peak - need)), monkeypatch)
        assert forms[0] in (75, 76)
        assert share > 0.0 or forms == [75, 75]
        for a, b, c in zip(base, full, got):
            assert np.isfinite(a).all()
            assert np.array_equal(a, b) and np.array_equal(a, c)
