"""GPU test of BiCGSTAB solves on memory that held something else: an allocator that hands out bytes of 0xff
(a NaN in every format) from the first solve on, and a solve after one that ended in NaNs, give the bits of
an undisturbed solve."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


class _Dirty:
    """Device memory of the context from torch tensors; while `dirty`, filled with 0xff."""

    def __init__(self, swm, ctx):
        import torch

        self.dirty, self.held = False, {}

        def alloc(nbytes, stream, user):
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            t.fill_(255 if self.dirty else 0)
            self.held[t.data_ptr()] = t
            return t.data_ptr()

        def free(ptr, nbytes, stream, user):
            del self.held[ptr]

        self.fns = swm.ALLOC_FN(alloc), swm.FREE_FN(free)
        assert swm.load().swm_set_allocator(ctx.handle, self.fns[0], self.fns[1], None) == swm.SWM_OK


@pytest.mark.parametrize("major", [0, 1])
@pytest.mark.parametrize("form", [74, 75, 76])
@pytest.mark.parametrize("n_inc", [2, 3, 9])
def test_solves_do_not_read_what_memory_held(n_inc, form, major, monkeypatch):
    from paper_2410_03060_gb300 import swm

    if form == 76 and major:
        pytest.skip("form 76 is the incidence-minor solve's")
    monkeypatch.setenv("SWM_PRODUCT_FORM", str(form))
    monkeypatch.setenv("SWM_BICGSTAB_MAJOR", str(major))
    cl = cloud_uniform_cube(120, 6.0, seed=3)
    inc = np.stack([np.linspace(0.1, 3.0, n_inc), np.zeros(n_inc), np.zeros(n_inc)], 1)

    def run(dirty, spoiled):
        ctx = swm.swm_create(0, torch_allocator=False)
        try:
            mem = _Dirty(swm, ctx)
            swm.swm_set_solver(ctx, "bicgstab")
            swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
            swm.swm_build(ctx, K, 2.0, swm.SWM_C64)
            mem.dirty = dirty
            x = np.zeros((n_inc, cl.n_unknowns), dtype=np.complex128)
            if spoiled:  # a guess of NaNs: the solve reports it
                with pytest.raises(swm.SwmError):
                    swm.swm_solve_guess(ctx, inc, np.full_like(x, np.nan), 1e-5, 50, 60, x)
            swm.swm_solve(ctx, inc, 1e-5, 50, 60, x)
            return x
        finally:
            swm.swm_destroy(ctx)

    want = run(False, False)
    assert np.isfinite(want).all()
    assert np.array_equal(run(True, False), want)
    assert np.array_equal(run(False, True), want)
