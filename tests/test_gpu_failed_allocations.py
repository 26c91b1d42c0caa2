"""GPU test of solves whose allocations fail: whichever of a solve's requests the caller's allocator refuses,
the call either manages without that buffer or reports SWM_ENOMEM, and the same call on the same context
gives the bits of an undisturbed one as soon as memory is granted again."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


class _Refusing:
    """Torch's allocator behind the context's hooks.  Requests are counted; from number `refuse` on, the
    next `times` of them get nothing."""

    def __init__(self, swm, ctx):
        import torch

        self.count, self.refuse, self.times, self.held, self.sizes = 0, None, 0, {}, []

        def alloc(nbytes, stream, user):
            self.count += 1
            self.sizes.append(int(nbytes))
            if self.refuse is not None and self.count > self.refuse and self.times > 0:
                self.times -= 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), ctx.device, stream or 0)
            self.held[p] = int(nbytes)
            return p

        def free(ptr, nbytes, stream, user):
            torch.cuda.caching_allocator_delete(ptr)
            del self.held[ptr]

        self.fns = swm.ALLOC_FN(alloc), swm.FREE_FN(free)
        assert swm.load().swm_set_allocator(ctx.handle, self.fns[0], self.fns[1], None) == swm.SWM_OK

    def next_refused(self, after):
        """Refuse request `after` from now on, and the one that follows it (dalloc asks twice when it has
        given spare buffers back in between)."""
        self.refuse, self.times = (None, 0) if after is None else (self.count + after, 2)


@pytest.mark.parametrize("solver,prec,major,guess", [("gmres", 1, 0, False), ("gmres", 0, 0, True),
                                                     ("gmres", 1, 0, True), ("bicgstab", 1, 0, False),
                                                     ("bicgstab", 1, 1, True), ("bicgstab", 0, 0, False)])
def test_a_refused_solve_can_be_repeated(solver, prec, major, guess, monkeypatch):
    from paper_2410_03060_gb300 import swm

    monkeypatch.setenv("SWM_PERSIST", "0")
    monkeypatch.setenv("SWM_PRODUCT_FORM", "76" if solver == "bicgstab" else "64")  # no choice by timing
    monkeypatch.setenv("SWM_BICGSTAB_MAJOR", str(major))
    cl = cloud_uniform_cube(150, 7.0, seed=5)
    n_inc = 13
    inc = np.stack([np.linspace(0.1, 3.0, n_inc), np.zeros(n_inc), np.zeros(n_inc)], 1)
    rng = np.random.default_rng(0)
    x0 = 1e-3 * (rng.standard_normal((n_inc, cl.n_unknowns)) + 1j * rng.standard_normal((n_inc, cl.n_unknowns)))

    def prepared():
        ctx = swm.swm_create(0, torch_allocator=False)
        mem = _Refusing(swm, ctx)
        swm.swm_set_solver(ctx, solver)
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_build(ctx, K, 2.0, prec)
        return ctx, mem

    def solve(ctx):
        x = np.zeros((n_inc, cl.n_unknowns), dtype=np.complex128)
        if guess:
            swm.swm_solve_guess(ctx, inc, x0, 1e-5, 20, 100, x)
        else:
            swm.swm_solve(ctx, inc, 1e-5, 20, 100, x)
        return x

    ctx, mem = prepared()
    try:
        before = mem.count
        want = solve(ctx)
        requests = mem.count - before
    finally:
        swm.swm_destroy(ctx)
    assert not mem.held and requests > 15
    refused = 0
    for k in range(requests):
        ctx, mem = prepared()
        try:
            mem.next_refused(k)
            try:
                got = solve(ctx)
            except swm.SwmError as e:
                assert e.code == swm.SWM_ENOMEM
                refused += 1
            else:
                assert np.array_equal(got, want)
            assert mem.times < 2
            mem.next_refused(None)
            assert np.array_equal(solve(ctx), want)
        finally:
            swm.swm_destroy(ctx)
    assert refused > 15
