"""GPU test of swm_set_cloud whose allocations fail: whichever request the caller's allocator refuses, the
context has no cloud afterwards (a build is refused), and the calls repeated on it give the bits of an
undisturbed context."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube
from test_gpu_failed_allocations import _Refusing

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("loaded", [False, True])
def test_a_refused_cloud_leaves_no_cloud(loaded):
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(60, 5.0, seed=5)
    old = cloud_uniform_cube(20, 4.0, seed=6)
    inc = np.array([[0.3, 0.2, 0.1]])

    def load(ctx, c):
        return swm.swm_set_cloud(ctx, c.centres, c.dirs, c.lengths, c.radii, c.nseg)

    def result(ctx):
        swm.swm_build(ctx, K, 2.0, swm.SWM_C64)
        x = np.zeros((1, cl.n_unknowns), dtype=np.complex128)
        swm.swm_solve(ctx, inc, 1e-5, 20, 100, x)
        return x

    want = None
    for k in (None, 0, 1, 2, 3, 4, 5):
        ctx = swm.swm_create(0, torch_allocator=False)
        try:
            mem = _Refusing(swm, ctx)
            if loaded:  # buffers of another cloud lie in the context's list of released ones
                load(ctx, old)
                swm.swm_build(ctx, K, 2.0, swm.SWM_C64)
            mem.next_refused(k)
            if k is None:
                load(ctx, cl)
                want = result(ctx)
                continue
            try:
                load(ctx, cl)
            except swm.SwmError as e:
                assert e.code == swm.SWM_ENOMEM
                mem.next_refused(None)
                with pytest.raises(swm.SwmError) as err:
                    swm.swm_build(ctx, K, 2.0, swm.SWM_C64)
                assert err.value.code == swm.SWM_ESTATE
                load(ctx, cl)
            else:
                assert mem.times == 2  # served from released buffers
                mem.next_refused(None)
            assert np.array_equal(result(ctx), want)
        finally:
            swm.swm_destroy(ctx)
