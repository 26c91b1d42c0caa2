"""GPU test of the float64 products without the table of their wire order: an allocator that refuses the
table's bytes leaves the product its value, and no error text behind."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rhs", [1, 3])
@pytest.mark.parametrize("prec", [0, 1])
def test_product_without_the_order(prec, n_rhs):
    import torch
    from paper_2410_03060_gb300 import swm

    nw = 7001
    table = (4 * nw + 255) // 256 * 256
    cl = cloud_uniform_cube(nw, 40.0, seed=1)
    rng = np.random.default_rng(0)
    x = rng.standard_normal((n_rhs, cl.n_unknowns)) + 1j * rng.standard_normal((n_rhs, cl.n_unknowns))
    out = []
    for refuse in (False, True):
        ctx = swm.swm_create(0, torch_allocator=False)
        state = {"armed": False, "once": False, "table": 0}

        def alloc(nbytes, stream, user):
            if state["armed"] and not state["once"]:
                state["once"] = True  # refused once: the context gives its spare buffers back and asks again
                return None
            if state["armed"] and int(nbytes) == table:
                state["table"] += 1
                return None
            return torch.cuda.caching_allocator_alloc(int(nbytes), ctx.device, stream or 0)

        def free(ptr, nbytes, stream, user):
            torch.cuda.caching_allocator_delete(ptr)

        fns = swm.ALLOC_FN(alloc), swm.FREE_FN(free)
        try:
            assert swm.load().swm_set_allocator(ctx.handle, fns[0], fns[1], None) == swm.SWM_OK
            swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
            swm.swm_build(ctx, K, 2.0, prec)
            text = swm.swm_last_error(ctx)
            state["armed"] = refuse
            y = np.zeros_like(x)
            swm.swm_apply(ctx, x, y)
            assert (state["table"] > 0) == refuse
            assert swm.swm_last_error(ctx) == text
            state["armed"] = False
            z = np.zeros_like(x)
            swm.swm_apply(ctx, x, z)
            assert np.array_equal(y, z)
            out.append(y)
        finally:
            swm.swm_destroy(ctx)
    assert np.array_equal(out[0], out[1])
