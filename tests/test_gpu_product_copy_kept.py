"""GPU test of what form 76's copy of E leaves behind: when the timed choice takes another form the copy made
for the timing is given back to the allocator, and a copy whose memory is refused leaves neither bytes nor an
error text behind a solve that went well."""
import numpy as np
import pytest

from gpu_helpers import K
from synth import cloud_uniform_cube
from test_gpu_failed_allocations import _Refusing

pytestmark = pytest.mark.gpu


def _solve(nw, side, n_inc, refuse_from=None):
    """(form, bytes held after the solve, requests of the solve by size, error text)"""
    from paper_2410_03060_gb300 import swm

    cl = cloud_uniform_cube(nw, side, seed=nw)
    inc = np.stack([np.linspace(0.1, 3.0, n_inc), np.zeros(n_inc), np.zeros(n_inc)], 1)
    ctx = swm.swm_create(0, torch_allocator=False)
    try:
        mem = _Refusing(swm, ctx)
        swm.swm_set_cloud(ctx, cl.centres, cl.dirs, cl.lengths, cl.radii, cl.nseg)
        swm.swm_set_solver(ctx, "bicgstab")
        swm.swm_build(ctx, K, 2.0, swm.SWM_C64)
        first = len(mem.sizes)
        mem.next_refused(refuse_from)
        x = np.zeros((n_inc, cl.n_unknowns), dtype=np.complex128)
        swm.swm_solve(ctx, inc, 1e-5, 50, 60, x)
        assert np.isfinite(x).all()
        return (swm.swm_get_stats(ctx)["step_rhs_block"], sum(mem.held.values()), mem.sizes[first:],
                swm.swm_last_error(ctx))
    finally:
        swm.swm_destroy(ctx)


def test_a_copy_made_for_the_timing_is_given_back(monkeypatch):
    others = 0
    for nw, side, n_inc in ((300, 14.7, 20), (1000, 22.0, 4), (1000, 22.0, 20), (1000, 60.0, 4)):
        monkeypatch.delenv("SWM_PRODUCT_FORM", raising=False)
        form, held, _, _ = _solve(nw, side, n_inc)
        if form == 76:
            continue
        others += 1
        monkeypatch.setenv("SWM_PRODUCT_FORM", str(form))
        _, forced, _, _ = _solve(nw, side, n_inc)
        monkeypatch.setenv("SWM_PRODUCT_FORM", "76")
        _, packed, _, _ = _solve(nw, side, n_inc)
        # the order of form 75 (32 bytes a wire) and scratch (16) may stay; the copy is 156 bytes a wire and more
        assert held <= forced + 64 * nw + 4096 < packed
    assert others  # short rows: little to gain, and the sort and the copy cost as much as on others


def test_a_refused_copy_leaves_nothing_behind(monkeypatch):
    nw, side, n_inc = 500, 10.0, 9
    monkeypatch.setenv("SWM_PRODUCT_FORM", "75")
    _, base, _, _ = _solve(nw, side, n_inc)
    monkeypatch.setenv("SWM_PRODUCT_FORM", "76")
    form, packed, sizes, err = _solve(nw, side, n_inc)
    assert form == 76 and not err and packed > base
    refused = 0
    for k in range(len(sizes)):
        try:
            form, held, _, err = _solve(nw, side, n_inc, k)
        except Exception:  # a buffer that the solve needs
            continue
        if form == 75:
            refused += 1
            assert held <= base and not err
    assert refused >= 2  # the records and the copy
