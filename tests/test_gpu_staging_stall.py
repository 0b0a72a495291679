"""A convolution whose staged spectrum never completes (debug_stall_once: the copy's
barrier expects 16 bytes more than arrive) gives up its bounded wait, waits, again
bounded, for the copy it has in flight, reports the error and leaves the context
usable.  Both limits are 1 s, so a CTA that left without the second wait, its
copy still in flight, would return in half the time: checked where the wait that
gives up is the CTA's last (one item) and where other items follow."""
import time

import numpy as np
import pytest

from gpu_common import contrast, small_workload, to_gpu, to_np
from paper_2604_15796_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rhs", [3, 600])
@pytest.mark.parametrize("pairs", [True, False])
def test_stalled_spectrum_copy_is_waited_for(pairs, n_rhs):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = small_workload((64, 32), n_elem=100, pitch=0.03e-3, freqs=np.linspace(1e6, 3e6, 6))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    ctx.set_col_pairs(pairs)
    m = to_gpu(contrast(w), torch.complex128)
    v = to_gpu(phantoms.complex_normal((n_rhs,) + tuple(w.shape), 3), torch.complex64)
    ref = to_np(ctx.apply("A", v, 1, m))
    ctx.debug_stall_once()
    t0 = time.perf_counter()
    to_np(ctx.apply("A", v, 1, m))
    waited = time.perf_counter() - t0
    with pytest.raises(libfwi.FwiError) as err:
        ctx.forward(m)
    assert err.value.status == libfwi.FWI_ERR_CUDA
    assert "column pass TMA staging: pipeline wait timed out (code 5)" in str(err.value)
    assert 1.9 < waited < 4.0, waited
    assert np.array_equal(to_np(ctx.apply("A", v, 1, m)), ref)
    assert ctx.forward(m).info.n_not_converged == 0
    ctx.close()


@pytest.mark.parametrize("tma", [True, False])
@pytest.mark.parametrize("n_elem", [61, 129])
def test_stalled_contraction_leaves_no_copy_behind(n_elem, tma):
    """The contraction (54 and 216 k-steps per CTA) and J^H (32 and 119, B blocks by
    bulk copies) stall at their first stage with their rings of raw tiles full: the
    waits run out once (1 s), no tile is issued again while its copy is pending,
    every copy in flight is seen to land (a second limit would double the time), and
    the next calls give the same bits."""
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = phantoms.scaled((256, 256), 0.1e-3, n_elem, 25e-3 / n_elem, np.array([1.0e6]), 11,
                        inclusions=[1520.0, 1580.0])
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    ctx.set_jac_tma(tma)
    m = to_gpu(contrast(w), torch.complex128)
    ctx.forward(m)
    a = to_gpu(phantoms.complex_normal(w.shape, 5), torch.complex128)
    b = to_gpu(phantoms.complex_normal((1, n_elem, n_elem), 6), torch.complex128)
    grad = torch.empty(w.shape, dtype=torch.complex128, device="cuda")
    zero = torch.zeros((1, n_elem, n_elem), dtype=torch.complex64, device="cuda")
    calls = {"J a": lambda: to_np(ctx.jac_forward(a)), "J^H b": lambda: to_np(ctx.jac_adjoint(b))}
    ref = {k: f() for k, f in calls.items()}
    for k, f in calls.items():
        ctx.debug_stall_once()
        t0 = time.perf_counter()
        f()
        waited = time.perf_counter() - t0
        with pytest.raises(libfwi.FwiError) as err:
            ctx.forward(m)
        assert "tensor-core contraction: pipeline wait timed out" in str(err.value)
        assert 0.9 < waited < 1.8, (k, waited)
        ctx.gradient(m, zero, grad)
        for k2, f2 in calls.items():
            assert np.array_equal(f2(), ref[k2]), (k, k2)
    ctx.close()


def test_adjoint_reports_a_wait_that_gave_up():
    """The error word is reported by the next call that synchronises, the adjoint
    solve among them."""
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = small_workload((32, 32), n_elem=6)
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    m = to_gpu(contrast(w), torch.complex128)
    v = to_gpu(phantoms.complex_normal((w.n_freq, 6) + tuple(w.shape), 3), torch.complex64)
    ref = ctx.empty_fields()
    ctx.adjoint(m, v, ref)
    ctx.debug_stall_once()
    ctx.apply("K", v[0], 0)
    lam = ctx.empty_fields()
    with pytest.raises(libfwi.FwiError) as err:
        ctx.adjoint(m, v, lam)
    assert err.value.status == libfwi.FWI_ERR_CUDA
    assert "column pass TMA staging: pipeline wait timed out" in str(err.value)
    ctx.adjoint(m, v, lam)
    ctx.close()
    assert torch.equal(lam, ref)
