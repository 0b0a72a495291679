"""Operand tiles of the tensor-core contractions cut to the elements there are:
element counts at the edges of the 8-row blocks, of one and of two tiles, for J a,
J^H b and the adjoint sources, with the operand tiles filled by TMA and by
cp.async.

Reference: the definitions (Eq. 15-17) in FP64 on the device's own fields.
Tolerance: the accumulators are FP32 chains of at most 256 terms (J^H; 512 pixels
for J a), each step off by at most 2^-23, so at most 6e-5 of the terms' size."""
import numpy as np
import pytest

from gpu_common import contrast, oracle_problem, rel_l2, to_gpu, to_np
from oracle import inverse
from paper_2604_15796_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_elem", [1, 8, 9, 61, 64, 65, 127, 129, 192, 250])
def test_contraction_tiles_follow_the_elements(n_elem):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = phantoms.scaled((16, 64), 0.1e-3, n_elem, 5.5e-3 / n_elem, np.array([1.0e6, 2.5e6]), 11,
                        inclusions=[1520.0, 1580.0], semi_mm=(0.2, 0.5))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    m = to_gpu(contrast(w), torch.complex128)
    a = phantoms.complex_normal(w.shape, 5)
    b = phantoms.complex_normal((w.n_freq, n_elem, n_elem), 6)
    zero = torch.zeros((w.n_freq, n_elem, n_elem), dtype=torch.complex64, device="cuda")
    out = {}
    for tma in (True, False):
        ctx.set_jac_tma(tma)
        f, data = ctx.empty_fields(), ctx.empty_data()
        ctx.forward(m, fields=f, data=data)
        out[tma] = [to_np(ctx.jac_forward(to_gpu(a, torch.complex128))),
                    to_np(ctx.jac_adjoint(to_gpu(b, torch.complex128))), to_np(data)]
        # d_obs = 0: the adjoint sources carry the data themselves
        grad = torch.empty(w.shape, dtype=torch.complex128, device="cuda")
        ctx.gradient(m, zero, grad)
        out[tma].append(to_np(grad))
    ctx.close()
    for x, y in zip(out[True], out[False]):
        assert np.array_equal(x, y)
    ja, jhb, data, grad = out[True]
    prob = oracle_problem(w)
    p = to_np(f).astype(np.complex128)
    k = 2 * np.pi * np.asarray(w.freqs) / w.c0
    q = p * (k ** 2 * w.h ** w.dim).reshape(-1, 1, 1, 1)
    assert rel_l2(ja, inverse.jac_forward(a, p, q, prob)) < 6e-5
    assert rel_l2(jhb.ravel(), inverse.jac_adjoint(b, p, q, prob).ravel()) < 6e-5
    assert rel_l2(data, inverse.forward_data(contrast(w), p, prob)) < 1e-4
    assert rel_l2(grad.ravel(), inverse.jac_adjoint(data, p, q, prob).ravel()) < 1e-3
