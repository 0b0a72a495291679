"""FP64 pixel products at the edges of their 16 x 16 tiles and 64-row blocks: J a
(symmetric: tiles on and above the diagonal), the data projection (all tiles), J^H b
and the adjoint sources (through the gradient), against the definitions on the
device's own fields (Eq. 4, 15-17).

Tolerance: sums of at most 1024 FP64 products, 1024 x 1.1e-16; 1e-11 (gradient:
the solves' 1e-12, amplified)."""
import numpy as np
import pytest

from gpu_common import contrast, oracle_problem, rel_l2, to_gpu, to_np
from oracle import inverse
from paper_2604_15796_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_elem,freqs", [(1, (2e6,)), (15, (1e6, 2e6)), (16, (2e6,)),
                                          (17, (1e6, 2e6, 3e6)), (33, (2e6,)), (65, (1e6, 2e6))])
def test_f64_products_match_definitions(n_elem, freqs):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = phantoms.scaled((16, 64), 0.1e-3, n_elem, 5.5e-3 / n_elem, np.array(freqs), 11,
                        inclusions=[1520.0, 1580.0], semi_mm=(0.2, 0.5))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs, precision=libfwi.FWI_FP64,
                         tol=1e-12)
    m = to_gpu(contrast(w), torch.complex128)
    a = phantoms.complex_normal(w.shape, 5)
    b = phantoms.complex_normal((w.n_freq, n_elem, n_elem), 6)
    f, data = ctx.empty_fields(), ctx.empty_data()
    ctx.forward(m, fields=f, data=data)
    ja = to_np(ctx.jac_forward(to_gpu(a, torch.complex128)))
    jhb = to_np(ctx.jac_adjoint(to_gpu(b, torch.complex128)))
    grad = torch.empty(w.shape, dtype=torch.complex128, device="cuda")
    ctx.gradient(m, torch.zeros_like(data), grad)
    ctx.close()
    prob, p = oracle_problem(w), to_np(f)
    k = 2 * np.pi * np.asarray(w.freqs) / w.c0
    q = p * (k ** 2 * w.h ** w.dim).reshape(-1, 1, 1, 1)
    assert rel_l2(ja, inverse.jac_forward(a, p, q, prob)) < 1e-11
    assert rel_l2(jhb.ravel(), inverse.jac_adjoint(b, p, q, prob).ravel()) < 1e-11
    assert rel_l2(to_np(data), inverse.forward_data(contrast(w), p, prob)) < 1e-11
    assert rel_l2(to_np(grad).ravel(),
                  inverse.jac_adjoint(to_np(data), p, q, prob).ravel()) < 1e-9
