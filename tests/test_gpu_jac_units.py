"""Tensor-core products whose CTAs each take many steps: 192 x 192 pixels x 3
frequencies leave J^H and the adjoint sources 5 to 12 pixel tiles per CTA (both
accumulators in turn; at 136 and 192 elements units of 128 and of 8 or 64 rows) and
J a and the data projection 2 to 6 accumulation sub-chunks per CTA.

Reference: the definitions (Eq. 4, 15-17) in FP64 on the device's own fields, at the
homogeneous model, where the adjoint field is the source itself, so that the
gradient for given data is the mix of the adjoint sources and its assembly.
Tolerance: an accumulator takes at most 6 products for each of 64 k-steps, each off
by at most 2^-23 of the sum so far, 384 x 1.2e-7 = 4.6e-5; the three-product
splitting adds 3 x 2^-22 and the FP32 sums over sub-chunks, elements and
frequencies less than 1e-6: 5e-5."""
import numpy as np
import pytest

from gpu_common import rel_l2, to_gpu, to_np
from paper_2604_15796_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tma", [True, False])
@pytest.mark.parametrize("n_elem", [61, 136, 192])
def test_products_over_many_units(n_elem, tma):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = phantoms.scaled((192, 192), 0.1e-3, n_elem, 18e-3 / n_elem,
                        np.array([1.0e6, 1.8e6, 2.5e6]), 11, inclusions=[1520.0, 1580.0])
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    ctx.set_jac_tma(tma)
    zero = torch.zeros(w.shape, dtype=torch.complex128, device="cuda")
    f = ctx.empty_fields()
    a = to_gpu(phantoms.complex_normal(w.shape, 5), torch.complex128)
    b = to_gpu(phantoms.complex_normal((3, n_elem, n_elem), 6), torch.complex64)
    b64 = b.to(torch.complex128)
    grad = torch.empty_like(zero)
    ctx.gradient(zero, -b, grad)  # data 0: the residual is b
    ctx.forward(zero, fields=f)
    ja, jhb = ctx.jac_forward(a), ctx.jac_adjoint(b64)
    m = 1e-3 * a
    fm, data = ctx.empty_fields(), ctx.empty_data()
    ctx.forward(m, fields=fm, data=data)
    ctx.close()
    p = f.reshape(3, n_elem, -1).to(torch.complex128)
    k = 2 * np.pi * torch.tensor(w.freqs, device="cuda", dtype=torch.float64) / w.c0
    q = p * (k ** 2 * w.h ** 2).reshape(3, 1, 1)
    ref_ja = torch.einsum("len,ljn->lej", p * a.reshape(1, 1, -1), q)
    ref_jhb = sum((p[l].conj() * (b64[l] @ q[l].conj())).sum(0) for l in range(3))
    pm = fm.reshape(3, n_elem, -1).to(torch.complex128)
    ref_data = torch.einsum("len,ljn->lej", pm * m.reshape(1, 1, -1), q)
    assert rel_l2(to_np(ja), to_np(ref_ja)) < 5e-5
    assert rel_l2(to_np(jhb).ravel(), to_np(ref_jhb)) < 5e-5
    assert rel_l2(to_np(data), to_np(ref_data)) < 5e-5
    assert rel_l2(to_np(grad).ravel(), to_np(ref_jhb)) < 5e-5
