"""The two-column convolution at every transform length: its plans (radices 2, 3,
5; lines whose threads idle in one phase; input staged beside or inside the
exchange; one to three spectrum boxes), tile counts that leave groups of 8, 4, 2
and 1 tiles, spectrum tiles that change with the frequency inside a CTA's range,
and solves whose active list shrinks.

Tolerance: two FP32 transforms of length L and their inverses round about
4 log2 L <= 40 times at 6e-8 per sample, 3.8e-7 in quadrature; two evaluations
differ by at most 1.4 times that, 1e-6 with a margin of 2.  Against the oracle
1e-5 (single applications) and 1e-4 (fields), as for every FP32 pass."""
import numpy as np
import pytest

from gpu_common import contrast, oracle_problem, rel_l2, small_workload, to_gpu, to_np
from oracle import inverse, operator
from paper_2604_15796_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 32), (16, 8), (32, 96), (64, 16), (96, 64), (128, 8),
                                   (160, 96), (192, 16), (256, 8), (320, 16), (384, 8), (512, 16),
                                   (96, 8, 16), (160, 16, 8)])
def test_every_length_matches_one_column(shape):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = small_workload(shape, n_elem=5, freqs=(1.5e6, 2.0e6, 3.5e6))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    m = contrast(w)
    m_gpu = to_gpu(m, torch.complex128)
    v = phantoms.complex_normal((13,) + tuple(shape), 31)
    v_gpu = to_gpu(v, torch.complex64)
    out = {}
    for pairs in (True, False):
        ctx.set_col_pairs(pairs)
        f = ctx.empty_fields()
        ctx.forward(m_gpu, fields=f)
        out[pairs] = [to_np(ctx.apply(k, v_gpu, 1, None if k == "K" else m_gpu))
                      for k in ("K", "A", "AH")] + [to_np(f)]
    ctx.close()
    for x, y in zip(out[True][:3], out[False][:3]):
        assert rel_l2(x, y) < 1e-6
    assert rel_l2(out[True][3], out[False][3]) < 1e-5  # solves stop at 1e-6
    prob = oracle_problem(w)
    vin = v.astype(np.complex64).astype(np.complex128)
    assert rel_l2(out[True][0], operator.apply_K(vin, prob, 1)) < 1e-5
    assert rel_l2(out[True][2], inverse.apply_AH(vin, m, prob, 1)) < 1e-5
    assert rel_l2(out[True][3], operator.solve_forward(m, prob, "bicgstab", tol=1e-10)) < 1e-4


def test_two_chains_repeat_one_chain():
    """Two chains share SMs, so that one chain's passes run beside the other's
    convolution and delay its shared-memory loads; every right-hand side still
    gets the bits it gets alone (a copy that lands in a staging area before the
    loads from it were performed would change them)."""
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = phantoms.scaled((128, 128), 0.156e-3, 100, 0.2e-3, np.linspace(0.3e6, 2.5e6, 4), 13,
                        inclusions=[1520.0, 1580.0], semi_mm=(1.0, 3.0))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    m = to_gpu(contrast(w), torch.complex128)
    f, ref = ctx.empty_fields(), ctx.empty_fields()
    ctx.set_overlap(False)
    ctx.forward(m, fields=ref)
    ctx.set_overlap(True)
    for _ in range(8):
        ctx.forward(m, fields=f)
        assert torch.equal(f, ref)
    ctx.close()
