"""Inner products of the BiCGSTAB passes for every row length: lines of 4 to 64
threads (reduce-scatter inside a warp, two warps, and the shared-memory sums of 20-
and 24-thread lines with ragged CTAs).  A wrong partial sum changes the step
lengths, so the solves are compared with the oracle's and the reported residuals
with those of the returned fields.

Tolerances: fields 1e-4 (FP32) and 1e-8 (FP64, solved to 1e-10); the recursive
residual agrees with the true one to FP32 rounding of a few iterations."""
import numpy as np
import pytest

from gpu_common import contrast, oracle_problem, rel_l2, small_workload, to_gpu, to_np
from oracle import operator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 8), (8, 16), (8, 32), (8, 64), (16, 96), (8, 128),
                                   (16, 160), (32, 192), (8, 256), (8, 320), (8, 384), (8, 512),
                                   (8, 16, 160), (8, 8, 192)])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_solves_for_every_row_length(shape, prec):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = small_workload(shape, n_elem=3, freqs=(1.5e6, 3.0e6))
    fp64 = prec == "fp64"
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs, tol=1e-10 if fp64 else 1e-6,
                         precision=libfwi.FWI_FP64 if fp64 else libfwi.FWI_MIXED)
    m = contrast(w)
    f = ctx.empty_fields()
    rep = ctx.forward(to_gpu(m, torch.complex128), fields=f)
    ctx.close()
    got = to_np(f).astype(np.complex128)
    prob = oracle_problem(w)
    ref = operator.solve_forward(m, prob, "bicgstab", tol=1e-12)
    assert rel_l2(got, ref) < (1e-8 if fp64 else 1e-4)
    assert rep.max_iters >= 2 and np.all(rep.rel_resid <= (1e-10 if fp64 else 1e-6))
    for l in range(w.n_freq):
        b = operator.apply_A(ref[l], m, prob, l)
        r = b - operator.apply_A(got[l], m, prob, l)
        for e in range(w.n_elem):
            true = np.linalg.norm(r[e]) / np.linalg.norm(b[e])
            assert true < (2e-10 if fp64 else 3e-6), (l, e, true)
