"""Ranges of several items per CTA in the two-column convolution, at every transform
length: 750 right-hand sides over 8 or more column tiles leave each CTA at least
three, so that input tiles are staged behind one another (beside the exchange or
inside it), a kept spectrum tile serves many right-hand sides, and ranges cross from
one frequency and one column tile to the next (spectra in one, two and three boxes).

Every right-hand side against one column per thread: single applications to the
FP32 rounding of two transforms of length L (3.8e-7 in quadrature, 1.4 times that
between two evaluations: 1e-6), whole solves, which stop at 1e-6, to 1e-5.  A wrong
tile or frequency changes a right-hand side by the order of its own size."""
import numpy as np
import pytest

from gpu_common import contrast, small_workload, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 128), (16, 128), (32, 128), (64, 64), (96, 64), (128, 64),
                                   (160, 64), (192, 64), (256, 128), (320, 64), (384, 64),
                                   (512, 64), (32, 16, 32), (96, 8, 32), (256, 8, 16)])
def test_every_right_hand_side_of_long_ranges(shape):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    n_elem = 250
    w = small_workload(shape, n_elem=n_elem, pitch=0.08e-3 * shape[-1] / n_elem,
                       freqs=(1.5e6, 2.0e6, 3.5e6))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    assert ctx.n_rhs == 3 * n_elem
    m = to_gpu(contrast(w), torch.complex128)
    gen = torch.Generator(device="cuda").manual_seed(3)
    v = torch.randn((3 * n_elem,) + tuple(shape), generator=gen, device="cuda",
                    dtype=torch.complex64)
    out = {}
    for pairs in (True, False):
        ctx.set_col_pairs(pairs)
        f = ctx.empty_fields()
        ctx.forward(m, fields=f)
        out[pairs] = [ctx.apply("A", v, 1, m).reshape(len(v), -1), f.reshape(len(v), -1)]
    ctx.close()
    for x, y, tol in zip(out[True], out[False], (1e-6, 1e-5)):
        err = torch.linalg.norm(x - y, dim=1) / torch.linalg.norm(y, dim=1)
        assert float(err.max()) < tol, (int(err.argmax()), float(err.max()))
