"""Two columns per thread with the kernel spectrum read from L2
(col_spectrum_stage = 0; transform lengths 16, 64, 256 and 512): the same
arithmetic on the same values as with the staged spectrum, in packed instructions
that nothing fuses, so single applications, whole solves and ranges of several
items per CTA across a frequency boundary give the same bits."""
import numpy as np
import pytest

from gpu_common import contrast, small_workload, to_gpu, to_np
from paper_2604_15796_gb300 import phantoms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n_elem", [((8, 32), 5), ((32, 64), 300), ((128, 32), 300),
                                          ((256, 16), 300), ((32, 16, 16), 9)])
def test_spectrum_from_l2_gives_the_staged_bits(shape, n_elem):
    import torch
    from paper_2604_15796_gb300 import build, libfwi
    build.build()
    w = small_workload(shape, n_elem=n_elem, pitch=0.08e-3 * shape[-1] / n_elem,
                       freqs=(1.5e6, 2.0e6, 3.5e6))
    ctx = libfwi.Context(w.shape, w.h, w.c0, w.elem, w.freqs)
    m = to_gpu(contrast(w), torch.complex128)
    v = to_gpu(phantoms.complex_normal((3 * n_elem,) + tuple(shape), 31), torch.complex64)
    out = {}
    for stage in (True, False):
        ctx.set_col_spectrum_stage(stage)
        assert ctx.tuning()["col_pairs"] == 1
        f = ctx.empty_fields()
        ctx.forward(m, fields=f)
        out[stage] = [to_np(ctx.apply(k, v, 1, None if k == "K" else m))
                      for k in ("K", "A", "AH")] + [to_np(f)]
    ctx.close()
    for x, y in zip(out[True], out[False]):
        assert np.array_equal(x, y)
