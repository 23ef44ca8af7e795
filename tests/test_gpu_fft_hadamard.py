"""The products of the FFT M2L at the edges of their blocks: parents that do not fill a warp's group or a
CTA's, frequencies that do not fill a slice of 32 (p = 5, 7, 9: 600, 1568 and 3240 in all), mostly empty neighbourhoods.
Compared with the FP64 oracle's own FFT M2L; tolerances as for the whole FFT form: FP32 potentials 1e-5 and
gradients 1e-4 relative L2, FP64 1e-8."""
import numpy as np
import pytest

from oracle import fft_m2l, kifmm
from synth import charges
from gpu_helpers import PINV_RTOL, make_fmm, rel, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,p,depth,power", [(3_001, 5, 4, 3), (700, 7, 2, 1), (900, 9, 3, 2), (40, 5, 3, 1)])
def test_products_at_block_edges(precision, n, p, depth, power):
    x = (np.random.default_rng(n).random((n, 3)) ** power).astype(np.float32)
    q = charges(n, "u11")
    dom = ((0, 0, 0), 1.0)
    ops = kifmm.build_operators(p, 1.0, depth, PINV_RTOL, alpha_inner=fft_m2l.lattice_alpha(p))
    ref = kifmm.evaluate(x.astype(np.float64), q.astype(np.float64), p, depth, *dom, pinv_rtol=PINV_RTOL, ops=ops, m2l="fft")
    f = make_fmm(x, p, depth, precision, dom, m2l="fft")
    phi, grad = run(f, q)
    f.sync()
    f.close()
    tp, tg = (1e-5, 1e-4) if precision == "fp32" else (1e-8, 1e-8)
    assert rel(phi, ref.phi) < tp and rel(grad, ref.grad) < tg, (rel(phi, ref.phi), rel(grad, ref.grad))
