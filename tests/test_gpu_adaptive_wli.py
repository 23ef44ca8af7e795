"""The W and X list kernels at the sizes where their work is divided differently: leaves of up to 8, 16, 32
and 64 points and of more than 64 (two passes), p = 2 (8 surface points, fewer than a warp) to p = 8 (296,
more than one staged chunk).  Against the FP64 adaptive oracle at the same p: the
FP64 tolerance is rounding and the M2L compression only (1e-8); FP32 potentials 1e-5, gradients 1e-4."""
import numpy as np
import pytest
import torch

from gpu_helpers import make_fmm, rel
from oracle import adaptive as ad
from synth import charges, mixed_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("capacity,p", [(5, 4), (14, 6), (30, 2), (60, 7), (150, 4), (90, 8)])
def test_w_and_x_lists(capacity, p, precision):
    n, depth, dom = 4000, 6, ((0.0, 0.0, 0.0), 1.0)
    x, q = mixed_points(n), charges(n, "u11")
    f = make_fmm(x, p, depth, precision, dom)
    f.adaptive_setup(capacity)
    dt = torch.float64 if precision == "fp64" else torch.float32
    phi, grad = f.adaptive_evaluate(torch.from_numpy(q).to("cuda", dt))
    o_phi, o_grad, _, il = ad.evaluate(x.astype(np.float64), q.astype(np.float64), p, capacity, depth, *dom)
    assert sum(len(m) for m in il.w.values()) > 0 and il.x
    tp, tg = (1e-8, 1e-8) if precision == "fp64" else (1e-5, 1e-4)
    e = rel(phi.cpu().numpy(), o_phi), rel(grad.cpu().numpy(), o_grad)
    assert e[0] < tp and e[1] < tg, e
    f.close()
