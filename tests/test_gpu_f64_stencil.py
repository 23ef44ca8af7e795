"""The FP64 M2L from integer digits (gemm_f64.cu) at the edges of its tiles: one to five CTAs across the
output columns, ranks of one to many 16-value chunks, levels of fewer boxes than a tile and of more.

A and its transpose run with operators that are cut into digits independently, so that the identity
<A q, g> = <q, A^T g> holds to the rounding of the two passes: at most 189 x 296 products a box, added
in FP64, sqrt(189 x 296) 2^-53 = 2.6e-14 of |A q| |g| if every one were rounded at random.  Charges
times a power of two give the same bits: every exponent is taken off before the digits.
"""
import numpy as np
import pytest
import torch

import paper_2604_19243_gb300 as pkg
from gpu_helpers import rel
from synth import charges, cube_points, sphere_points

pytestmark = pytest.mark.gpu
CUBE, BALL = ((0.0, 0.0, 0.0), 1.0), ((-1.0, -1.0, -1.0), 2.0)


def context(p, depth, dist, n, **kw):
    x = cube_points(n) if dist == "cube" else sphere_points(n)
    f = pkg.FMM(p=p, depth=depth, precision="fp64", domain=CUBE if dist == "cube" else BALL, **kw)
    f.build_tree(torch.from_numpy(x).cuda().double()).precompute()
    return f, torch.from_numpy(charges(n, "u11")).cuda().double()


@pytest.mark.parametrize("p,depth,dist,n", [(2, 2, "cube", 9), (3, 4, "sphere", 2001), (4, 3, "cube", 1025),
                                            (6, 2, "cube", 130), (6, 5, "sphere", 8001), (7, 3, "sphere", 3001),
                                            (8, 3, "cube", 2001)])
def test_transpose_identity_and_scaling(p, depth, dist, n):
    f, q = context(p, depth, dist, n)
    g = torch.from_numpy(charges(n, "normal", seed=2)).cuda().double()
    phi, _ = f.evaluate(q, gradient=False)
    psi, _ = f.adjoint(g)
    gap = abs(float(torch.dot(phi, g) - torch.dot(q, psi))) / float(phi.norm() * g.norm())
    assert gap < 2.6e-14
    for k in (-300, 300):
        big, _ = f.evaluate(q * 2.0 ** k, gradient=False)
        assert torch.equal(big, phi * 2.0 ** k)
    f.sync()


def test_helmholtz_rows_match_the_direct_sum_of_the_other_precision():
    """304-entry real forms (19 chunks of K): the FP32 context, whose M2L is computed otherwise, agrees
    to FP32 accuracy."""
    n, kw = 3001, dict(kernel="helmholtz", kappa=2.0)
    x = torch.from_numpy(sphere_points(n)).cuda()
    q = torch.from_numpy(charges(n, "u11") + 1j * charges(n, "u11", seed=101)).cuda()
    out = []
    for prec, dt, ct in (("fp64", torch.float64, torch.complex128), ("fp32", torch.float32, torch.complex64)):
        f = pkg.FMM(p=6, depth=3, precision=prec, domain=BALL, **kw)
        f.build_tree(x.to(dt)).precompute()
        out.append(f.evaluate(q.to(ct), gradient=False)[0].cpu().numpy())
    assert rel(out[1], out[0]) < 1e-5


def test_zero_and_non_finite_charges():
    f, q = context(6, 3, "sphere", 2001)
    ref, _ = f.evaluate(q, gradient=False)
    assert torch.count_nonzero(f.evaluate(torch.zeros_like(q), gradient=False)[0]) == 0
    r = q.clone()
    r[5] = float("nan")
    assert not torch.isfinite(f.evaluate(r, gradient=False)[0]).any()
    assert torch.equal(f.evaluate(q, gradient=False)[0], ref)
