"""The contractions from FP16 planes (three planes under fp32's M2L, two under fp16x3) at the edges of
their tiles: orders whose box vectors fill one CTA, several, and a ragged last chunk; trees whose
levels hold fewer boxes than a tile, more, and remainders.

Reference: the FP64 context of the same points (SIMT arithmetic, itself held to the oracle).
Tolerance: the parity bars, 1e-5 of the potential and of every level's check rows; the planes hold
2^-22 (fp16x3) and 2^-33 (fp32) of an entry, and FP32 sums of at most 189 x 488 terms add about
sqrt(189 x 488) 2^-24 = 2e-5 in the worst (fully cancelling) direction, far less in the norm.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import rel
from synth import charges, cube_points, sphere_points

pytestmark = pytest.mark.gpu
BOX = ((-1.0, -1.0, -1.0), 2.0)
CUBE = ((0.0, 0.0, 0.0), 1.0)


def contexts(p, depth, dist, n, **kw):
    import paper_2604_19243_gb300 as pkg
    x = cube_points(n) if dist == "cube" else sphere_points(n)
    q = charges(n, "u11")
    out = []
    for prec in ("fp64", kw.pop("precision")):
        f = pkg.FMM(p=p, depth=depth, precision=prec, domain=CUBE if dist == "cube" else BOX, **kw)
        dt = torch.float64 if prec == "fp64" else torch.float32
        f.build_tree(torch.from_numpy(x).cuda().to(dt)).precompute()
        out.append((f, torch.from_numpy(q).cuda().to(dt)))
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp16x3"])
@pytest.mark.parametrize("p,depth,dist,n", [(2, 2, "cube", 7), (3, 3, "sphere", 301), (4, 4, "cube", 9001),
                                            (5, 3, "cube", 129), (6, 2, "cube", 1000), (6, 5, "sphere", 20001),
                                            (6, 6, "sphere", 9001), (7, 3, "cube", 4001), (8, 4, "sphere", 6001),
                                            (10, 3, "cube", 2001)])
def test_levels_and_outputs_match_fp64(precision, p, depth, dist, n):
    (d, qd), (f, qf) = contexts(p, depth, dist, n, precision=precision)
    want, _ = d.evaluate(qd)
    got, _ = f.evaluate(qf)
    assert rel(got.cpu(), want.cpu()) < 1e-5
    for level in range(2, depth + 1):
        for kind in ("upward", "downward"):
            w, g = d.export_check(level, kind), f.export_check(level, kind)
            if np.linalg.norm(w) > 0:
                assert rel(g, w) < 1e-5, (level, kind)
    psi, _ = f.adjoint(qf)
    want, _ = d.adjoint(qd)
    assert rel(psi.cpu(), want.cpu()) < 1e-5
    f.sync()


@pytest.mark.parametrize("precision", ["fp32", "fp16x3"])
@pytest.mark.parametrize("k", [-60, -20, 20, 60])
def test_power_of_two_charges_scale_exactly(precision, k):
    """Every scale is a power of two, so charges times 2^k give outputs times 2^k, bit for bit."""
    (_, _), (f, q) = contexts(6, 3, "cube", 3001, precision=precision)
    a, ga = f.evaluate(q)
    b, gb = f.evaluate(q * 2.0 ** k)
    assert torch.equal(b, a * 2.0 ** k) and torch.equal(gb, ga * 2.0 ** k)


@pytest.mark.parametrize("precision", ["fp32", "fp16x3"])
def test_zero_and_non_finite_charges(precision):
    (_, _), (f, q) = contexts(6, 4, "sphere", 4001, precision=precision)
    ref, _ = f.evaluate(q)
    phi, _ = f.evaluate(torch.zeros_like(q))
    assert torch.count_nonzero(phi) == 0
    for bad in (float("inf"), float("nan")):
        r = q.clone()
        r[17] = bad
        phi, _ = f.evaluate(r)
        assert not torch.isfinite(phi).any()      # every target sees every charge
    phi, _ = f.evaluate(q)                         # nothing of it stays behind
    assert torch.equal(phi, ref)
