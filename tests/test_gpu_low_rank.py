"""FP16X3 with M2L operators of low rank: the compressed vectors then fill one 64-column chunk while the
box vectors of the same contraction (the decompress joined with D2D) fill several, each with its own scale.

Reference: the FP64 context of the same tolerance, hence of the same ranks and operators.  Tolerance: the
parity bar, 1e-5, of every level's check rows (the planes hold 2^-22 of an entry).  The outputs follow from
them by the FP32 closing in every mode: at svd_rtol 0.1 the rows are no smooth field, and the closing's
pseudo-inverse enlarges rounding errors to 1e-3 of the potentials, in FP32 SIMT arithmetic as well.  So an
output may be off by 1e-5 or by twice what the FP32 context's is, whichever is more.
"""
import pytest
import torch

from gpu_helpers import rel
from synth import charges, cube_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,svd_rtol", [(5, 1e-2), (6, 1e-3), (7, 0.1), (7, 1e-4), (8, 0.2), (8, 1e-4)])
def test_low_rank_matches_fp64(p, svd_rtol):
    import paper_2604_19243_gb300 as pkg
    n, depth = 6001, 4
    x, q = torch.from_numpy(cube_points(n)).cuda(), torch.from_numpy(charges(n, "u11")).cuda()
    out, rows = {}, {}
    for prec, dt in (("fp64", torch.float64), ("fp32", torch.float32), ("fp16x3", torch.float32)):
        f = pkg.FMM(p=p, depth=depth, precision=prec, domain=((0.0, 0.0, 0.0), 1.0), svd_rtol=svd_rtol)
        f.build_tree(x.to(dt)).precompute()
        phi = f.evaluate(q.to(dt))[0].cpu()
        rows[prec] = {(level, kind): f.export_check(level, kind) for level in range(2, depth + 1)
                      for kind in ("upward", "downward")}
        out[prec] = {"evaluate": phi, "adjoint": f.adjoint(q.to(dt))[0].cpu()}
        f.sync()
    for at, want in rows["fp64"].items():
        assert rel(rows["fp16x3"][at], want) < 1e-5, at
    for call, want in out["fp64"].items():
        assert rel(out["fp16x3"][call], want) < max(1e-5, 2 * rel(out["fp32"][call], want)), call
