"""Helmholtz at the high orders: complex box vectors of 592 real entries (p = 8), longer than any real
kernel's, through every FP16-plane contraction (fp16x3) and the three-plane M2L (fp32).  (p = 10 and p = 8
at depth 4 run the same way; their operators take minutes of host time.)

Reference: the FP64 context of the same operators, whose compressed vectors are too long for the digit
products: SIMT arithmetic.  Tolerance: the parity bar, 1e-5 of the potentials and of every level's check rows.
"""
import pytest
import torch

from gpu_helpers import rel
from synth import charges, sphere_points

pytestmark = pytest.mark.gpu


def test_matches_fp64():
    import paper_2604_19243_gb300 as pkg
    n, p, depth, precisions = 3001, 8, 3, ("fp32", "fp16x3")
    x = torch.from_numpy(sphere_points(n)).cuda()
    q = torch.complex(torch.from_numpy(charges(n, "u11")).cuda(), torch.from_numpy(charges(n, "u01")).cuda())
    out, rows = {}, {}
    for prec in ("fp64",) + precisions:
        f = pkg.FMM(p=p, depth=depth, precision=prec, domain=((-1.0, -1.0, -1.0), 2.0), kernel="helmholtz", kappa=2.0)
        f.build_tree(x.double() if prec == "fp64" else x).precompute()
        out[prec] = f.evaluate(q.to(torch.complex128) if prec == "fp64" else q)[0].cpu()
        rows[prec] = {(level, kind): f.export_check(level, kind) for level in range(2, depth + 1)
                      for kind in ("upward", "downward")}
        f.sync()
        f.close()
    for prec in precisions:
        for at, want in rows["fp64"].items():
            assert rel(rows[prec][at], want) < 1e-5, (prec, at)
        assert rel(out[prec], out["fp64"]) < 1e-5, prec
