"""Contexts whose M2L has planes or digits beside its rows, where there is memory for the rows alone: the
evaluation runs in SIMT arithmetic instead of failing.  The limit (on one allocation, 16 MB) lies below the
partial sums of the coarse levels' groups (26 and 25 MB here) and above every other array.

Reference: the same context without a limit.  Tolerance: 1e-12 in FP64 (56-bit digits against FP64 products);
1e-5, the parity bar, in FP32.
"""
import pytest
import torch

from gpu_helpers import rel
from synth import charges, cube_points, mixed_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,call,depth", [("fp64", "evaluate", 4), ("fp64", "adjoint", 4), ("fp32", "adaptive", 6)])
def test_rows_alone_are_enough(precision, call, depth):
    import paper_2604_19243_gb300 as pkg
    n, dt = 40_000, torch.float64 if precision == "fp64" else torch.float32
    x = torch.from_numpy(mixed_points(n) if call == "adaptive" else cube_points(n)).cuda().to(dt)
    q = torch.from_numpy(charges(n, "u11")).cuda().to(dt)
    out = []
    for limit in (None, 16 << 20, None):
        f = pkg.FMM(p=4, depth=depth, precision=precision, domain=((0.0, 0.0, 0.0), 1.0)).build_tree(x).precompute()
        if call == "adaptive":
            f.adaptive_setup(16)
        try:
            pkg.set_alloc_limit(limit)
            r = f.adaptive_evaluate(q) if call == "adaptive" else getattr(f, call)(q)
            f.sync()
        finally:
            pkg.set_alloc_limit(None)
        out.append([v.cpu() for v in r if v is not None])
        f.close()
    for full, scarce, again in zip(*out):
        assert rel(scarce, full) < (1e-12 if precision == "fp64" else 1e-5)
        assert torch.equal(full, again) and not torch.equal(full, scarce)   # the limit did take the other route
