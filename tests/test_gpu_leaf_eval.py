"""The FP32 evaluation at the leaves where a block takes several leaves: 8 (few points each, mostly one or
two), 8 again within its shared memory limit (p = 8), 3, and 1, ragged ends, potentials or gradients alone, the
adaptive tree's rows.  Every point's sum is the same whatever the grouping, so the far part in FP32 is held
against the FP64 evaluation: potentials 1e-5, gradients 1e-4 relative L2."""
import numpy as np
import pytest
import torch

import paper_2604_19243_gb300 as pkg
from gpu_helpers import make_fmm, rel
from synth import charges, cube_points, mixed_points, sphere_points

pytestmark = pytest.mark.gpu


def _pair(x, p, depth, dom, capacity=None):
    q = charges(len(x), "u11")
    out = []
    for precision, dt in (("fp32", torch.float32), ("fp64", torch.float64)):
        f = make_fmm(x, p, depth, precision, dom)
        qd = torch.from_numpy(q).to("cuda", dt)
        if capacity:
            f.adaptive_setup(capacity)
            out.append([v.cpu().numpy() for v in f.adaptive_evaluate(qd)])
        else:
            phi, grad = f.evaluate(qd)
            g_only = f.evaluate(qd, potential=False)[1]
            p_only = f.evaluate(qd, gradient=False)[0]
            assert torch.equal(g_only, grad) and rel(p_only.cpu().numpy(), phi.cpu().numpy()) < 2e-6
            out.append([phi.cpu().numpy(), grad.cpu().numpy()])
        f.close()
    return rel(out[0][0], out[1][0]), rel(out[0][1], out[1][1])


@pytest.mark.parametrize("dist,n,p,depth", [("sphere", 20_001, 4, 6), ("cube", 60_001, 6, 4), ("cube", 50_003, 8, 4),
                                            ("cube", 150_007, 2, 4), ("cube", 20_003, 5, 2)])
def test_grouped_leaves(dist, n, p, depth):
    x = cube_points(n) if dist == "cube" else sphere_points(n)
    e = _pair(x, p, depth, ((0, 0, 0), 1.0) if dist == "cube" else ((-1, -1, -1), 2.0))
    assert e[0] < 1e-5 and e[1] < 1e-4, e


def test_grouped_rows():
    e = _pair(mixed_points(60_000), 4, 7, ((0, 0, 0), 1.0), capacity=20)
    assert e[0] < 1e-5 and e[1] < 1e-4, e
