"""The FP32 Helmholtz near field where its work is divided differently: leaves of fewer than 32 targets, of
more than 128 (a block's second turn), more than one staged chunk of 1024 sources.  Against the FP64 direct sum over the
same pairs (depth 1: every leaf is a neighbour); FP32 rounding, sincos included: 2e-6."""
import numpy as np
import pytest
import torch

import paper_2604_19243_gb300 as pkg
from gpu_helpers import rel
from oracle import direct
from synth import charges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("outputs", ["both", "grad", "phi"])
@pytest.mark.parametrize("n,power", [(1, 1), (70, 1), (517, 1), (2500, 3)])
def test_near_field_is_the_direct_sum(n, power, outputs):
    x = (np.random.default_rng(n).random((n, 3)) ** power).astype(np.float32)
    q = charges(n, "u11") + 1j * charges(n, "u11", seed=9)
    f = pkg.FMM(p=4, depth=1, precision="fp32", domain=((0, 0, 0), 1.0), kernel="helmholtz", kappa=5.0)
    f.build_tree(torch.from_numpy(x).cuda()).precompute()
    kw = {"potential": outputs != "grad", "gradient": outputs != "phi"}
    phi, grad = f.evaluate(torch.from_numpy(q).to("cuda", torch.complex64), **kw)
    dp, dg = direct.direct_self(x.astype(np.float64), q, wavenumber=5.0)
    for got, want in ((phi, dp), (grad, dg)):
        if got is None:
            continue
        g = got.cpu().numpy().astype(np.complex128)
        assert (np.linalg.norm(g) == 0) if n == 1 else rel(g, want) < 2e-6
    f.close()
