"""Outputs past half of the L2 cache are written in windows: every output is written once, with the value that
one window writes.  4300001 points' potentials and gradients (69 MB) take two windows, the gradients alone
(52 MB) and the potentials alone one.  Gradients are equal; the potential-only sums round differently (2e-6)."""
import pytest
import torch

import paper_2604_19243_gb300 as pkg
from gpu_helpers import rel

pytestmark = pytest.mark.gpu


def test_windows_cover_every_output():
    n = 4_300_001
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.rand(n, 3, device="cuda", generator=gen)
    q = torch.rand(n, device="cuda", generator=gen) - 0.5
    f = pkg.FMM(p=3, depth=6, precision="fp32", domain=((0, 0, 0), 1.0))
    f.build_tree(x).precompute()
    phi, grad = f.evaluate(q)
    g_only = f.evaluate(q, potential=False)[1]
    p_only = f.evaluate(q, gradient=False)[0]
    assert torch.equal(grad, g_only)
    assert rel(phi.cpu().numpy(), p_only.cpu().numpy()) < 2e-6
    assert bool((phi != 0).all())
    f.close()
