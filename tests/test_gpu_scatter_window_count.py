"""The output windows are few however large the outputs are (each reads every point's sums again): 26 million
points take no more launches than 13 million on a tree of the same depth.  The gradients of one call are
those of a gradient-only call, bit for bit (other windows, the same sums)."""
import pytest
import torch

import paper_2604_19243_gb300 as pkg

pytestmark = pytest.mark.gpu


def test_windows_do_not_grow_with_the_outputs():
    launches = []
    for n in (13_000_001, 26_000_003):
        gen = torch.Generator(device="cuda").manual_seed(5)
        x = torch.rand(n, 3, device="cuda", generator=gen)
        q = torch.rand(n, device="cuda", generator=gen) - 0.5
        f = pkg.FMM(p=2, depth=6, precision="fp32", domain=((0, 0, 0), 1.0))
        f.build_tree(x).precompute()
        phi, grad = f.evaluate(q)
        before = pkg.kernel_launches()
        f.evaluate(q)
        launches.append(pkg.kernel_launches() - before)
        assert torch.equal(grad, f.evaluate(q, potential=False)[1])
        assert bool((phi != 0).all())
        f.close()
    assert launches[0] == launches[1]
