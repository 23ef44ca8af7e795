"""FP32 contexts deeper than the depth up to which the uniform M2L runs from FP16 planes: the planes of the
adaptive tree come and go with it, in either order of set-up and precomputation and between uniform
evaluations, whose results they leave alone.

Reference: the same calls on contexts of their own.  Every sum has one order, so results are the same bits.
"""
import pytest
import torch

from synth import charges, mixed_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ops_first", [True, False])
def test_adaptive_and_uniform_evaluations_in_turn(ops_first):
    import paper_2604_19243_gb300 as pkg
    x, q = torch.from_numpy(mixed_points(5001)).cuda(), torch.from_numpy(charges(5001, "u11")).cuda()

    def context():
        return pkg.FMM(p=4, depth=6, precision="fp32", domain=((0.0, 0.0, 0.0), 1.0)).build_tree(x)

    uniform, adaptive = context().precompute(), context().precompute()
    adaptive.adaptive_setup(32)
    want_u, want_a = uniform.evaluate(q), adaptive.adaptive_evaluate(q)
    f = context()
    if ops_first:
        f.precompute()
        assert all(torch.equal(a, b) for a, b in zip(f.evaluate(q), want_u))
    f.adaptive_setup(32)
    f.precompute()
    for _ in range(2):
        assert all(torch.equal(a, b) for a, b in zip(f.adaptive_evaluate(q), want_a))
        assert all(torch.equal(a, b) for a, b in zip(f.evaluate(q), want_u))
        f.build_tree(x).adaptive_setup(32)
    f.sync()
