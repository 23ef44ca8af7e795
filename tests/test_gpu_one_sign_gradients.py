"""Gradients of one-sign charges keep the rounding they have always had.

A potential of charges of one sign is 2^depth times its variation across a leaf, so the far field's gradients
carry the rounding of the FP32 sums of the check potentials (2e-5 to 5e-5 in deep trees).  Another order of
the same sums gives gradients as exact that differ by as much, so their order is part of the results.

Reference: far-field gradients at 16 of the points, recorded from the code that sums the transfer vectors of
a box one after the other (FP16X3: the products of one in one tensor-memory accumulator).  Tolerance: 2e-6.
The same sequence gives the same bits; another order, or another split of the operands, has measured 1.8e-5
to 6.3e-5 on these inputs.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import rel
from synth import charges, cube_points

pytestmark = pytest.mark.gpu

# (precision, p, depth, points): x, y, z of every (points // 16)-th point
GRADIENTS = {
    ("fp16x3", 4, 6, 20000): """
        -311.159393 430.308716 1723.25317 -190.770233 -378.834839 -1078.75708
        -206.707016 321.96347 1155.38843 -428.608521 -1428.31091 -896.144226
        871.782532 619.096985 -947.258484 -426.635834 991.537659 -1230.13086
        1108.36218 -839.081604 -653.198608 1861.70386 124.032318 -112.263916
        -31.3612499 -203.280441 -1355.32056 -1216.29456 -926.593384 535.913818
        -55.1736755 -1674.27539 -367.583862 -479.083954 340.453125 1254.86584
        -433.846954 283.935333 1649.24365 -180.977386 1914.34119 -395.484467
        917.209839 -1456.67175 372.177612 -1684.07593 731.988464 -478.834717
        """,
    ("fp16x3", 6, 6, 20000): """
        -310.562836 434.726807 1719.32153 -193.858932 -376.637115 -1074.35608
        -216.961044 353.770264 1134.8562 -428.029877 -1428.51575 -895.102905
        886.717896 619.876648 -959.435669 -421.50708 988.368469 -1225.29102
        1129.33325 -844.340271 -679.505188 1867.16882 110.129128 -101.305229
        -29.7160454 -209.339294 -1378.34949 -1193.37366 -915.651001 538.315491
        -59.0062904 -1667.07324 -379.517395 -474.919952 340.146393 1254.36035
        -433.553925 296.304962 1650.71338 -164.558899 1914.01624 -383.136902
        916.584778 -1439.60339 379.218353 -1689.44019 733.041077 -457.328613
        """,
}


@pytest.mark.parametrize("precision,p,depth,n", list(GRADIENTS))
def test_far_gradients_keep_their_rounding(precision, p, depth, n):
    import paper_2604_19243_gb300 as pkg
    x, q = torch.from_numpy(cube_points(n)).cuda(), torch.from_numpy(charges(n, "u01")).cuda()
    f = pkg.FMM(p=p, depth=depth, precision=precision, domain=((0.0, 0.0, 0.0), 1.0))
    f.build_tree(x).precompute()
    _, grad = f.evaluate(q, parts=pkg.PART_FAR)
    want = np.array(GRADIENTS[precision, p, depth, n].split(), dtype=np.float64)
    assert rel(grad[:: n // 16][:16].cpu(), want) < 2e-6
    f.sync()
