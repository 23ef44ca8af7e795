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
    ("fp32", 6, 5, 20000): """
        -271.47229 530.546082 1653.13391 -176.295609 -382.850311 -1074.22925
        -150.85585 290.25943 1145.61865 -357.963623 -1428.53601 -946.206238
        824.21991 582.674744 -997.928833 -456.460724 992.460754 -1208.0752
        1053.38159 -766.326843 -670.746643 1883.73743 172.914658 -80.2765656
        -132.252625 -305.791931 -1262.67126 -1268.31934 -958.301392 567.910828
        -7.05098915 -1663.63635 -332.546478 -549.006958 280.18985 1231.08765
        -430.354401 343.201233 1692.43127 -212.095383 1826.69275 -362.433411
        976.777344 -1437.77954 361.888794 -1525.14697 779.133911 -364.748291
        """,
    ("fp32", 8, 4, 9001): """
        -167.748932 224.343292 713.613098 684.383179 -129.419876 -172.992126
        409.929077 224.38559 -548.593018 -421.16275 -111.402542 -592.931458
        429.622284 -298.127533 -277.235107 -498.992432 145.139999 441.901184
        223.674881 348.91452 -596.879089 57.9263535 378.565857 646.773071
        404.501984 -385.007568 416.325836 249.265656 537.219543 -395.474182
        -490.302032 -402.560028 -308.880615 534.984863 489.651123 159.238983
        -132.681702 295.656586 -650.249512 41.9355888 267.110443 117.946396
        -305.161987 -35.0608826 714.598755 -393.281006 -225.448853 470.173401
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
