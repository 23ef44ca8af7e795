"""The tree build at the edges of its blocks: rounds of 32 points, 1024 and 4096 keys of a sort tile and
the change between the two sizes (152 tiles of 4096), 2048 points of a level block, more than one block of
a scan.  Whole numbers: every table equals the oracle's."""
import numpy as np
import pytest
import torch

import paper_2604_19243_gb300 as pkg
from oracle import tree as otree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,depth", [(1, 0), (1, 4), (31, 10), (33, 2), (1023, 3), (1025, 7), (2047, 5), (2048, 1),
                                     (2049, 6), (4097, 4), (152 * 4096 - 1, 6), (152 * 4096, 5), (152 * 4096 + 1, 7)])
def test_tables_at_block_edges(n, depth):
    rng = np.random.default_rng(n + depth)
    x = rng.random((n, 3)).astype(np.float32)
    x[n // 2:] = x[n // 2:] ** 4        # crowded boxes beside empty ones
    f = pkg.FMM(p=3, depth=depth, domain=((0, 0, 0), 1.0))
    f.build_tree(torch.from_numpy(x).cuda()).precompute()
    got, o = f.export_tree(), otree.build_tree(x.astype(np.float64), depth, (0, 0, 0), 1.0)
    for name, want in (("perm", o.perm), ("leaf_keys", o.leaf_keys), ("leaf_offsets", o.leaf_offsets)):
        np.testing.assert_array_equal(got[name], want)
    for level in range(depth + 1):
        np.testing.assert_array_equal(f.export_level(level, lists=False)["keys"], o.level_keys[level])
    if n < 10_000:
        uo, ui = otree.u_lists(o)
        np.testing.assert_array_equal(got["u_offsets"], uo)
        np.testing.assert_array_equal(got["u_idx"], ui)
    assert f.debug_check()[0] == []     # parent, child and dense tables, orders and masks
    f.close()
