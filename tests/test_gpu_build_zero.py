"""Negative zeros in a periodic build: a coordinate of -0.0 and a shift of -0.0
are zeros (the tree's positions lie in [0, box) and the sums are those of 0)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [(-0.0, -0.0, -0.0), (0.0, -0.0, 0.25)])
def test_negative_zero(oracle_mod, shift):
    import torch

    import paper_1909_04667_gb300 as tpm

    pos, mass = W.zeldovich(10, 4)
    pos[5, 0] = -0.0
    pos[300] = -0.0
    pos[77, 1:] = -0.0
    with tpm.Context(0) as ctx:
        s = ctx.build_tree(torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(),
                           tpm.BuildParams(h=0.01, periodic=True, box=1.0, shift=shift, leaf_bucket=4))
        got = s.tree_export()
    ref = oracle_mod.Tree(np.abs(pos), mass, bucket=4, periodic=True, box=1.0, shift=tuple(np.abs(shift))).export()
    assert got["xtree"].min() >= 0.0 and got["xtree"].max() < 1.0
    for k in ("key", "perm", "level", "prefix", "first", "count", "skip", "mass", "com", "xtree"):
        np.testing.assert_array_equal(got[k], ref[k], err_msg=k)
