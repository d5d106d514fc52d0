"""The tree build at the edges of its stretches (1024 sorted particles a block,
32 blocks a further level of sums), of its leaf classes (more than 16 particles
a leaf) and of its coordinate scaling (roots of very small and large side):
bit for bit the oracle's tree, masses and centres of mass included."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.device("cuda", 0))


@pytest.fixture(scope="module")
def ctx():
    import paper_1909_04667_gb300 as tpm

    c = tpm.Context(0)
    yield tpm, c
    c.close()


def check(oracle_mod, ctx, pos, mass, bucket, periodic=False, box=1.0):
    tpm, c = ctx
    shift = tuple(W.root_shift(len(pos)))
    bp = tpm.BuildParams(G=1.0, h=0.01, periodic=periodic, box=box, shift=shift, leaf_bucket=bucket)
    s = c.build_tree(dev(pos), dev(mass), bp)
    ex = s.tree_export()
    s.release()
    ref = oracle_mod.Tree(pos, mass, bucket=bucket, periodic=periodic, box=box, shift=shift)
    rx = ref.export()
    assert ex["n_nodes"] == ref.nnodes and ex["L0"] == ref.L0
    for k in ("key", "perm", "level", "prefix", "first", "count", "skip", "mass", "com", "xtree"):
        np.testing.assert_array_equal(ex[k], rx[k], err_msg=k)


@pytest.mark.parametrize("bucket", [1, 16, 40])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 32767, 32769, 66000])
def test_stretches(oracle_mod, ctx, n, bucket):
    pos, mass = W.hernquist(n, n)
    mass = (mass * np.random.default_rng(n).uniform(0.5, 1.5, n)).astype(np.float32)
    check(oracle_mod, ctx, pos, mass, bucket)


def test_coincident_particles_across_stretches(oracle_mod, ctx):
    """One leaf at the depth cap that spans several stretches."""
    pos, mass = W.plummer(6000, 3)
    pos[1000:4500] = pos[0]
    check(oracle_mod, ctx, pos, mass, 8)


@pytest.mark.parametrize("n", [255, 513, 20480, 20481])
def test_sorts(oracle_mod, ctx, n):
    """Both sorts, with equal keys (ties by index) and a last ragged block."""
    pos, mass = W.plummer(n, n)
    pos[::7] = pos[3]
    pos[n // 2:n // 2 + 40] = pos[n - 1]
    check(oracle_mod, ctx, pos, mass, 4)


@pytest.mark.parametrize("scale", [1e-200, 1e-30, 1e30])
def test_scales(oracle_mod, ctx, scale):
    pos, mass = W.plummer(3000, 5)
    check(oracle_mod, ctx, pos * scale, mass, 8)


@pytest.mark.parametrize("box", [1.0, 0.7, 3.0e4])
def test_boxes(oracle_mod, ctx, box):
    pos, mass = W.zeldovich(18, 4)
    check(oracle_mod, ctx, np.minimum(pos * box, np.nextafter(box, 0.0)), mass, 8, True, box)
