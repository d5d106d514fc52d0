"""The periodic short-range walk at the edges of its bounds, against the FP64
oracle TreePM: few particles in large leaves, a ragged last group, sparse
targets (groups wider than an eighth of the box, whose nodes have different
images for different targets), leaves of more than 32 particles, boxes that are
no power of two, particles clustered across the box's corner, and four and two
warps per group (one: the full-size box of test_gpu_fullsize).  Identical counts
up to FP32 margin flips; forces within 1e-4 (p99) and 1e-3 (max) of the rms
force, the tolerance of the FP32 mesh."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.device("cuda", 0))


CASES = [("uniform", 40, 40, 1.0, 32, 8), ("uniform", 3001, 3001, 0.7, 32, 8), ("uniform", 3001, 50, 1.0, 32, 64),
         ("uniform", 20000, 20000, 2.5, 64, 4), ("uniform", 20000, 33, 2.5, 64, 1), ("corner", 2500, 2500, 1.0, 64, 48),
         ("one", 1000, 1, 3.0, 32, 8), ("uniform", 150000, 150000, 1.0, 64, 8)]


@pytest.mark.parametrize("crit", ["bh", "rel"])
@pytest.mark.parametrize("kind,n,count,box,pm_n,bucket", CASES)
def test_matches_oracle_treepm(oracle_mod, kind, n, count, box, pm_n, bucket, crit):
    import paper_1909_04667_gb300 as tpm

    rng = np.random.default_rng(n + count)
    pos = rng.uniform(0.0, box, (n, 3)) if kind != "corner" else np.mod(0.02 * box * rng.standard_normal((n, 3)), box)
    pos = np.minimum(pos, np.nextafter(box, 0.0))
    mass = (rng.uniform(0.5, 1.5, n) / n).astype(np.float32)
    ids = np.sort(rng.choice(n, count, replace=False)).astype(np.uint32)
    a_old = (10.0 ** rng.uniform(-1.0, 0.5, count) / box ** 2).astype(np.float32)
    h, shift = box * n ** (-1.0 / 3.0) / 40.0, tuple(W.root_shift(n))
    kw = dict(treepm=True, pm_n=pm_n, asmth=1.25, rcut=4.5)
    fp = (tpm.ForceParams(theta=0.6, **kw) if crit == "bh" else
          tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=0.005, **kw))
    ctx = tpm.Context(0)
    s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=h, periodic=True, box=box, shift=shift,
                                                            leaf_bucket=bucket))
    s.pm_long_range(fp)
    acc, _, nint = s.compute_forces(active_ids=dev(ids.astype(np.int32)), a_old=dev(a_old), fp=fp)
    s.sync_status()
    xtree = s.tree_export()["xtree"]  # shifted and wrapped: the mesh lies in this frame
    s.release()
    ctx.close()
    okw = dict(theta=0.6) if crit == "bh" else dict(crit="rel", alpha=0.005, a_old=a_old)
    a_o, _, n_o = oracle_mod.treepm(xtree, mass, ids, box, pm_n, 1.25, 4.5, 1.0, h, bucket=bucket, **okw)
    nint = nint.cpu().numpy()
    same = nint == n_o
    assert np.mean(~same) <= 0.005 or (~same).sum() <= 1, np.mean(~same)
    e = np.linalg.norm(acc.cpu().numpy() - a_o, axis=1) / np.sqrt(np.mean(np.sum(a_o * a_o, axis=1)))
    assert np.percentile(e[same], 99) <= 1e-4 and e[same].max() <= 1e-3, (np.percentile(e[same], 99), e[same].max())
