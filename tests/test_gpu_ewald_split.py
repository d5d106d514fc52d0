"""The Ewald tree's walk with several warps sharing a chunk's nodes, against
the FP64 oracle walk at the edges of that split: trees of few nodes (empty
segments), one target, a ragged last chunk, and each number of warps per chunk
down to one.  Tolerances of test_gpu_ewald (p99 1e-5, max 5e-5)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.device("cuda", 0))


@pytest.mark.parametrize("crit", ["bh", "rel"])
@pytest.mark.parametrize("n,count", [(2, 2), (33, 33), (1000, 1), (8000, 33), (8000, 8000), (30000, 20000)])
def test_split_matches_oracle(oracle_mod, n, count, crit):
    import paper_1909_04667_gb300 as tpm

    rng = np.random.default_rng(n + count)
    pos, mass = rng.uniform(0.0, 1.0, (n, 3)), np.full(n, 1.0 / n, np.float32)
    h, shift = n ** (-1.0 / 3.0) / 40.0, tuple(W.root_shift(n))
    ids = np.sort(rng.choice(n, count, replace=False)).astype(np.uint32)
    a_old = (10.0 ** rng.uniform(-1.0, 0.5, count)).astype(np.float32)
    ctx = tpm.Context(0)
    s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=h, periodic=True, box=1.0, shift=shift, leaf_bucket=8))
    fp = (tpm.ForceParams(theta=0.7) if crit == "bh" else tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=0.005))
    acc, _, nint = s.compute_forces(active_ids=dev(ids.astype(np.int32)), a_old=dev(a_old), fp=fp)
    s.sync_status()
    s.release()
    ctx.close()
    tree = oracle_mod.Tree(pos, mass, bucket=8, periodic=True, box=1.0, shift=shift)
    kw = dict(theta=0.7) if crit == "bh" else dict(crit="rel", alpha=0.005, a_old=a_old)
    a_o, _, n_o = tree.walk(ids, 1.0, h, ewald=True, **kw)
    acc, nint = acc.cpu().numpy().astype(np.float64), nint.cpu().numpy()
    same = nint == n_o
    assert np.mean(~same) <= 0.005 or (~same).sum() <= 1
    e = np.linalg.norm(acc - a_o, axis=1) / np.linalg.norm(a_o, axis=1)
    assert np.percentile(e[same], 99) <= 1e-5 and e[same].max() <= 5e-5, (np.percentile(e[same], 99), e[same].max())
