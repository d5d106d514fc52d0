"""A plan's memory and its lists: what a plan takes per id and request (a plan
that fitted a budget keeps fitting it), and a batch of single ids, in which
every id is a group of its own on the two-target list."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ids,requests", [(1, 1), (1 << 20, 512), (100, 5000)])
def test_plan_bytes(ids, requests):
    import paper_1909_04667_gb300 as tpm

    with tpm.Context(0) as ctx:
        plan = ctx.create_plan(ids, requests)
        used = ctx.memory()[0]
        plan.close()
    assert used <= 43 * ids + 260 * requests + 4608, used


@pytest.mark.parametrize("presorted", [False, True])
def test_single_ids(presorted):
    import torch

    import paper_1909_04667_gb300 as tpm

    n, m = 30000, 80000
    pos, mass = W.plummer(n, 2)
    with tpm.Context(0) as ctx:
        s = ctx.build_tree(torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(),
                           tpm.BuildParams(h=0.01, leaf_bucket=8))
        ids = torch.from_numpy(np.random.default_rng(1).integers(0, n, m).astype(np.int32)).cuda()
        fp = tpm.ForceParams(theta=0.6)
        acc = torch.zeros((m, 3), device="cuda")
        nint = torch.zeros(m, dtype=torch.int32, device="cuda")
        plan = ctx.create_plan(m, m)
        plan.compute_forces_batch([s] * m, np.arange(m + 1), fp, ids, acc, n_int=nint, presorted=presorted)
        plan.sync_status()
        plan.close()
        a, _, k = s.compute_forces(fp=fp)
        a, k, acc, nint = (x.cpu().numpy() for x in (a[ids.long()], k[ids.long()], acc, nint))
    same = nint == k
    assert np.mean(~same) <= 0.005
    e = np.linalg.norm(acc - a, axis=1) / np.linalg.norm(a, axis=1)
    assert np.percentile(e[same], 99) <= 2e-5 and e[same].max() <= 2e-4, (np.percentile(e[same], 99), e[same].max())
