"""The device memory that a build needs, beyond what its tree keeps, of systems
with few nodes per particle (large leaves, all particles at one place): a system
that fitted a budget keeps fitting it.  Bytes per particle of the smallest budget
that holds the build."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,bucket,limit", [("large leaves", 5000, 124.28), ("one place", 8, 124.25)])
def test_smallest_budget(kind, bucket, limit):
    import torch

    import paper_1909_04667_gb300 as tpm

    n = 300000
    pos = np.random.default_rng(3).uniform(0.0, 1.0, (n, 3))
    if kind == "one place":
        pos[:] = pos[0]
    pos, mass = torch.from_numpy(pos).cuda(), torch.ones(n, device="cuda")
    with tpm.Context(0, budget_bytes=int(limit * n)) as ctx:
        ctx.build_tree(pos, mass, tpm.BuildParams(h=0.01, leaf_bucket=bucket)).release()
