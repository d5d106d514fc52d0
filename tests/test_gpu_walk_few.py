"""The walk with two targets per warp against the FP64 oracle walk, over the
forms that its rule takes (small systems, sparse requests, repeated and
unsorted ids, a last lone target, cut chunks, mesh and per-particle softening)
and at the edges of the rule, and its results in a batch against the plain
call.  Tolerances as for the other walks: identical interaction counts up to
FP32 margin flips, forces p99 2e-5 and max 2e-4 (with the mesh 1e-4, 1e-3)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tpm():
    import paper_1909_04667_gb300 as m

    return m


@pytest.fixture(scope="module")
def ctx(tpm):
    c = tpm.Context(0)
    yield c
    c.close()


def dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.device("cuda", 0))


def compare(acc, a_o, nint, n_o, p99=2e-5, mx=2e-4):
    same = nint == n_o
    assert np.mean(~same) <= 0.005 or (~same).sum() <= 1, np.mean(~same)
    e = np.linalg.norm(acc - a_o, axis=1) / np.maximum(np.linalg.norm(a_o, axis=1), 1e-300)
    assert np.percentile(e[same], 99) <= p99 and e[same].max() <= mx, (np.percentile(e[same], 99), e.max())


def ids_of(kind, n, pos):
    rng = np.random.default_rng(n)
    if kind == "all":
        return np.arange(n)
    if kind == "one":
        return np.array([n // 2])
    if kind == "sparse33":
        return rng.choice(n, 33, replace=False)
    if kind == "sparse1000":
        return rng.choice(n, 1000, replace=False)
    if kind == "repeated":
        return np.repeat(rng.choice(n, 50, replace=False), 3)
    return np.argsort(np.sum(pos * pos, axis=1))[:1000]  # dense: the innermost particles


CASES = [(n, "all") for n in (1, 2, 31, 33, 4097)] + [(20000, "one"), (20000, "sparse1000"), (20000, "repeated"),
                                                      (32768, "sparse33"), (32769, "sparse33"), (50000, "one"),
                                                      (50000, "sparse1000"), (50000, "repeated"), (50000, "dense")]


@pytest.mark.parametrize("crit", ["bh", "rel"])
@pytest.mark.parametrize("n,kind", CASES)
def test_matches_oracle_walk(oracle_mod, tpm, ctx, n, kind, crit):
    pos, mass = W.hernquist(n, 40 + n % 7)
    shift, h = tuple(W.root_shift(n % 13)), 0.005
    ids = ids_of(kind, n, pos).astype(np.uint32)
    a_old = (10.0 ** np.random.default_rng(n).uniform(-1.5, 0.5, len(ids))).astype(np.float32)
    s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=h, shift=shift, leaf_bucket=8))
    fp = tpm.ForceParams(theta=0.6) if crit == "bh" else tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=0.0025)
    acc, pot, nint = s.compute_forces(active_ids=dev(ids.astype(np.int32)), a_old=dev(a_old), fp=fp)
    s.sync_status()
    tree = oracle_mod.Tree(pos, mass, bucket=8, shift=shift)
    kw = dict(theta=0.6) if crit == "bh" else dict(crit="rel", alpha=0.0025, a_old=a_old)
    a_o, p_o, n_o = tree.walk(ids, 1.0, h, **kw)
    compare(acc.cpu().numpy().astype(np.float64), a_o, nint.cpu().numpy(), n_o)
    np.testing.assert_allclose(pot.cpu().numpy(), p_o, rtol=5e-5)
    # the same request in a batch, between others: the same bits
    other = np.arange(min(n, 700), dtype=np.int32)
    cat = np.concatenate([other, ids.astype(np.int32), other])
    off = np.cumsum([0, len(other), len(ids), len(other)])
    old = np.concatenate([np.ones(len(other)), a_old, np.ones(len(other))]).astype(np.float32)
    import torch

    b = torch.empty((len(cat), 3), device="cuda:0")
    bn = torch.empty(len(cat), dtype=torch.int32, device="cuda:0")
    plan = ctx.create_plan(len(cat), 3)
    plan.compute_forces_batch([s, s, s], off, fp, dev(cat), b, a_old=dev(old), n_int=bn)
    plan.sync_status()
    np.testing.assert_array_equal(b[off[1]:off[2]].cpu().numpy(), acc.cpu().numpy())
    np.testing.assert_array_equal(bn[off[1]:off[2]].cpu().numpy(), nint.cpu().numpy())
    plan.close()
    s.release()


@pytest.mark.parametrize("crit", ["bh", "rel"])
def test_cut_chunks(oracle_mod, tpm, ctx, crit):
    """Chunks that reach from a dense cluster to isolated particles are walked
    in several frames; every particle within the standard tolerances."""
    pos, mass = W.clusters_with_outliers(6000, 3)
    n, shift, h = len(pos), tuple(W.root_shift(3)), 0.01
    a_old = (10.0 ** np.random.default_rng(3).uniform(-5, -1, n)).astype(np.float32)
    s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=h, shift=shift, leaf_bucket=8))
    fp = tpm.ForceParams(theta=0.6) if crit == "bh" else tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=0.0025)
    acc, _, nint = s.compute_forces(a_old=dev(a_old), fp=fp)
    s.sync_status()
    s.release()
    kw = dict(theta=0.6) if crit == "bh" else dict(crit="rel", alpha=0.0025, a_old=a_old)
    a_o, _, n_o = oracle_mod.Tree(pos, mass, bucket=8, shift=shift).walk(np.arange(n), 1.0, h, **kw)
    compare(acc.cpu().numpy().astype(np.float64), a_o, nint.cpu().numpy(), n_o)


@pytest.mark.parametrize("n_halo", [9000, 40000])
def test_per_particle_softening_and_mesh(oracle_mod, tpm, ctx, n_halo):
    """The forms that no batch runs, below and above the small-system size."""
    pos, mass, hs, _ = W.two_species(n_halo, n_halo // 3, 7)
    n, shift = len(pos), tuple(W.root_shift(7))
    ids = np.random.default_rng(7).choice(n, 1500, replace=False).astype(np.uint32)
    fp = tpm.ForceParams(theta=0.5, treepm=True, pm_n=32, asmth=2.5, rcut=4.5)
    s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.0123, shift=shift, leaf_bucket=8), hsoft=dev(hs))
    acc, _, nint = s.compute_forces(active_ids=dev(ids.astype(np.int32)), fp=tpm.ForceParams(theta=0.5))
    s.release()
    tree = oracle_mod.Tree(pos, mass, bucket=8, shift=shift, hsoft=hs)
    a_o, _, n_o = tree.walk(ids, 1.0, 0.0123, theta=0.5)
    compare(acc.cpu().numpy().astype(np.float64), a_o, nint.cpu().numpy(), n_o)
    s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.005, shift=shift, leaf_bucket=8))
    s.pm_long_range(fp)
    acc, _, nint = s.compute_forces(active_ids=dev(ids.astype(np.int32)), fp=fp)
    s.sync_status()
    s.release()
    a_o, _, n_o = oracle_mod.treepm_isolated(pos, mass, ids, 32, 2.5, 4.5, 1.0, 0.005, shift=shift, theta=0.5)
    compare(acc.cpu().numpy().astype(np.float64), a_o, nint.cpu().numpy(), n_o, 1e-4, 1e-3)
