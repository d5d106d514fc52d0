"""Which walk a call gets.  Calls that fill the chip keep the group walk: all
particles of several small systems in one batch, and a large call with
per-particle softening, have the bits that TPM_WALK=group gives them.  A request
has the same bits alone and in any mix of up to 49152 ids (those of the plain
call) and in any larger batch."""
import os
import subprocess
import sys

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DEV = "cuda:0"


def dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def batch(tpm, ctx, room, requests, fps):
    """Forces of the requests (system, ids, |a|) from one batched call."""
    import torch

    ids = np.concatenate([i for _, i, _ in requests]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum([len(i) for _, i, _ in requests])])
    old = np.concatenate([a for _, _, a in requests]).astype(np.float32)
    acc = torch.empty((len(ids), 3), device=DEV)
    nint = torch.empty(len(ids), dtype=torch.int32, device=DEV)
    plan = ctx.create_plan(room, 16)
    plan.compute_forces_batch([s for s, _, _ in requests], off, fps, dev(ids), acc, a_old=dev(old), n_int=nint)
    plan.sync_status()
    plan.close()
    acc, nint = acc.cpu().numpy(), nint.cpu().numpy()
    return [(acc[a:b], nint[a:b]) for a, b in zip(off[:-1], off[1:])]


def large_calls():
    """A batch of four small systems, and one call for 40000 particles of two species."""
    import paper_1909_04667_gb300 as tpm

    out = {}
    with tpm.Context(0) as ctx:
        requests = []
        for k in range(4):
            pos, mass = W.plummer(20000, k)
            s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.01, shift=tuple(W.root_shift(k)), leaf_bucket=8))
            requests.append((s, np.arange(20000), np.full(20000, 0.3)))
        for name, fp in (("bh", tpm.ForceParams(theta=0.6)),
                         ("rel", tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=0.0025))):
            got = batch(tpm, ctx, 80000, requests, fp)
            out["batch_" + name] = np.concatenate([a for a, _ in got])
        pos, mass, hs, _ = W.two_species(32000, 8000, 3)
        s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.01, shift=tuple(W.root_shift(3)), leaf_bucket=8),
                           hsoft=dev(hs))
        out["two_bh"] = s.compute_forces(fp=tpm.ForceParams(theta=0.6))[0].cpu().numpy()
        s.sync_status()
    return out


def test_calls_that_fill_the_chip_keep_the_group_walk(tmp_path):
    out = tmp_path / "group.npz"
    code = "import sys; sys.path[:0] = [%r, %r]; import numpy as np, test_gpu_walk_rule as t; " \
           "np.savez(sys.argv[1], **t.large_calls())" % (ROOT, os.path.join(ROOT, "tests"))
    subprocess.run([sys.executable, "-c", code, str(out)], check=True, env=dict(os.environ, TPM_WALK="group"),
                   timeout=600)
    group = np.load(out)
    for k, v in large_calls().items():
        np.testing.assert_array_equal(v, group[k], err_msg=k)


@pytest.mark.parametrize("filler", [0, 60000])
def test_alone_and_in_a_mix(filler):
    """Requests alone, in a mix and in a plain call; with a filler request behind each batch it is a large one."""
    import paper_1909_04667_gb300 as tpm

    rng = np.random.default_rng(5)
    bh, rel = tpm.ForceParams(theta=0.6), tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=0.0025)
    with tpm.Context(0) as ctx:
        requests, fps = [], []
        for k, n in enumerate((3000, 20000, 70000)):
            pos, mass = W.hernquist(n, k)
            s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.005, shift=tuple(W.root_shift(k)), leaf_bucket=8))
            inner = np.argsort(np.sum(pos * pos, axis=1))
            for ids in (rng.choice(n, 1, replace=False), rng.choice(n, 330, replace=False), inner[:1100]):
                requests.append((s, ids, 10.0 ** rng.uniform(-1.0, 0.5, len(ids))))
                fps.append((bh, rel)[len(fps) % 2])
        rest = [(s, np.arange(filler), np.full(filler, 0.3))]
        mix = batch(tpm, ctx, 70000, requests + rest, fps + [bh])
        for r, fp, (a, n) in zip(requests, fps, mix):
            (a1, n1), _ = batch(tpm, ctx, 70000, [r] + rest, [fp, bh])
            np.testing.assert_array_equal(a1, a)
            np.testing.assert_array_equal(n1, n)
            if not filler:
                a1, _, n1 = r[0].compute_forces(active_ids=dev(r[1].astype(np.int32)),
                                                a_old=dev(r[2].astype(np.float32)), fp=fp)
                np.testing.assert_array_equal(a1.cpu().numpy(), a)
                np.testing.assert_array_equal(n1.cpu().numpy(), n)


def test_both_walks_in_a_captured_graph():
    """A large batch and a large plain call whose chunks go to both walks, each
    followed at once by copies of its results: replays of the captured stream
    give the eager call's bits (what follows waits for both walks)."""
    import torch

    import paper_1909_04667_gb300 as tpm

    pos, mass = W.hernquist(200000, 9)
    rng = np.random.default_rng(9)
    inner = np.argsort(np.sum(pos * pos, axis=1))
    far = rng.choice(inner[60000:], 3001, replace=False)
    ids = np.concatenate([inner[:50000], far]).astype(np.int32)
    fp = tpm.ForceParams(theta=0.5)
    with tpm.Context(0) as ctx:
        s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.005, leaf_bucket=8))
        off = np.array([0, 40000, len(ids)], np.int64)
        plan = ctx.create_plan(len(ids), 2)
        t = dev(ids)
        acc, copy = (torch.zeros((2, len(ids), 3), device=DEV) for _ in range(2))

        def calls():
            plan.compute_forces_batch([s, s], off, fp, t, acc[0])
            copy[0].copy_(acc[0])
            s.compute_forces_noalloc(t, fp=fp, acc=acc[1])
            copy[1].copy_(acc[1])

        calls()
        torch.cuda.synchronize()
        eager = copy.cpu().numpy().copy()
        assert (np.linalg.norm(eager, axis=2) > 0.0).all()
        g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st), torch.cuda.graph(g, stream=st):
            calls()
        torch.cuda.current_stream().wait_stream(st)
        for _ in range(5):
            acc.zero_()
            copy.zero_()
            g.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(copy.cpu().numpy(), eager)
        plan.sync_status()
        s.sync_status()
        plan.close()


def test_groups_of_64_have_the_same_bits_in_any_mix():
    """A plan with groups of 64 particles has one walk for all: what a request gets does not depend on the batch."""
    import torch

    import paper_1909_04667_gb300 as tpm

    rng = np.random.default_rng(8)
    with tpm.Context(0) as ctx:
        pos, mass = W.plummer(70000, 8)
        s = ctx.build_tree(dev(pos), dev(mass), tpm.BuildParams(h=0.01, leaf_bucket=8))
        ids, rest = rng.choice(70000, 3333, replace=False).astype(np.int32), np.arange(70000, dtype=np.int32)
        plan = ctx.create_plan(80000, 2)
        plan.group_size = 64
        out = []
        for more in (rest[:0], rest[:9000], rest):
            acc = torch.empty((len(ids) + len(more), 3), device=DEV)
            plan.compute_forces_batch([s, s], np.array([0, len(more), len(more) + len(ids)]), tpm.ForceParams(theta=0.6),
                                      dev(np.concatenate([more, ids])), acc)
            plan.sync_status()
            out.append(acc[len(more):].cpu().numpy())
        plan.close()
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])
