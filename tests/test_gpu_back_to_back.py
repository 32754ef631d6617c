"""Calls queued behind one another while the GPU is busy, so that each kernel is
started early, against the same calls with a wait after each: every call reads
what the one before it wrote (indices, entries of a packed batch, advantages,
the tree), with other values in each round, so that anything read too early
shows.  Bit for bit."""
import numpy as np
import pytest
import torch

from gpu_util import cuda, fx, to_np, tree_levels

pytestmark = pytest.mark.gpu

ROUNDS, CAP, H, W, K = 4, 4096, 8, 16, 2


def _replay(edp, seed):
    """(calls, outputs, ring) of prioritized replay rounds."""
    rng = np.random.default_rng(seed)
    n = CAP + 300
    frames, action, reward, done = fx.dqn_transitions(seed, n, H * W, done_p=0.05)
    ring = edp.Ring(edp.make_config(CAP, (1, H, W), edp.EDP_XFORM_STACK_F32, frame_stack=K,
                                    next_obs=True, prioritized=True))
    q = rng.integers(1, 1 << 22, size=n).astype(np.uint32)
    for lo, hi in [(0, CAP), (CAP, n)]:
        edp.edp_ingest(ring.ctx, cuda(frames[lo:hi]), hi - lo, action=cuda(action[lo:hi]),
                       reward=cuda(reward[lo:hi]), done=cuda(done[lo:hi]), q=cuda(q[lo:hi]))
    calls, outs = [], []
    for k in range(ROUNDS):
        for B in (300, 2500):  # either kernel of the update
            new = [cuda(x[k * 7:k * 7 + 50 + k]) for x in (frames, action, reward, done, q)]
            td = cuda(fx.td_errors(seed + k, B))
            idx = torch.zeros(B, dtype=torch.int64, device="cuda")
            qs, act = (torch.zeros(B, dtype=torch.int32, device="cuda") for _ in range(2))
            obs, nxt = (torch.zeros(B * K * H * W, device="cuda") for _ in range(2))
            rew, isw = (torch.zeros(B, device="cuda") for _ in range(2))
            dn = torch.zeros(B, dtype=torch.uint8, device="cuda")
            tot = torch.zeros(1, dtype=torch.int64, device="cuda")
            batch = edp.make_batch(obs, nxt, act, rew, dn, q=qs, isw=isw, beta=0.5)
            calls += [
                lambda new=new: edp.edp_ingest(ring.ctx, new[0], len(new[1]), action=new[1],
                                               reward=new[2], done=new[3], q=new[4]),
                lambda i=idx, q=qs, B=B, k=k: edp.edp_sample(
                    ring.ctx, edp.EDP_SAMPLE_PRIORITIZED, B, 3, k, i, q),
                lambda i=idx, B=B, b=batch: edp.edp_deliver(ring.ctx, i, B, b),
                lambda i=idx, t=td, B=B: edp.edp_update_priorities_td(ring.ctx, i, t, B, 0.6, 1e-6),
                lambda t=tot: edp.edp_tree_total(ring.ctx, t)]
            outs += [idx, qs, act, obs, nxt, rew, isw, dn, tot]
    return calls, outs, ring


def _packs(edp, seed):
    """Packed batches of every way of copying them, other lengths in each."""
    rng = np.random.default_rng(seed)
    ring = edp.Ring(edp.make_config(16, (1, 4, 4), edp.EDP_XFORM_HWC_CHW_BF16), action=False,
                    reward=False, done=False)
    calls, outs = [], []
    for k in range(ROUNDS):
        for B, lmax, longer in ((1500, 60 + 40 * k, 3000), (9000, 90 - 20 * k, 2000),
                                (70_000, 12 + k, 0), (200, 900 + 300 * k, 0),
                                (20, 9000 - 1000 * k, 0)):
            lens = rng.integers(0, lmax + 1, size=B)
            if longer:
                lens[rng.integers(0, B, size=5)] = longer
            off = np.zeros(B + 1, np.uint64)
            np.cumsum(lens, out=off[1:])
            total = int(off[-1])
            group = np.arange(0, B + 1, 10, dtype=np.uint64)
            t = [cuda(x) for x in (rng.integers(0, 1 << 30, size=total + 1, dtype=np.int32), off,
                                   rng.permutation(B).astype(np.int64),
                                   rng.standard_normal(B).astype(np.float32), group)]
            adv = torch.zeros(B, device="cuda")
            ot = torch.zeros(total, dtype=torch.int32, device="cuda")
            ov = torch.zeros(total, device="cuda")
            oo = torch.zeros(B + 1, dtype=torch.int64, device="cuda")
            calls.append(lambda t=t, B=B, a=adv, ot=ot, oo=oo, ov=ov, n=total:
                         edp.edp_grpo_pack_deliver(ring.ctx, t[3], t[4], len(t[4]) - 1, 1e-6, a,
                                                   t[0], t[1], B, t[2], B, ot, oo, n,
                                                   out_value=ov))
            outs += [adv, ot, ov, oo]
    calls.append(calls[2])  # the most scratch first
    calls.insert(0, calls[-1])
    return calls, outs, ring


def _rollouts(edp, seed):
    """Insertion, advantages, shuffle and delivery of one rollout after another."""
    rng = np.random.default_rng(seed)
    ring = edp.Ring(edp.make_config(CAP, (2, 8, 8), edp.EDP_XFORM_HWC_CHW_BF16), action=False,
                    reward=False, done=False)
    calls, outs = [], []
    for k in range(ROUNDS):
        for T, E in ((128, 32), (4096, 1), (1, 4096)):
            t = [cuda(x) for x in (rng.integers(0, 256, (CAP, 128), dtype=np.uint8),
                                   rng.standard_normal((T, E)).astype(np.float32),
                                   rng.standard_normal((T + 1, E)).astype(np.float32),
                                   (rng.random((T, E)) < 0.02).astype(np.uint8))]
            adv, ret, norm = (torch.zeros(T, E, device="cuda") for _ in range(3))
            a, r = (torch.zeros(CAP, device="cuda") for _ in range(2))
            idx = torch.zeros(CAP, dtype=torch.int64, device="cuda")
            obs = torch.zeros(CAP * 128, dtype=torch.bfloat16, device="cuda")
            batch = edp.make_batch(obs, gather=[(norm, a), (ret, r)])
            calls += [
                lambda t=t: edp.edp_ingest(ring.ctx, t[0], CAP),
                lambda t=t, T=T, E=E, o=(adv, ret, norm): edp.edp_gae(
                    ring.ctx, t[1], t[2], t[3], T, E, 0.99, 0.95, *o),
                lambda i=idx, k=k: edp.edp_sample(ring.ctx, edp.EDP_SAMPLE_PERMUTE, CAP, 5, k, i),
                lambda i=idx, b=batch: edp.edp_deliver(ring.ctx, i, CAP, b)]
            outs += [adv, ret, norm, a, r, idx, obs.view(torch.int16)]
    return calls, outs, ring


def _flat(tree):
    leaves, levels, pending, qmax = tree
    return [leaves, *levels, pending, qmax]


@pytest.mark.parametrize("make", [_replay, _packs, _rollouts])
@pytest.mark.parametrize("graph", [False, True])
def test_queued_calls(edp_lib, make, graph):
    edp = edp_lib
    calls, want, ring = make(edp, 11)
    for f in calls:
        f()
        torch.cuda.synchronize()
    edp.edp_sync(ring.ctx)
    tree = tree_levels(ring) if make is _replay else None
    want = [to_np(t) for t in want]
    ring.close()
    calls, got, ring = make(edp, 11)
    if make is not _replay:  # these repeat themselves: once for the scratch
        for f in calls:
            f()
        torch.cuda.synchronize()
        for t in got:
            t.zero_()
    if graph:
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            for f in calls:
                f()
        g.replay()
    else:
        torch.cuda._sleep(20_000_000)  # about 10 ms, in which all is queued
        for f in calls:
            f()
    torch.cuda.synchronize()
    edp.edp_sync(ring.ctx)
    for i, (w, t) in enumerate(zip(want, got)):
        x = to_np(t)
        assert np.array_equal(w.view(np.uint8), x.view(np.uint8)), i
    if tree is not None:
        for w, x in zip(_flat(tree), _flat(tree_levels(ring))):
            assert np.array_equal(w, x)
    ring.close()
