"""Frame-stack delivery against the oracle, bit for bit, at frame sizes that
do not divide a warp's span of 128 or 256 words (one 16-byte run more or
less, primes and squares of primes of runs), with and without successors,
stacks of 1 to 16, batches on both sides of the kernel's change of span and
past a multiple of the samples a collating CTA takes; and small frames, which
take the flat kernel (the smallest, whose CTA touches as many samples as it
can, and the largest, on either side of its two larger ranges of words);
importance weights on the prioritized ones."""
import numpy as np
import pytest
import torch

from gpu_util import bits, cuda, dqn_outputs, fx, to_np, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w,K,nxt,B", [
    (4, 1792, 3, True, 129), (4, 1796, 3, True, 400), (92, 92, 3, False, 400),
    (116, 116, 2, True, 60), (16, 1361, 1, False, 97), (16, 64, 4, True, 513),
    (16, 65, 16, True, 70), (32, 32, 1, False, 3000), (4, 260, 5, False, 1),
    (4, 4, 1, False, 777), (4, 4, 1, True, 20_000), (4, 4, 16, True, 65), (8, 16, 4, True, 5),
    (4, 36, 3, False, 40_001), (8, 16, 2, True, 50_000), (4, 188, 16, True, 33),
    (16, 48, 4, True, 1001),
])
def test_frame_sizes(edp_lib, orc, h, w, K, nxt, B):
    edp = edp_lib
    F, cap = h * w, 300
    n = cap + 37
    frames, action, reward, done = fx.dqn_transitions(h * w, n, F, done_p=0.05)
    q = np.random.default_rng(F).integers(1, 1 << 24, size=n).astype(np.uint32)
    prio = bool(B % 2)
    ring = edp.Ring(edp.make_config(cap, (1, h, w), edp.EDP_XFORM_STACK_F32, frame_stack=K,
                                    next_obs=nxt, prioritized=prio))
    r_frames = np.zeros((cap, F), np.uint8)
    r_act, r_rew = np.zeros(cap, np.int32), np.zeros(cap, np.float32)
    r_done = np.zeros(cap, np.uint8)
    for lo, hi in [(0, cap), (cap, n)]:
        edp.edp_ingest(ring.ctx, cuda(frames[lo:hi]), hi - lo, action=cuda(action[lo:hi]),
                       reward=cuda(reward[lo:hi]), done=cuda(done[lo:hi]),
                       q=cuda(q[lo:hi]) if prio else None)
        for dst, src in ((r_frames, frames), (r_act, action), (r_rew, reward), (r_done, done)):
            orc.ring_write(dst, cap, lo, np.ascontiguousarray(src[lo:hi]))
    idx = torch.zeros(B, dtype=torch.int64, device="cuda")
    qs = torch.zeros(B, dtype=torch.int32, device="cuda") if prio else None
    isw = torch.full((B,), float("nan"), device="cuda") if prio else None
    mode = edp.EDP_SAMPLE_PRIORITIZED if prio else edp.EDP_SAMPLE_UNIFORM
    edp.edp_sample(ring.ctx, mode, B, 5, 0, idx, qs)
    if B > 3:
        idx[2] = cap + 9  # a bad slot: zeros
    obs, nx, act, rew, dn = dqn_outputs(B, K, F, with_next=nxt)
    edp.edp_deliver(ring.ctx, idx, B, edp.make_batch(obs, nx, act, rew, dn, q=qs, isw=isw,
                                                     beta=0.5))
    status, _ = edp.edp_sync_status(ring.ctx)
    assert status == (edp.EDP_ERR_INVALID if B > 3 else edp.EDP_OK)
    at = to_np(idx).copy()
    good = at < cap
    at[~good] = at[0]
    want = orc.deliver_dqn(r_frames, r_done, r_act, r_rew, cap, n, K, at, with_next=nxt)
    for got, ref in zip((obs, nx, act, rew, dn), want):
        if got is None:
            continue
        g = bits(got).reshape(B, -1)
        r = ref.view(np.uint32 if ref.dtype == np.float32 else ref.dtype).reshape(B, -1)
        assert np.array_equal(g[good], r[good])
        assert not g[~good].any()
    if prio:
        ulp = to_np(isw).view(np.int32) - orc.is_weights(u32(qs), 0.5).view(np.int32)
        assert np.abs(ulp).max() <= 1
    ring.close()


@pytest.mark.parametrize("h,w,K,B", [(84, 84, 4, 512), (4, 1796, 3, 700), (64, 64, 2, 1501),
                                     (4, 4228, 5, 301), (84, 84, 4, 2300)])
def test_beside_the_sampler(edp_lib, h, w, K, B):
    """A delivery on another stream than the sampling may give its warps twice the
    span (stacks of three frames or more, 2.8 to 16 waves): the same bits as on the
    sampler's stream, with a bad slot and importance weights."""
    edp = edp_lib
    F, cap = h * w, 300
    frames, action, reward, done = fx.dqn_transitions(h + w, cap + 37, F, done_p=0.05)
    ring = edp.Ring(edp.make_config(cap, (1, h, w), edp.EDP_XFORM_STACK_F32, frame_stack=K,
                                    next_obs=True, prioritized=True))
    for lo, hi in [(0, cap), (cap, cap + 37)]:
        edp.edp_ingest(ring.ctx, cuda(frames[lo:hi]), hi - lo, action=cuda(action[lo:hi]),
                       reward=cuda(reward[lo:hi]), done=cuda(done[lo:hi]))
    idx = torch.zeros(B, dtype=torch.int64, device="cuda")
    q = torch.zeros(B, dtype=torch.int32, device="cuda")
    edp.edp_sample(ring.ctx, edp.EDP_SAMPLE_PRIORITIZED, B, 5, 0, idx, q)
    idx[B // 2] = cap + 1
    outs = []
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        out = list(dqn_outputs(B, K, F)) + [torch.full((B,), -1.0, device="cuda")]
        torch.cuda.synchronize()
        edp.edp_deliver(ring.ctx, idx, B, edp.make_batch(*out[:5], q=q, isw=out[5], beta=0.5),
                        stream=stream)
        assert edp.edp_sync_status(ring.ctx, stream)[0] == edp.EDP_ERR_INVALID
        outs.append([bits(t) for t in out])
    for x, y in zip(*outs):
        assert np.array_equal(x, y)
    ring.close()
