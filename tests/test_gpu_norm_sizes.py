"""Normalised image delivery against the oracle, bit for bit, where its runs end:
the smallest image with the shortest token row (a CTA touches as many rows as it
can), images a CTA cannot outgrow, batches that end inside a CTA, one round and
two, no tokens, both ways of normalising, one tier and two, with a bad slot, and
importance weights on prioritized rings."""
import numpy as np
import pytest
import torch

from gpu_util import bits, cuda, to_np, u32

pytestmark = pytest.mark.gpu

FMA = ((0.485, 0.456, 0.406, 0.31), (0.229, 0.224, 0.225, 0.27))
# no single FMA gives the bits of this channel 0, so the chain is evaluated
CHAIN = ((0.560784519, 0.456, 0.406, 0.31), (0.604448199, 0.224, 0.225, 0.27))


@pytest.mark.parametrize("C,h,w,L,B,norm,two", [
    (1, 4, 4, 4, 1, FMA, False), (1, 4, 4, 4, 3001, FMA, True), (1, 4, 4, 0, 1025, CHAIN, False),
    (3, 16, 16, 4, 700, FMA, True), (4, 12, 20, 12, 129, CHAIN, True),
    (3, 64, 64, 128, 65, FMA, False), (3, 64, 64, 1028, 66, FMA, True),
    (2, 36, 28, 2048, 33, FMA, False), (3, 96, 96, 0, 1021, FMA, False),
    (1, 512, 512, 4, 5, FMA, False), (3, 512, 516, 8, 7, CHAIN, True)])
def test_norm_sizes(edp_lib, orc, C, h, w, L, B, norm, two):
    edp = edp_lib
    F, cap = C * h * w, 70 if h > 100 else 600
    cap_h = cap // 3 if two else cap
    n = cap + cap // 3
    prio = bool(B % 2)
    rng = np.random.default_rng(F + B + L)
    obs = rng.integers(0, 256, size=(n, F), dtype=np.uint8)
    tok = rng.integers(-9, 1 << 30, size=(n, max(L, 1))).astype(np.int32)
    rew = rng.standard_normal(n).astype(np.float32)
    q = rng.integers(1, 1 << 24, size=n).astype(np.uint32)
    ring = edp.Ring(edp.make_config(cap, (C, h, w), edp.EDP_XFORM_CHW_NORM_BF16, tokens=L,
                                    hbm_capacity=cap_h, prioritized=prio, norm_mean=norm[0],
                                    norm_std=norm[1]), action=False, done=False)
    held = np.zeros((cap, F), np.uint8), np.zeros((cap, max(L, 1)), np.int32), np.zeros(
        cap, np.float32)
    for lo, hi in [(0, cap // 2), (cap // 2, cap), (cap, n)]:
        edp.edp_ingest(ring.ctx, cuda(obs[lo:hi]), hi - lo, reward=cuda(rew[lo:hi]),
                       tokens=cuda(tok[lo:hi]) if L else None,
                       q=cuda(q[lo:hi]) if prio else None)
        for to, new in zip(held, (obs, tok, rew)):
            orc.ring_write(to, cap, lo, np.ascontiguousarray(new[lo:hi]))
    idx = torch.zeros(B, dtype=torch.int64, device="cuda")
    qs = torch.zeros(B, dtype=torch.int32, device="cuda") if prio else None
    isw = torch.full((B,), float("nan"), device="cuda") if prio else None
    edp.edp_sample(ring.ctx, edp.EDP_SAMPLE_PRIORITIZED if prio else edp.EDP_SAMPLE_UNIFORM, B,
                   3, 1, idx, qs)
    if B > 3:
        idx[1] = -4
    out = torch.full((B, F), 7.0, dtype=torch.bfloat16, device="cuda")
    tk = torch.full((B, L), -1, dtype=torch.int32, device="cuda") if L else None
    rw = torch.full((B,), float("nan"), device="cuda")
    edp.edp_deliver(ring.ctx, idx, B, edp.make_batch(out, tokens=tk, reward=rw, q=qs, isw=isw,
                                                     beta=0.7))
    status, _ = edp.edp_sync_status(ring.ctx)
    assert status == (edp.EDP_ERR_INVALID if B > 3 else edp.EDP_OK)
    at = to_np(idx).copy()
    good = at >= 0
    at[~good] = at[0]
    w_obs, w_tok, w_rew = orc.deliver_mm(*held, C, h * w, at, norm[0][:C], norm[1][:C])
    pairs = [(bits(out), w_obs), (bits(rw), w_rew.view(np.uint32))]
    if L:
        pairs.append((to_np(tk), w_tok))
    for got, want in pairs:
        assert np.array_equal(got[good], want[good])
        assert not got[~good].any()
    if prio:
        ulp = to_np(isw).view(np.int32) - orc.is_weights(u32(qs), 0.7).view(np.int32)
        assert np.abs(ulp).max() <= 1
    ring.close()
