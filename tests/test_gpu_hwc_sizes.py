"""HWC -> CHW bf16 delivery against the oracle, bit for bit, from the smallest
image (two 8-pixel groups, so that a CTA touches as many images as it can) to
one whose images a CTA cannot outgrow, 1 to 4 channels, batches that end
inside a CTA, with a bad slot; gathered scalars, and importance weights on
prioritized rings."""
import numpy as np
import pytest
import torch

from gpu_util import bits, cuda, to_np, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w,C,B", [(4, 4, 1, 1), (4, 4, 1, 3001), (4, 4, 4, 1025),
                                     (4, 4, 3, 127), (8, 16, 1, 5000), (12, 20, 2, 700),
                                     (36, 28, 3, 129), (84, 84, 4, 33), (512, 512, 1, 5),
                                     (512, 516, 3, 4)])
def test_hwc_sizes(edp_lib, orc, h, w, C, B):
    edp = edp_lib
    F, cap = h * w * C, 70 if h > 100 else 900
    n = cap + cap // 3
    prio = bool(B % 2)
    rng = np.random.default_rng(F + B)
    obs = rng.integers(0, 256, size=(n, F), dtype=np.uint8)
    q = rng.integers(1, 1 << 24, size=n).astype(np.uint32)
    ring = edp.Ring(edp.make_config(cap, (C, h, w), edp.EDP_XFORM_HWC_CHW_BF16,
                                    prioritized=prio), action=False, reward=False, done=False)
    held = np.zeros((cap, F), np.uint8)
    for lo, hi in [(0, cap), (cap, n)]:
        edp.edp_ingest(ring.ctx, cuda(obs[lo:hi]), hi - lo, q=cuda(q[lo:hi]) if prio else None)
        orc.ring_write(held, cap, lo, np.ascontiguousarray(obs[lo:hi]))
    adv = rng.standard_normal(cap).astype(np.float32)
    ret = rng.standard_normal(cap).astype(np.float32)
    idx = torch.zeros(B, dtype=torch.int64, device="cuda")
    qs = torch.zeros(B, dtype=torch.int32, device="cuda") if prio else None
    isw = torch.full((B,), float("nan"), device="cuda") if prio else None
    edp.edp_sample(ring.ctx, edp.EDP_SAMPLE_PRIORITIZED if prio else edp.EDP_SAMPLE_UNIFORM, B,
                   3, 1, idx, qs)
    if B > 3:
        idx[1] = -4
    out = torch.full((B, F), 7.0, dtype=torch.bfloat16, device="cuda")
    a, r = (torch.full((B,), float("nan"), device="cuda") for _ in range(2))
    edp.edp_deliver(ring.ctx, idx, B, edp.make_batch(
        out, q=qs, isw=isw, beta=0.7, gather=[(cuda(adv), a), (cuda(ret), r)]))
    status, _ = edp.edp_sync_status(ring.ctx)
    assert status == (edp.EDP_ERR_INVALID if B > 3 else edp.EDP_OK)
    at = to_np(idx).copy()
    good = at >= 0
    at[~good] = at[0]
    w_obs, w_a, w_r = orc.deliver_ppo(held, cap, n, h, w, C, at, adv, ret)
    for got, want in ((bits(out), w_obs.reshape(B, -1)), (bits(a), w_a.view(np.uint32)),
                      (bits(r), w_r.view(np.uint32))):
        assert np.array_equal(got[good], want[good])
        assert not got[~good].any()
    if prio:
        ulp = to_np(isw).view(np.int32) - orc.is_weights(u32(qs), 0.7).view(np.int32)
        assert np.abs(ulp).max() <= 1
    ring.close()
