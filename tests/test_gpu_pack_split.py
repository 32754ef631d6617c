"""Packed delivery against the oracle where the way it is copied changes with
the batch and the room: many short sequences, one to four per warp, with a few
that a whole CTA copies, and a CTA's sequences cut by the end of the room; long
ones among many short that their own CTA keeps or a list deals out; few
long sequences over several CTAs each, in chunks of 1,024 to 4,096 tokens, and
a long one that the room does not announce."""
import numpy as np
import pytest
import torch

from gpu_util import cuda, to_np

from oracle import llm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ring(edp_lib):
    r = edp_lib.Ring(edp_lib.make_config(16, (1, 4, 4), edp_lib.EDP_XFORM_HWC_CHW_BF16),
                     action=False, reward=False, done=False)
    yield r
    r.close()


@pytest.mark.parametrize("B,lmax,longer,room,values", [
    (1000, 90, 3000, 1000 * 200, True),      # one per warp, three by whole CTAs
    (15_000, 60, 1025, 15_000 * 64, True),   # two per warp
    (60_003, 40, 5000, 60_003 * 64, False),  # four per warp, a ragged last CTA
    (60_003, 40, 9000, 700_000, True),       # the room ends inside a CTA
    (1, 20_000, 0, 20_000, True),            # one sequence over 20 CTAs
    (7, 9000, 0, 7 * 9000, True),
    (300, 6000, 0, 300 * 6000, False),
    (5, 50, 30_000, 40_000, True),           # the long one is not announced
])
def test_pack_ways(edp_lib, ring, B, lmax, longer, room, values):
    edp = edp_lib
    rng = np.random.default_rng(B + lmax)
    n = B + 11
    lens = rng.integers(0, lmax + 1, size=n)
    lens[0] = lmax
    if longer:
        lens[rng.integers(0, n, size=3)] = longer
    off = np.zeros(n + 1, np.uint64)
    np.cumsum(lens, out=off[1:])
    tokens = rng.integers(0, 1 << 30, size=int(off[-1]) + 1, dtype=np.int32)
    idx = rng.permutation(n)[:B].astype(np.int64)
    idx[B // 2] = 0
    bad = B > 100
    if bad:
        idx[B // 3] = n + 5
    val = rng.standard_normal(n).astype(np.float32)
    ot = torch.full((room + 8,), -3, dtype=torch.int32, device="cuda")
    ov = torch.full((room + 8,), -3.0, device="cuda") if values else None
    oo = torch.zeros(B + 1, dtype=torch.int64, device="cuda")
    want, want_off, want_val = llm.pack(tokens, off, idx, val)
    fits = len(want) <= room
    m = min(len(want), room)
    edp.edp_pack_deliver(ring.ctx, cuda(tokens), cuda(off), n, cuda(idx), B, ot, oo, room,
                         seq_value=cuda(val) if values else None, out_value=ov)
    status, msg = edp.edp_sync_status(ring.ctx)
    assert status == (edp.EDP_ERR_INVALID if bad or not fits else edp.EDP_OK), msg
    assert np.array_equal(to_np(oo).view(np.uint64), want_off)
    assert np.array_equal(to_np(ot)[:m], want[:m]) and (to_np(ot)[m:] == -3).all()
    if values:
        assert np.array_equal(to_np(ov)[:m], want_val[:m]) and (to_np(ov)[m:] == -3).all()


@pytest.mark.parametrize("B,long,each,first,room", [
    (913, 20, 16_000, True, None), (1000, 900, 1025, False, None),
    (2000, 200, 4097, False, 300_000), (7288, 1500, 2000, True, None),
    (7297, 1500, 2000, True, None),           # three of a CTA's eight kept, five listed
    (8192, 4096, 1500, False, None), (20_000, 2500, 6144, True, None),
    (20_000, 400, 6145, False, 2_000_000), (60_003, 1300, 16_000, True, None),
    (70_000, 3000, 1100, False, None)])
def test_long_among_short(edp_lib, ring, B, long, each, first, room):
    """Long sequences at the head of the batch or anywhere in it, cut by the end
    of the room or not; then a batch without any and one with other long ones (the
    list starts empty in each call)."""
    edp = edp_lib
    rng = np.random.default_rng(B)
    for n_long in (long, 0, long // 3 + 1):
        lens = rng.integers(0, 40, size=B)
        lens[:n_long] = each
        if n_long:
            lens[n_long - 1] = 1024  # the longest that a warp copies
        order = np.arange(B) if first else rng.permutation(B)
        off = np.zeros(B + 1, np.uint64)
        np.cumsum(lens, out=off[1:])
        tokens = rng.integers(0, 1 << 30, size=int(off[-1]) + 1, dtype=np.int32)
        val = rng.standard_normal(B).astype(np.float32)
        want, want_off, want_val = llm.pack(tokens, off, order.astype(np.int64), val)
        cap = room if room else len(want)
        m = min(len(want), cap)
        ot = torch.full((cap + 8,), -3, dtype=torch.int32, device="cuda")
        ov = torch.full((cap + 8,), -3.0, device="cuda")
        oo = torch.zeros(B + 1, dtype=torch.int64, device="cuda")
        edp.edp_pack_deliver(ring.ctx, cuda(tokens), cuda(off), B, cuda(order.astype(np.int64)), B,
                             ot, oo, cap, seq_value=cuda(val), out_value=ov)
        status, msg = edp.edp_sync_status(ring.ctx)
        assert status == (edp.EDP_OK if len(want) <= cap else edp.EDP_ERR_INVALID), msg
        assert np.array_equal(to_np(oo).view(np.uint64), want_off)
        assert np.array_equal(to_np(ot)[:m], want[:m]) and (to_np(ot)[m:] == -3).all()
        assert np.array_equal(to_np(ov)[:m], want_val[:m]) and (to_np(ov)[m:] == -3).all()
