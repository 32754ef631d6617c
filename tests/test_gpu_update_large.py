"""Priority updates above the single-pass kernel's 2,048 pairs: at the edges
of the scan's chunk of 8,192 pairs, with every pair on one slot, with few
slots, with every pair of one owner CTA (more than its list and table hold: they
are then applied in parts), and with more distinct slots of one owner than its
table.  Every node of the tree against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from gpu_util import MirroredDqn, check_tree, cuda, fx, u32

pytestmark = pytest.mark.gpu

ALPHA, EPS = 0.6, 1e-6
CAP, FILL = 200_000, 230_000


@pytest.fixture(scope="module")
def big(edp_lib, orc):
    frames, action, reward, done = fx.dqn_transitions(41, FILL, 84 * 4)
    q = orc.priorities_from_td(fx.td_errors(41, FILL), ALPHA, EPS)
    m = MirroredDqn(CAP, F=84 * 4, prioritized=True)
    for lo, hi in [(0, CAP), (CAP, FILL)]:
        m.ingest(orc, frames[lo:hi], action[lo:hi], reward[lo:hi], done[lo:hi], q=q[lo:hi])
    yield m
    m.ring.close()


def _one_owner(n, cap=CAP):
    """Slots that one CTA of an n-pair update owns (the kernel's split)."""
    grid = min((n + 63) // 64, torch.cuda.get_device_properties(0).multi_processor_count)
    s = np.arange(cap, dtype=np.uint64)
    owner = (((s * np.uint64(0x9E3779B1)) & np.uint64(0xFFFFFFFF)) * np.uint64(grid)) >> np.uint64(32)
    return np.flatnonzero(owner == 1)


@pytest.mark.parametrize("n", [2049, 8191, 8192, 8193, 16384, 30011])
@pytest.mark.parametrize("slots", ["spread", "one", "few", "owner"])
def test_large_update(edp_lib, orc, big, n, slots):
    edp, m = edp_lib, big
    rng = np.random.default_rng(n)
    pick = {"spread": np.arange(CAP), "one": np.array([77]), "few": np.arange(100, 140),
            "owner": _one_owner(n)}[slots]
    idx = rng.choice(pick, size=n).astype(np.int64)
    idx[n // 2] = idx[3]
    idx[7] = (m.total - 1) % CAP  # the newest transition: deferred priority
    if n % 2:
        qu = rng.integers(0, 1 << 32, size=n, dtype=np.uint64).astype(np.uint32)
        edp.edp_update_priorities(m.ring.ctx, cuda(idx), cuda(qu), n)
    else:
        td = cuda(fx.td_errors(n, n))
        qd = torch.zeros(n, dtype=torch.int32, device="cuda")
        edp.edp_priorities_from_td(m.ring.ctx, td, n, ALPHA, EPS, qd)
        edp.edp_update_priorities_td(m.ring.ctx, cuda(idx), td, n, ALPHA, EPS)
        qu = u32(qd)
    edp.edp_sync(m.ring.ctx)
    orc.update_leaves(m.st, m.total, idx, qu)
    check_tree(orc, m.ring, m.st)


@pytest.mark.parametrize("slots", ["spread", "few"])
def test_beyond_the_list(edp_lib, orc, big, slots):
    """More pairs per CTA than the scan lists: entered in batch order."""
    edp, m = edp_lib, big
    n = 1024 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    rng = np.random.default_rng(5)
    idx = rng.choice(CAP if slots == "spread" else 40, size=n).astype(np.int64)
    qu = rng.integers(0, 1 << 32, size=n, dtype=np.uint64).astype(np.uint32)
    edp.edp_update_priorities(m.ring.ctx, cuda(idx), cuda(qu), n)
    edp.edp_sync(m.ring.ctx)
    orc.update_leaves(m.st, m.total, idx, qu)
    check_tree(orc, m.ring, m.st)


@pytest.mark.parametrize("n", [8192, 30_011])
def test_more_slots_of_one_owner_than_its_table(edp_lib, orc, n):
    edp, cap, fill = edp_lib, 600_000, 600_500
    rng = np.random.default_rng(n)
    m = MirroredDqn(cap, F=84 * 4, prioritized=True)
    q = rng.integers(1, 1 << 24, size=fill).astype(np.uint32)
    for lo, hi in [(0, cap), (cap, fill)]:
        k = hi - lo
        m.ingest(orc, np.zeros((k, 84 * 4), np.uint8), np.zeros(k, np.int32),
                 np.zeros(k, np.float32), np.zeros(k, np.uint8), q=q[lo:hi])
    idx = rng.choice(_one_owner(n, cap), size=n).astype(np.int64)
    assert len(np.unique(idx)) > 3072  # the table takes no more
    idx[5] = (m.total - 1) % cap
    qu = rng.integers(0, 1 << 32, size=n, dtype=np.uint64).astype(np.uint32)
    edp.edp_update_priorities(m.ring.ctx, cuda(idx), cuda(qu), n)
    edp.edp_sync(m.ring.ctx)
    orc.update_leaves(m.st, m.total, idx, qu)
    check_tree(orc, m.ring, m.st)
    m.ring.close()
