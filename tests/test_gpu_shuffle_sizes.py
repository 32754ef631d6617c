"""The shuffle against the oracle at the sizes where its split changes: one
bucket, few buckets per CTA, the most buckets (from 32,769 elements on they
grow), and buckets that span several shared-memory tiles; twice each, so
that the second call finds the counters the first left."""
import numpy as np
import pytest
import torch

from gpu_util import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 5, 255, 257, 1000, 32768, 32769, 262144, 1_000_003,
                               9_000_000])
def test_shuffle_sizes(edp_lib, orc, n):
    edp = edp_lib
    cap = n + n // 3
    ring = edp.Ring(edp.make_config(cap, (1, 4, 4), edp.EDP_XFORM_HWC_CHW_BF16), action=False,
                    reward=False, done=False)
    rows = torch.zeros(cap * 16, dtype=torch.uint8, device="cuda")
    if n % 2:  # full and wrapped: the oldest transition is not in slot 0
        cap_n = cap
        edp.edp_ingest(ring.ctx, rows, cap)
        edp.edp_ingest(ring.ctx, rows, n // 3)
        oldest = (n // 3) % cap
    else:
        cap_n, oldest = n, 0
        edp.edp_ingest(ring.ctx, rows, n)
    idx = torch.full((cap_n,), -1, dtype=torch.int64, device="cuda")
    for rnd in range(2):
        edp.edp_sample(ring.ctx, edp.EDP_SAMPLE_PERMUTE, cap_n, 9, rnd, idx)
        edp.edp_sync(ring.ctx)
        assert np.array_equal(to_np(idx), (oldest + orc.permutation(cap_n, 9, rnd)) % cap)
    ring.close()
