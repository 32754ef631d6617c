"""A ring that the cyclic garbage collector finds while its thread captures a
CUDA graph (a test's or a program's exception that kept the frame alive is
enough) must not break the capture: destroying a context synchronises and
frees, neither of which a capture allows.  It is destroyed later instead."""
import gc

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_ring_collected_during_capture(edp_lib):
    edp = edp_lib

    def make():
        return edp.Ring(edp.make_config(16, (1, 4, 4), edp.EDP_XFORM_HWC_CHW_BF16))

    gc.collect()  # rings of earlier tests are not collected in the capture
    lost = make()
    lost.itself = lost  # only the cyclic collector can find it
    ctx = lost.ctx
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    gc.disable()
    try:
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            x += 1
            del lost
            gc.collect()
    finally:
        gc.enable()
    assert [w["ctx"] for w in edp.Ring._waiting] == [ctx]
    g.replay()
    torch.cuda.synchronize()
    assert (x == 1).all()
    make().close()  # a ring made outside a capture destroys what waits
    assert not edp.Ring._waiting
