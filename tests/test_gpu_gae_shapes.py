"""Advantages against the oracle at the shapes where the scan's split changes:
one step, one environment, a segment and a chunk more or less, few
environments over several chunks (fewer environments per CTA), a rollout that
one CTA normalises, many environments; arrays off 16-byte alignment, and each
output alone.  The bound is the rounding of the stored fp32 advantages: 4 ulp
of the value, or of the rollout's largest where it cancels."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

from gpu_util import cuda, to_np

pytestmark = pytest.mark.gpu


def _shifted(x, k):
    """x on the device, k elements past an aligned address."""
    flat = torch.zeros(x.numel() + 8, dtype=x.dtype, device="cuda")
    out = flat[k:k + x.numel()].view(x.shape)
    out.copy_(x)
    return out


@pytest.mark.parametrize("T,E", [(1, 1), (1, 9), (3, 8), (4, 1), (5, 16), (128, 8), (256, 8),
                                 (257, 8), (512, 9), (513, 8), (2048, 1), (2049, 3), (1000, 7),
                                 (5000, 2), (8192, 64), (64, 1001), (300, 610), (17, 5000)])
def test_gae_shapes(edp_lib, orc, T, E):
    edp = edp_lib
    rng = np.random.default_rng(T * 10007 + E)
    r = rng.standard_normal((T, E)).astype(np.float32)
    v = rng.standard_normal((T + 1, E)).astype(np.float32)
    d = (rng.random((T, E)) < 0.01).astype(np.uint8)
    ring = edp.Ring(edp.make_config(16, (1, 4, 4), edp.EDP_XFORM_HWC_CHW_BF16), action=False,
                    reward=False, done=False)
    A, R = orc.gae(r, v, d, 0.99, 0.95)
    N, _, _ = orc.normalize(A)
    want = dict(adv=A, ret=R, adv_norm=N)
    for k, keep in enumerate([("adv", "ret", "adv_norm"), ("adv_norm",), ("ret", "adv_norm"),
                              ("ret",), ("adv",)]):
        out = {n: _shifted(torch.full((T, E), float("nan")), k % 4) for n in keep}
        edp.edp_gae(ring.ctx, _shifted(cuda(r), k), _shifted(cuda(v), 1), _shifted(cuda(d), 3), T,
                    E, 0.99, 0.95, **out)
        edp.edp_sync(ring.ctx)
        for n in keep:
            ref = np.asarray(want[n], np.float64).reshape(T, E)
            bound = 4 * 2.0**-24 * np.maximum(np.abs(ref), np.abs(ref).max())
            assert (np.abs(to_np(out[n]) - ref) <= bound).all(), (n, keep)
    stats = torch.zeros(3, dtype=torch.float64, device="cuda")
    adv = torch.zeros(T, E, device="cuda")
    edp.edp_gae_stats(ring.ctx, cuda(r), cuda(v), cuda(d), T, E, 0.99, 0.95, adv, stats)
    edp.edp_gae_normalize(ring.ctx, adv, T * E, stats, adv)
    edp.edp_sync(ring.ctx)
    a64 = np.asarray(A, np.float64)
    s = to_np(stats)
    assert s[0] == T * E
    assert abs(s[1] - a64.sum()) <= 1e-11 * np.abs(a64).sum()
    assert abs(s[2] - (a64**2).sum()) <= 1e-11 * (a64**2).sum()
    ref = np.asarray(N, np.float64).reshape(T, E)
    assert (np.abs(to_np(adv) - ref) <= 4 * 2.0**-24 * np.maximum(
        np.abs(ref), np.abs(ref).max())).all()
    ring.close()


@pytest.mark.parametrize("T,E", [(2048, 1), (128, 8), (2048, 8), (8192, 2), (128, 256)])
@pytest.mark.parametrize("mean", [0.0, 10.0, 1e3, 1e5])
def test_sums_keep_64_bits(edp_lib, T, E, mean):
    """Sums of A and A^2 of advantages whose mean is up to 1e5 of their
    deviations (the variance is a difference of the two): every step ends an
    episode and V = 0, so A = r.  The bound on the root mean square over 24
    rollouts is 2^-52, two roundings to fp64 (a CTA's sums round once, their sum
    again: 1.3e-16 at most); double-float over a CTA gave 5e-16 to 2e-15 in the
    first four shapes, fp64 behind double-float over a thread 3e-16 to 4e-15."""
    edp = edp_lib
    ring = edp.Ring(edp.make_config(16, (1, 4, 4), edp.EDP_XFORM_HWC_CHW_BF16), action=False,
                    reward=False, done=False)
    v = torch.zeros(T + 1, E, device="cuda")
    d = torch.ones(T, E, dtype=torch.uint8, device="cuda")
    adv = torch.zeros(T, E, device="cuda")
    stats = torch.zeros(3, dtype=torch.float64, device="cuda")
    off = []
    for seed in range(24):
        rng = np.random.default_rng(seed * 1000 + T + E)
        r = (mean + rng.standard_normal((T, E))).astype(np.float32)
        edp.edp_gae_stats(ring.ctx, cuda(r), v, d, T, E, 0.99, 0.95, adv, stats)
        edp.edp_sync(ring.ctx)
        n, s1, s2 = to_np(stats)
        assert n == T * E and np.array_equal(to_np(adv), r)
        x = r.astype(np.float64).ravel()
        want = math.fsum(x * x)  # the squares of fp32 values are exact in fp64
        off.append((s2 - want) / want)
        assert abs(s1 - math.fsum(x)) <= 2.0**-51 * math.fsum(np.abs(x))
    assert math.sqrt(np.mean(np.square(off))) <= 2.0**-52
    ring.close()


@pytest.mark.parametrize("mean,std", [(1000.37, 1.0), (-731.0123456789, 0.9), (3e-4, 1.7),
                                      (0.0, 2.5), (-5e12, 7e9), (2e-19, 1e-18), (1.25, 0.0)])
def test_normalised_values_round_once(edp_lib, mean, std):
    """(A - mean) / (std + 1e-8) for values next to the mean, where the
    difference cancels, and for ordinary, large and infinite ones: within 0.51 ulp
    of the exact product of fp64's mean and scale (half an ulp is the result's
    own rounding; fp64 arithmetic gives 0.56 at a mean of 1e3 deviations, a mean
    held in two fp32 words 2).  The scale is formed from s2 - s1 mean, contracted
    or not: the two differ by 2^-53 s2, below 1e-9 of the variance for a mean of
    up to 1e3 deviations and nothing at all at 1.25 (exact products)."""
    edp = edp_lib
    ring = edp.Ring(edp.make_config(16, (1, 4, 4), edp.EDP_XFORM_HWC_CHW_BF16), action=False,
                    reward=False, done=False)
    nn = 4096.0
    s1 = nn * mean
    m = s1 / nn
    s2 = s1 * m + (nn - 1.0) * std * std
    inv = 1.0 / (math.sqrt(max((s2 - s1 * m) / (nn - 1.0), 0.0)) + 1e-8)
    near = np.float32(m) + np.spacing(np.float32(m)) * np.arange(-300, 301, dtype=np.float32)
    rng = np.random.default_rng(1)
    x = np.concatenate([near, (m + (std + 1e-8) * rng.standard_normal(400)), [0.0, 1e30, -2e19]])
    a = np.concatenate([x.astype(np.float32), np.array([np.inf, -np.inf, np.nan], np.float32)])
    stats = torch.tensor([nn, s1, s2], dtype=torch.float64, device="cuda")
    out = torch.zeros(len(a), device="cuda")
    edp.edp_gae_normalize(ring.ctx, cuda(a), len(a), stats, out)
    edp.edp_sync(ring.ctx)
    y = to_np(out)
    assert y[-3] == np.inf and y[-2] == -np.inf and np.isnan(y[-1])
    for got, v in zip(y[:-3], a[:-3]):
        want = (Fraction(float(v)) - Fraction(m)) * Fraction(inv)
        if abs(want) > 3e38:
            assert np.isinf(got) and (got > 0) == (want > 0)
            continue
        ulp = Fraction(float(np.spacing(np.float32(abs(float(want))))))
        assert abs(Fraction(float(got)) - want) <= Fraction(51, 100) * ulp, (v, got)
    ring.close()
