"""The tiled blur passes of the real-scan preprocessing at the edges of their tiles: lines and segments that
do not fill a tile, one-pixel images, radii below, at and above the register window, results written over
the input, and non-finite pixels (which reach exactly the pixels within the radius)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _blur(x, sigma):
    from oracle import filters
    return np.stack([filters.blur(v, sigma) for v in x]) if sigma > 0 else x


@pytest.mark.parametrize("n,H,W,sigma", [(1, 1, 1, 1.0), (3, 5, 7, 5.0), (2, 257, 33, 0.3), (1, 300, 523, 32.0),
                                         (40, 16, 16, 5.3), (2, 31, 256, 2.5), (1, 256, 257, 2.7), (5, 272, 48, 12.0)])
def test_blur_passes_parity(n, H, W, sigma):
    import torch
    import paper_1907_05993_gb300 as P
    rng = np.random.default_rng(n * H + W)
    x = rng.uniform(0.5, 2.0, (n, H, W)).astype(np.float32)
    x64 = x.astype(np.float64)
    bg = rng.uniform(0.5, 2.0, (H, W)).astype(np.float32)
    dev = lambda a: torch.from_numpy(a.copy()).cuda()
    ctx = P.hrebsd_create(0)
    # FP32: a pass of T taps errs by at most (T + 1) u max|x|, two passes by twice that
    tol = 2 * (2 * math.ceil(3 * sigma) + 2) * 2.0 ** -24 * 2.0
    out = torch.empty((n, H, W), device="cuda")
    P.hrebsd_bandpass_batch(ctx, dev(x), n, H, W, sigma, 0.0, out)
    low = _blur(x64, sigma)
    assert np.abs(out.cpu().numpy() - low).max() <= tol
    d = dev(x)
    P.hrebsd_bandpass_batch(ctx, d, n, H, W, 0.5, sigma, d)   # over the input
    assert np.abs(d.cpu().numpy() - (_blur(x64, 0.5) - low)).max() <= tol + 2 * 6 * 2.0 ** -24 * 2.0 + 2.0 ** -22
    corr = x64 / bg.astype(np.float64)
    d = dev(x)
    P.hrebsd_background_batch(ctx, d, n, H, W, dev(bg), sigma, d)
    exp = corr / _blur(corr, sigma)
    assert np.abs(d.cpu().numpy() / exp - 1).max() <= 2 * tol / 0.25 + 2.0 ** -21
    P.hrebsd_background_batch(ctx, dev(x), n, H, W, None, sigma, out)
    assert np.abs(out.cpu().numpy() / (x64 / low) - 1).max() <= 2 * tol / 0.5 + 2.0 ** -21
    mean = torch.empty((H, W), device="cuda")
    P.hrebsd_mean_pattern(ctx, dev(x), n, H, W, mean)
    assert np.abs(mean.cpu().numpy() - x64.mean(axis=0)).max() <= 2.0 ** -24 * 1.01 * 2.0
    # a NaN and an infinity spread over the radius and no further
    x[0, H // 2, W // 3] = np.nan
    x[n - 1, 0, W - 1] = np.inf
    P.hrebsd_bandpass_batch(ctx, dev(x), n, H, W, sigma, 0.0, out)
    r = math.ceil(3 * sigma)
    yy, xx = np.mgrid[0:H, 0:W]
    bad = np.zeros((n, H, W), bool)
    bad[0] |= (abs(yy - H // 2) <= r) & (abs(xx - W // 3) <= r)
    bad[n - 1] |= (yy <= r) & (W - 1 - xx <= r)
    assert np.array_equal(~np.isfinite(out.cpu().numpy()), bad)
    P.hrebsd_destroy(ctx)


@pytest.mark.parametrize("n", [1, 7, 8, 33, 100])
def test_mean_pattern_groups(n):
    import torch
    import paper_1907_05993_gb300 as P
    x = np.random.default_rng(n).normal(100, 30, (n, 9, 11)).astype(np.float32)
    ctx = P.hrebsd_create(0)
    mean = torch.empty((9, 11), device="cuda")
    P.hrebsd_mean_pattern(ctx, torch.from_numpy(x).cuda(), n, 9, 11, mean)
    P.hrebsd_destroy(ctx)
    exp = x.astype(np.float64).mean(axis=0)
    assert (np.abs(mean.cpu().numpy() - exp) <= np.spacing(exp.astype(np.float32)) * 0.51).all()
