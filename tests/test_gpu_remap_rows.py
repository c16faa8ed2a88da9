"""The remap's row groups: heights that are no multiple of a group, patterns narrower than a warp and wider
than a block, and patterns too small for an unclamped footprint."""
import math

import numpy as np
import pytest

from synth import kikuchi as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,B", [(2, 2, 1), (3, 5, 2), (5, 3, 3), (9, 40, 5), (33, 300, 2), (6, 513, 1), (31, 31, 700)])
def test_remap_row_groups(H, W, B):
    import torch
    import oracle
    import paper_1907_05993_gb300 as P
    rng, geom = np.random.default_rng(H + W), K.Geometry()
    refs = rng.standard_normal((2, H, W)).astype(np.float32)
    Rs = np.stack([K.axis_angle(rng.normal(size=3), math.radians(rng.uniform(0, 8))) for _ in range(min(B, 4))])
    idx = (np.arange(B) % 2).astype(np.int32)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)
    out = torch.empty((B, H, W), device="cuda")
    ctx = P.hrebsd_create(0)
    P.hrebsd_remap(ctx, dev(refs, torch.float32), dev(idx, torch.int32), dev(Rs[np.arange(B) % len(Rs)].reshape(B, 9), torch.float64),
                   B, H, W, P.hrebsd_geometry(geom.xstar, geom.ystar, geom.zstar), out)
    P.hrebsd_destroy(ctx)
    got = out.cpu().numpy()
    # FP32 coordinates: a few roundings of numbers up to 2 W, times the slope of white noise (at most ~6 per px)
    tol = 6.0 * 8 * 2 * W * 2.0 ** -24 + 1e-5
    for b in range(min(B, 4)):
        assert np.abs(got[b] - oracle.remap(refs[idx[b]].astype(np.float64), Rs[b % len(Rs)], geom)).max() <= tol
    for b in range(4, B):
        assert np.array_equal(got[b], got[b % 4])
