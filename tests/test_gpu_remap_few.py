"""The remap by one and by four rows per thread: a pair gives the same bits alone (single rows) as in batches of every
size around the rules between them, and one pair takes no longer than a row does."""
import math

import numpy as np
import pytest

from synth import kikuchi as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(33, 40), (64, 64), (61, 300)])
def test_a_pair_alone_equals_the_pair_in_a_batch(H, W):
    import torch
    import paper_1907_05993_gb300 as P
    rng = np.random.default_rng(H)
    ref = torch.from_numpy(rng.standard_normal((1, H, W)).astype(np.float32)).cuda()
    Rs = np.stack([K.axis_angle(rng.normal(size=3), math.radians(a)).reshape(9) for a in (0.0, 2.0, 7.0)])
    geom, ctx = P.hrebsd_geometry(0.5, 0.5, 0.6), P.hrebsd_create(0)

    def run(B):
        R = torch.from_numpy(Rs[np.arange(B) % 3].copy()).cuda()
        out = torch.empty((B, H, W), device="cuda")
        P.hrebsd_remap(ctx, ref, torch.zeros(B, dtype=torch.int32, device="cuda"), R, B, H, W, geom, out)
        return out.cpu().numpy()

    few = run(3)
    for B in (6, 17, 18, 19, 36, 37, 40, 75, 76, 77, 150, 152, 160, 700):
        out = run(B)
        for b in (0, 1, 2, B - 2, B - 1):
            assert np.array_equal(out[b], few[b % 3]), (B, b)
    P.hrebsd_destroy(ctx)


def test_one_pair_is_quick():
    """2.5 to 2.8 us by single rows, 4.1 to 4.4 by four rows per thread."""
    import torch
    import paper_1907_05993_gb300 as P
    ctx, geom = P.hrebsd_create(0), P.hrebsd_geometry(0.5, 0.5, 0.6)
    ref, out = torch.rand((1, 128, 128), device="cuda"), torch.empty((1, 128, 128), device="cuda")
    R = torch.eye(3, dtype=torch.float64, device="cuda").reshape(1, 9)
    idx = torch.zeros(1, dtype=torch.int32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(32):
            P.hrebsd_remap(ctx, ref, idx, R, 1, 128, 128, geom, out)
    best = 1e9
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / 32 * 1e3)
    P.hrebsd_destroy(ctx)
    assert best <= 3.9, best
