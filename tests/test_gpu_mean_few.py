"""The mean over the patterns at every split of the images: few images (one thread per pixel) and many (groups that
share a pixel), the correctly rounded mean either way; and a few patterns cost little more than their read."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 31, 32, 128])
@pytest.mark.parametrize("H,W", [(1, 1), (9, 31), (256, 130)])
def test_mean_at_the_edges_of_the_split(n, H, W):
    import torch
    import paper_1907_05993_gb300 as P
    rng = np.random.default_rng(n * H + W)
    x = (rng.normal(100, 30, (n, H, W)) * 10.0 ** rng.integers(-3, 4, (n, 1, 1))).astype(np.float32)
    if n > 2:
        x[0, 0, 0], x[1, 0, 0] = 3e38, 3e38   # leaves FP32: summed in FP64
    ctx = P.hrebsd_create(0)
    mean = torch.empty((H, W), device="cuda")
    P.hrebsd_mean_pattern(ctx, torch.from_numpy(x).cuda(), n, H, W, mean)
    P.hrebsd_destroy(ctx)
    exp = x.astype(np.float64).mean(axis=0)
    # one rounding to FP32, of a sum in FP64 where it left FP32 (relative 2^-52 per term of the largest)
    assert (np.abs(mean.cpu().numpy() - exp) <= np.spacing(np.abs(exp).astype(np.float32)) * 0.51).all()


@pytest.mark.parametrize("n", [1, 4])
def test_mean_of_a_few_patterns_is_quick(n):
    """A read of 5 to 20 MB: 28 and 43 us with one thread per pixel, 156 with 32 pixels to a CTA."""
    import torch
    import paper_1907_05993_gb300 as P
    ctx = P.hrebsd_create(0)
    x, mean = torch.rand((n, 1024, 1244), device="cuda"), torch.empty((1024, 1244), device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(8):
            P.hrebsd_mean_pattern(ctx, x, n, 1024, 1244, mean)
    best = 1e9
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / 8 * 1e3)
    P.hrebsd_destroy(ctx)
    assert best <= 80.0, best
