"""A level's cached graph ends in the prolongation to the next finer level, so a size that shares a coarse level
with an earlier one (100 and 101 rows are both 50 at level 1) must not replay that one's launches: calls of
several sizes on one context, in the same buffers, against a context of its own for each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pin", [False, True])
@pytest.mark.parametrize("sizes", [[(100, 92), (101, 92), (100, 92)], [(100, 92), (100, 93), (101, 93)]])
def test_sizes_that_share_a_coarse_level(sizes, pin):
    import torch
    import paper_1907_05993_gb300 as P
    B, R, L = 3, 2, 2
    big = max(h * w for h, w in sizes)
    buf = {k: torch.empty(n * big, device="cuda") for k, n in (("ref", R), ("test", B), ("field", 2 * B))}
    idx = torch.tensor([0, 1, 1], dtype=torch.int32, device="cuda")
    iters = torch.empty((B, L), dtype=torch.int32, device="cuda")
    status = torch.empty((B,), dtype=torch.int32, device="cuda")
    prm = P.demons_params(L, [8, 8])

    def run(ctx, H, W):
        rng = np.random.default_rng(H * W)
        y, x = np.mgrid[0:H, 0:W]
        img = lambda s: np.cos(0.21 * x + s) + np.cos(0.17 * y - 0.1 * x + 2 * s) + 0.05 * rng.standard_normal((H, W))
        view = {k: b[:n * H * W] for (k, b), n in zip(buf.items(), (R, B, 2 * B))}
        view["ref"].copy_(torch.from_numpy(np.stack([img(0.0), img(1.0)]).astype(np.float32)).ravel())
        view["test"].copy_(torch.from_numpy(np.stack([img(0.2), img(1.3), img(0.8)]).astype(np.float32)).ravel())
        view["field"].fill_(-9)
        if pin:
            for l in range(L):
                P.hrebsd_set_tile_variant(ctx, H >> l, W >> l, 0)
        P.hrebsd_demons_register_batch(ctx, view["ref"], view["test"], idx, R, B, H, W, prm, None, view["field"], iters,
                                       status)
        P.hrebsd_device_error(ctx)
        return view["field"].cpu().numpy().copy()

    shared = P.hrebsd_create(0)
    for H, W in sizes:
        own = P.hrebsd_create(0)
        assert np.array_equal(run(shared, H, W), run(own, H, W)), (H, W)
        P.hrebsd_destroy(own)
    P.hrebsd_destroy(shared)
