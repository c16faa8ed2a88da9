"""The cluster form of a pyramid level (few pairs, sizes the row sweep does not cover) against the pinned
tile and sweep shapes: same fields, same iteration counts, at bands of every size, ragged sizes, with the
stop rule (the SSD regrouped as the other shape sums it) and without."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _images(rng, n, h, w):
    y, x = np.mgrid[0:h, 0:w]
    out = np.zeros((n, h, w))
    for i in range(n):
        for _ in range(6):
            a, p = rng.uniform(0, np.pi), rng.uniform(0, 6)
            out[i] += np.cos(rng.uniform(8, 30) / 100 * (np.cos(a) * x + np.sin(a) * y) + p)
    return (out / out.std(axis=(1, 2), keepdims=True)).astype(np.float32)


# (B, H, W, levels, caps, stop, pinned shape per level); -1: the shape that runs when none is pinned
@pytest.mark.parametrize("B,H,W,levels,cap,stop", [
    (1, 128, 128, 3, 50, False), (1, 128, 128, 3, 60, True), (3, 256, 256, 2, 25, True), (5, 100, 92, 3, 40, True),
    (160, 46, 50, 1, 30, True), (2, 77, 33, 2, 30, True), (1, 8, 8, 1, 12, True), (1, 37, 200, 1, 20, True),
    (40, 64, 64, 2, 30, True), (1, 9, 300, 1, 9, False), (1, 300, 9, 1, 9, False), (2, 64, 48, 1, 1, True),
])
def test_cluster_level_matches_pinned_shapes(B, H, W, levels, cap, stop):
    import torch
    import paper_1907_05993_gb300 as P
    rng = np.random.default_rng(B + H * W)
    refs = _images(rng, min(B, 3), H, W)
    idx = np.arange(B) % len(refs)
    tests = np.stack([np.roll(refs[i], (int(rng.integers(-2, 3)), int(rng.integers(-2, 3))), (0, 1)) for i in idx])
    tests = (tests + 0.05 * rng.standard_normal(tests.shape)).astype(np.float32)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)
    refs, tests, idx = dev(refs, torch.float32), dev(tests, torch.float32), dev(idx, torch.int32)
    prm = P.demons_params(levels, [cap] * levels, 1.0, 1.0, 1.0, 1e-3 if stop else 0.0, 5 if stop else 0)

    def run(pins):
        ctx = P.hrebsd_create(0)
        for l, v in enumerate(pins):
            P.hrebsd_set_tile_variant(ctx, H >> l, W >> l, v)
        field = torch.empty((B, 2, H, W), device="cuda")
        iters = torch.full((B, levels), -1, dtype=torch.int32, device="cuda")
        status = torch.full((B,), -1, dtype=torch.int32, device="cuda")
        for _ in range(2):
            P.hrebsd_demons_register_batch(ctx, refs, tests, idx, len(refs), B, H, W, prm, None, field, iters, status)
        P.hrebsd_device_error(ctx)
        n = P.hrebsd_launch_count(ctx)
        P.hrebsd_destroy(ctx)
        return field.cpu().numpy(), iters.cpu().numpy(), status.cpu().numpy(), n

    field, iters, status, n = run([])
    # the shape that a level of this size runs in when nothing is chosen: the row sweep, else 64 x 32 tiles
    f0, i0, s0, n0 = run([5 if (W >> l) in (64, 128, 256) else 0 for l in range(levels)])
    assert np.array_equal(field, f0) and np.array_equal(iters, i0) and np.array_equal(status, s0)
    assert n < n0 or cap == 1   # the cluster form ran: one launch per level instead of two per iteration
    if not stop:   # any shape gives the same field
        f1, i1, s1, _ = run([1] * levels)
        assert np.array_equal(field, f1) and np.array_equal(iters, i1) and np.array_equal(status, s1)


def test_cluster_level_nonfinite_pair_stops():
    import torch
    import paper_1907_05993_gb300 as P
    x = _images(np.random.default_rng(1), 2, 100, 92)
    x[1, 50, 40] = np.nan
    t = torch.from_numpy(x).cuda()
    out = {}
    for pin in (False, True):
        ctx = P.hrebsd_create(0)
        if pin:
            for l in range(2):
                P.hrebsd_set_tile_variant(ctx, 100 >> l, 92 >> l, 0)
        field = torch.empty((2, 2, 100, 92), device="cuda")
        iters, status = (torch.empty(s, dtype=torch.int32, device="cuda") for s in ((2, 2), (2,)))
        P.hrebsd_demons_register_batch(ctx, t[:1].contiguous(), t, torch.zeros(2, dtype=torch.int32, device="cuda"), 1, 2,
                                       100, 92, P.demons_params(2, [7, 7]), None, field, iters, status)
        out[pin] = (field.cpu().numpy(), iters.cpu().numpy(), status.cpu().numpy())
        P.hrebsd_destroy(ctx)
    for a, b in zip(out[False], out[True]):
        assert np.array_equal(a, b, equal_nan=True)
    assert out[False][2][1] & P.PAIR_NONFINITE and not out[False][2][0] & P.PAIR_NONFINITE
