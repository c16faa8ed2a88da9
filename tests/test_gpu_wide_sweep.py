"""The sweep over strips of columns and bands of rows (level widths that the row sweep of whole rows does not
cover) against the pinned 64 x 32 tiles: same fields, iteration counts and status, at one and several strips
and bands, every position of the right edge in its warp, with the stop rule (the SSD regrouped as the tiles
sum it) and without."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(rng, B, H, W):
    y, x = np.mgrid[0:H, 0:W]
    refs = np.zeros((3, H, W))
    for r in refs:
        for _ in range(6):
            a, p = rng.uniform(0, np.pi), rng.uniform(0, 6)
            r += np.cos(rng.uniform(8, 30) / 100 * (np.cos(a) * x + np.sin(a) * y) + p)
    refs = (refs / refs.std(axis=(1, 2), keepdims=True)).astype(np.float32)
    idx = np.arange(B) % 3
    tests = np.stack([np.roll(refs[i], (int(rng.integers(-2, 3)), int(rng.integers(-2, 3))), (0, 1)) for i in idx])
    return refs, tests + 0.05 * rng.standard_normal(tests.shape, dtype=np.float32), idx.astype(np.int32)


def _run(refs, tests, idx, levels, cap, stop, pin):
    import torch
    import paper_1907_05993_gb300 as P
    (B, H, W), dev = tests.shape, lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    refs, tests, idx = dev(refs), dev(tests), dev(idx)
    ctx = P.hrebsd_create(0)
    if pin:
        for l in range(levels):
            P.hrebsd_set_tile_variant(ctx, H >> l, W >> l, 0)
    field = torch.empty((B, 2, H, W), device="cuda")
    iters = torch.full((B, levels), -1, dtype=torch.int32, device="cuda")
    status = torch.full((B,), -1, dtype=torch.int32, device="cuda")
    prm = P.demons_params(levels, [cap] * levels, 1.0, 1.0, 1.0, 1e-3 if stop else 0.0, 5 if stop else 0)
    P.hrebsd_demons_register_batch(ctx, refs, tests, idx, len(refs), B, H, W, prm, None, field, iters, status)
    P.hrebsd_device_error(ctx)
    n = P.hrebsd_launch_count(ctx)
    P.hrebsd_destroy(ctx)
    return field.cpu().numpy(), iters.cpu().numpy(), status.cpu().numpy(), n


def _compare(refs, tests, idx, levels, cap, stop):
    a, b = (_run(refs, tests, idx, levels, cap, stop, pin) for pin in (False, True))
    assert np.array_equal(a[0], b[0], equal_nan=True) and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    if stop:   # the sweep ran: its SSD is formed in a launch of its own
        assert a[3] > b[3]


@pytest.mark.parametrize("B,H,W,levels,cap,stop", [
    (16, 512, 622, 1, 20, True), (16, 1024, 1244, 2, 6, False), (152, 300, 311, 1, 25, True), (600, 92, 100, 1, 30, True),
    (600, 92, 100, 1, 1, False), (400, 77, 270, 1, 7, False), (60, 61, 1021, 1, 12, False), (1200, 131, 101, 1, 12, True),
])
def test_strip_band_sweep_matches_tiles(B, H, W, levels, cap, stop):
    _compare(*_batch(np.random.default_rng(B + H * W), B, H, W), levels, cap, stop)


def test_strip_band_sweep_at_every_right_edge():
    refs, tests, idx = _batch(np.random.default_rng(3), 300, 150, 226)
    for w in range(195, 227):
        _compare(refs[:, :, :w], tests[:, :, :w], idx, 1, 8, True)


def test_strip_band_sweep_nonfinite_pair_stops():
    import paper_1907_05993_gb300 as P
    refs, tests, idx = _batch(np.random.default_rng(4), 300, 150, 202)
    tests[7, 80, 201] = np.nan
    _compare(refs, tests, idx, 1, 8, True)
    status = _run(refs, tests, idx, 1, 8, True, False)[2]
    assert status[7] & P.PAIR_NONFINITE and not status[8] & P.PAIR_NONFINITE
